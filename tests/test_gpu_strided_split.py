"""Strided operands (B of a row-major product, A of a column-major one) on
both sides of the rule for the number of vectors per block of the splits:
blocks of eight vectors (small operands) and of 32, ragged vector counts,
unaligned leading dimensions, K around a group of 128.  Bit for bit against
the oracle (exact integers fix every rounding)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_25453_gb300 as emu  # noqa: E402


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("n", [1, 7, 8, 9, 33, 250, 4999])
@pytest.mark.parametrize("k", [127, 129, 700])
@pytest.mark.parametrize("scheme,p", [("I", 7), ("II", 14), ("II_NORM", 14)])
def test_real(orc, scheme, p, n, k):
    A, B = synth.gemm_pair(5, n, k, 1.0, n + k)
    h = emu.Handle(0)
    C = emu.dgemm(dev(A), dev(B), scheme=scheme, p=p, handle=h).cpu().numpy()
    F = emu.sgemm(dev(A.astype(np.float32)), dev(B.astype(np.float32)), scheme=scheme, p=p, handle=h).cpu().numpy()
    assert h.status() == 0
    h.close()
    Af, Bf = A.astype(np.float32).astype(np.float64), B.astype(np.float32).astype(np.float64)
    if scheme == "I":
        assert np.array_equal(C, orc.emu_I(A, B, p))
        assert np.array_equal(F, orc.emu_I(Af, Bf, p, out_f32=True))
    else:
        assert np.array_equal(C, orc.emu_II(A, B, p, norm=scheme == "II_NORM"))
        assert np.array_equal(F, orc.emu_II(Af, Bf, p, out_f32=True, norm=scheme == "II_NORM"))


@pytest.mark.parametrize("n", [1, 9, 17, 3001])
def test_complex(orc, n):
    A, B = synth.gemm_pair_complex(5, n, 300, 1.0, n)
    h = emu.Handle(0)
    C = emu.zgemm(dev(A), dev(B), nm=14, handle=h).cpu().numpy()
    assert h.status() == 0
    h.close()
    assert np.array_equal(C, orc.emu_Z3M(A, B, 14))
