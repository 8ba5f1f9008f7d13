"""The CRT by pairs of moduli for every number of moduli (odd ones leave a
pair with one modulus; P has one to five 32-bit limbs), columns around the
four a thread takes, exact zeros and both signs.  Bit for bit against the
oracle (exact integers fix every rounding)."""
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


@pytest.mark.parametrize("nm", range(1, 21))
def test_real(orc, nm):
    m, n, k = 37, 17 + nm % 4, 2 + nm
    A, B = synth.gemm_pair(m, n, k, 1.0, 100 + nm)
    A[3] = 0.0
    A[5] = -A[4]
    h = emu.Handle(0)
    C = emu.dgemm(dev(A), dev(B), scheme="II", p=nm, handle=h).cpu().numpy()
    assert h.status() == 0
    h.close()
    assert np.array_equal(C, orc.emu_II(A, B, nm))


@pytest.mark.parametrize("nm", range(1, 21))
def test_complex(orc, nm):
    A, B = synth.gemm_pair_complex(19, 9 + nm % 4, 5, 1.0, 200 + nm)
    A[2] = 0.0
    h = emu.Handle(0)
    C = emu.zgemm(dev(A), dev(B), nm=nm, handle=h).cpu().numpy()
    assert h.status() == 0
    h.close()
    assert np.array_equal(C, orc.emu_Z3M(A, B, nm))
