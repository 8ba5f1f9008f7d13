"""The residue GEMM on CTA pairs and on single CTAs at the edges of its
dispatch and tiles: K around the 896 where pairs begin, their 128-deep stages
and 896-deep exact segments; rows around 128- and 256-row tiles; columns
around the MMA's steps of 32 and the 256-column tile.  Bit for bit against
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


@pytest.mark.parametrize("m,n,k", [(256, 256, 895), (256, 256, 896), (200, 31, 897), (129, 33, 960), (257, 257, 1024),
                                   (640, 17, 1793), (513, 300, 1855), (641, 250, 2689), (128, 64, 1000)])
@pytest.mark.parametrize("nm", [3, 16, 20])
def test_edges(orc, m, n, k, nm):
    A, B = synth.gemm_pair(m, n, k, 1.0, m + n + k + nm)
    h = emu.Handle(0)
    C = emu.dgemm(dev(A), dev(B), scheme="II", p=nm, handle=h).cpu().numpy()
    assert h.status() == 0
    h.close()
    assert np.array_equal(C, orc.emu_II(A, B, nm))


@pytest.mark.parametrize("m,n,k", [(130, 70, 899), (260, 120, 1400)])
def test_complex_edges(orc, m, n, k):
    A, B = synth.gemm_pair_complex(m, n, k, 1.0, 5 * m)
    h = emu.Handle(0)
    C = emu.zgemm(dev(A), dev(B), nm=14, handle=h).cpu().numpy()
    assert h.status() == 0
    h.close()
    assert np.array_equal(C, orc.emu_Z3M(A, B, 14))
