"""Grouped products on the bf16 tensor cores (up to eight slices) at tile and
segment edges, in batches of one and of several products, and the mma.sync
kernels that nine and more slices keep, with a tuning that mixes their
configurations.  Bit for bit against the oracle (exact integers fix every
rounding, so the tolerance is zero)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_25453_gb300 as emu  # noqa: E402


def check(orc, h, shapes, p, seed, alpha=None, beta=None, pads=None):
    mats = [synth.gemm_pair(m, n, k, 1.0, seed + i) for i, (m, n, k) in enumerate(shapes)]
    pads = pads or [0] * len(shapes)

    def dev(x, pad):  # rows padded by `pad` elements: every alignment of the row starts
        t = torch.full((x.shape[0], x.shape[1] + pad), float("nan"), dtype=torch.float64, device="cuda")
        t[:, :x.shape[1]] = torch.from_numpy(x).cuda()
        return t[:, :x.shape[1]]

    As, Bs = [dev(A, q) for (A, _), q in zip(mats, pads)], [dev(B, q) for (_, B), q in zip(mats, pads)]
    C0 = [synth.test_matrix(m, n, 1.0, seed + 500 + i) for i, (m, n, _) in enumerate(shapes)]
    Cs = [dev(c, 0) for c in C0]
    d = emu.grouped_descs(As, Bs, Cs, alpha, beta)
    emu.dgemm_grouped(d, p, handle=h)
    torch.cuda.synchronize()
    assert h.status() == 0
    for i, ((A, B), C) in enumerate(zip(mats, Cs)):
        want = orc.emu_I(A, B, p, alpha=alpha[i] if alpha else 1.0, beta=beta[i] if beta else 0.0, C=C0[i])
        assert np.array_equal(C.cpu().numpy(), want), (i, shapes[i])


EDGES = [(1, 1, 1), (7, 31, 63), (8, 32, 64), (9, 33, 65), (128, 256, 256), (129, 257, 257), (60, 500, 961),
         (300, 20, 1300), (131, 264, 2500)]


@pytest.mark.parametrize("p", [1, 2, 5, 8])
def test_edges_in_one_batch(orc, p):
    h = emu.Handle(0)
    check(orc, h, EDGES, p, 900 + p, pads=[i % 4 for i in range(len(EDGES))])
    h.close()


def test_single_product_and_update(orc):
    h = emu.Handle(0)
    check(orc, h, [(140, 300, 700)], 7, 40)
    check(orc, h, [(64, 40, 90), (200, 100, 300)], 6, 60, alpha=[-0.5, 2.0], beta=[1.5, 0.0])
    h.close()


@pytest.mark.parametrize("p", [9, 12])
def test_more_than_eight_slices_mixed_configurations(orc, tmp_path, p):
    path = tmp_path / "mixed.json"
    lines = ['  "p%d_s%d_k%d": %d' % (p, sc, kc, (sc + 2 * kc) % 6) for sc in range(5) for kc in range(5)]
    path.write_text("{\n" + ",\n".join(lines) + "\n}\n")
    h = emu.Handle(0)
    emu.check(emu.emu_load_tuning(h.h, str(path).encode()))
    rng = np.random.Generator(np.random.PCG64(3))
    shapes = [tuple(int(x) for x in rng.integers((20, 20, 60), (500, 500, 900))) for _ in range(12)]
    check(orc, h, shapes, p, 70)
    h.close()
