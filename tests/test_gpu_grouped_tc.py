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


@pytest.mark.parametrize("p", [9])
def test_one_stage_of_the_mma_kernels(orc, tmp_path, p):
    # three stages by default (the test above), here one
    path = tmp_path / "one.json"
    lines = ['  "p%d_s%d_k%d": %d' % (p, sc, kc, (2 * sc + kc) % 6) for sc in range(5) for kc in range(5)]
    path.write_text("{\n" + ",\n".join(lines + ['  "p%d_stages": 1' % p]) + "\n}\n")
    h = emu.Handle(0)
    emu.check(emu.emu_load_tuning(h.h, str(path).encode()))
    rng = np.random.Generator(np.random.PCG64(4))
    shapes = [tuple(int(x) for x in rng.integers((20, 20, 60), (500, 500, 900))) for _ in range(12)]
    check(orc, h, shapes, p, 170)
    h.close()


def test_tuned_batch_of_nine_slices_is_bit_exact(orc, tmp_path):
    # nine slices run on the mma.sync kernels that the tuner times
    p = 9
    mats = [synth.gemm_pair(m, n, k, 1.0, 270 + i) for i, (m, n, k) in enumerate([(60, 200, 300), (250, 40, 100)] * 5)]
    As, Bs = [torch.from_numpy(A).cuda() for A, _ in mats], [torch.from_numpy(B).cuda() for _, B in mats]
    Cs = [torch.full((A.shape[0], B.shape[1]), float("nan"), dtype=torch.float64, device="cuda") for A, B in mats]
    d = emu.grouped_descs(As, Bs, Cs)
    h = emu.Handle(0)
    path = str(tmp_path / "tune.json")
    assert emu.tune_grouped(d, p, path=path, handle=h) > 0
    h2 = emu.Handle(0)
    emu.check(emu.emu_load_tuning(h2.h, path.encode()))
    for hd in (h, h2):
        for C in Cs:
            C.fill_(float("nan"))
        emu.dgemm_grouped(d, p, handle=hd)
        torch.cuda.synchronize()
        assert hd.status() == 0
        for (A, B), C in zip(mats, Cs):
            assert np.array_equal(C.cpu().numpy(), orc.emu_I(A, B, p))
    h.close()
    h2.close()


def test_tuning_leaves_a_bf16_plan_alone(tmp_path):
    """A tuning concerns the mma.sync kernels: loading one must not make the
    next call of a batch on the bf16 engine synchronise the device and build
    its plan again."""
    A, B = synth.gemm_pair(300, 200, 500, 1.0, 6)
    As, Bs = [torch.from_numpy(A).cuda()] * 4, [torch.from_numpy(B).cuda()] * 4
    Cs = [torch.empty((300, 200), dtype=torch.float64, device="cuda") for _ in As]
    d = emu.grouped_descs(As, Bs, Cs)
    h = emu.Handle(0)
    emu.dgemm_grouped(d, 6, handle=h)
    ref = Cs[0].clone()
    torch.cuda.synchronize()
    path = tmp_path / "t.json"
    path.write_text("{\n" + ",\n".join('  "p6_s%d_k%d": 3' % (i, j) for i in range(5) for j in range(5)) +
                    ',\n  "p6_stages": 1\n}\n')
    emu.check(emu.emu_load_tuning(h.h, str(path).encode()))
    done = torch.cuda.Event()
    torch.cuda._sleep(200_000_000)  # about 0.1 s of a busy stream
    emu.dgemm_grouped(d, 6, handle=h)
    done.record()
    assert not done.query()  # a rebuild would have waited for the device
    torch.cuda.synchronize()
    assert torch.equal(Cs[0], ref)
    h.close()


# both sides of the lines between the engines for batches of many small
# products of short K: items per SM, mean K, fill
@pytest.mark.parametrize("count,n,k,p,bf16", [
    (320, 32, 32, 8, False), (300, 32, 32, 8, True), (320, 32, 65, 8, True), (160, 200, 64, 8, True),
    (160, 150, 40, 8, False), (320, 32, 32, 4, True), (1100, 16, 32, 8, False), (1000, 16, 32, 8, True),
    (2800, 16, 32, 6, False), (2700, 16, 32, 6, True)])
def test_engine_lines_of_small_products(orc, count, n, k, p, bf16):
    rng = np.random.Generator(np.random.PCG64(count + n))
    A = torch.from_numpy(rng.standard_normal((count, n, k))).cuda()
    B = torch.from_numpy(rng.standard_normal((count, k, n))).cuda()
    C = torch.full((count, n, n), float("nan"), dtype=torch.float64, device="cuda")
    h = emu.Handle(0)
    h.trace(True)
    h.trace_read()
    emu.dgemm_grouped(emu.grouped_descs(list(A), list(B), list(C)), p, handle=h)
    t = h.trace_read()
    h.trace(False)
    assert h.status() == 0
    h.close()
    # scan, split, GEMM, combine; else three stages of scan, split and GEMMs
    assert (t["kernel_launches"] == 4) == bf16, t
    for i in (0, 1, count // 2, count - 1):
        assert np.array_equal(C[i].cpu().numpy(), orc.emu_I(A[i].cpu().numpy(), B[i].cpu().numpy(), p)), i
