"""Emulated GEMMs captured into a CUDA graph: after one uncaptured call of
the same shape (which sizes the handle's workspace) DGEMM with every scheme
and ZGEMM 3M capture on the caller's stream and, replayed after the inputs
were overwritten in place, give bit for bit what an uncaptured call on the
new inputs gives.  A call that would have to grow the workspace while its
stream is capturing is refused with EMU_ERR_ALLOC before it enqueues
anything, and the handle keeps working afterwards."""
import os
import subprocess
import sys

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


@pytest.mark.parametrize("scheme,p", [("I", 7), ("I_F8", 11), ("II", 16), ("II_NORM", 14)])
def test_dgemm_capture_and_replay(scheme, p):
    h = emu.Handle(0)
    m, n, k = 300, 260, 1100
    A, B = synth.gemm_pair(m, n, k, 1.0, 171)
    A2, B2 = synth.gemm_pair(m, n, k, 2.0, 172)
    Ad, Bd = dev(A), dev(B)
    C = torch.empty((m, n), dtype=torch.float64, device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    emu.dgemm(Ad, Bd, C, scheme=scheme, p=p, handle=h, stream=s)  # sizes the workspace
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        emu.dgemm(Ad, Bd, C, alpha=0.5, scheme=scheme, p=p, handle=h, stream=s)
    Ad.copy_(dev(A2))
    Bd.copy_(dev(B2))
    C.fill_(float("nan"))
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert h.status() == 0
    ref = emu.dgemm(dev(A2), dev(B2), alpha=0.5, scheme=scheme, p=p, handle=h)
    assert np.array_equal(C.cpu().numpy(), ref.cpu().numpy())
    h.close()


def test_zgemm_capture_and_replay():
    h = emu.Handle(0)
    m, n, k, nm = 200, 150, 700, 12
    A, B = synth.gemm_pair_complex(m, n, k, 1.0, 173)
    Ad, Bd = dev(A), dev(B)
    C = torch.empty((m, n), dtype=torch.complex128, device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    emu.zgemm(Ad, Bd, C, nm=nm, handle=h, stream=s)
    s.synchronize()
    ref = C.cpu().numpy()
    C.zero_()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        emu.zgemm(Ad, Bd, C, nm=nm, handle=h, stream=s)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    assert h.status() == 0
    assert np.array_equal(C.cpu().numpy(), ref)
    h.close()


@pytest.mark.filterwarnings("ignore:The CUDA Graph is empty")  # nothing was enqueued, as intended
def test_workspace_growth_refused_while_capturing(orc):
    h = emu.Handle(0)  # no workspace yet
    A, B = synth.gemm_pair(128, 96, 256, 1.0, 174)
    Ad, Bd = dev(A), dev(B)
    C = torch.zeros((128, 96), dtype=torch.float64, device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with pytest.raises(emu.EmuError) as e:
        with torch.cuda.graph(g, stream=s):
            emu.dgemm(Ad, Bd, C, scheme="I", p=6, handle=h, stream=s)
    assert e.value.code == 5  # EMU_ERR_ALLOC
    torch.cuda.synchronize()
    assert h.status() == 0
    # outside the capture the same call allocates and runs
    emu.dgemm(Ad, Bd, C, scheme="I", p=6, handle=h)
    assert np.array_equal(C.cpu().numpy(), orc.emu_I(A, B, 6))
    h.close()


def test_graph_outlives_workspace_growth(orc):
    # larger calls after the capture: the graph's workspace stays allocated
    h = emu.Handle(0)
    A, B = synth.gemm_pair(128, 96, 256, 1.0, 175)
    Ad, Bd = dev(A), dev(B)
    C = torch.zeros((128, 96), dtype=torch.float64, device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    emu.dgemm(Ad, Bd, C, scheme="I", p=6, handle=h, stream=s)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        emu.dgemm(Ad, Bd, C, scheme="I", p=6, handle=h, stream=s)
    A2, B2 = synth.gemm_pair(400, 300, 700, 1.0, 176)
    for p in (7, 8):
        C2 = emu.dgemm(dev(A2), dev(B2), scheme="I", p=p, handle=h)
        C.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(C.cpu().numpy(), orc.emu_I(A, B, 6))
        assert np.array_equal(C2.cpu().numpy(), orc.emu_I(A2, B2, p))
    assert h.status() == 0
    h.close()


CHILD_FULL = r"""
import sys, torch
sys.path.insert(0, %r)
import paper_2606_25453_gb300 as emu
import synth
h = emu.Handle(0)
A, B = (torch.from_numpy(x).cuda() for x in synth.gemm_pair(200, 150, 300, 1.0, 177))
C = torch.zeros((200, 150), dtype=torch.float64, device="cuda")
s = torch.cuda.Stream()
s.wait_stream(torch.cuda.current_stream())
def call(hd):
    emu.dgemm(A, B, C, scheme="I", p=8, handle=hd, stream=s)
call(h)
s.synchronize()
first = C.clone()
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=s):
    call(h)
ok = True
for _ in range(3):  # the same shape again, uncaptured, then a replay
    call(h)
    s.synchronize()
    ok = ok and torch.equal(C, first)
    C.zero_()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    ok = ok and torch.equal(C, first)
print("same", ok, "status", h.status(), float(first.abs().sum()))
"""


def test_fallback_keeps_its_workspace_for_graphs(orc):
    """No room for the digit planes (allocations above the slices' size fail):
    the INT8 kernel runs, and a graph captured on its workspace still replays
    after more uncaptured calls of the same shape."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    A, B = synth.gemm_pair(200, 150, 300, 1.0, 177)
    slices = (emu.emu_split_rows(200) + emu.emu_split_rows(150)) * emu.emu_split_cols_I(300, 8) + 16384
    env = dict(os.environ, EMU_FAULT="alloc:%d" % (slices * 9 // 8))
    r = subprocess.run([sys.executable, "-c", CHILD_FULL % root], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    want = float(np.abs(orc.emu_I(A, B, 8)).sum())
    assert r.stdout.startswith("same True status 0 "), r.stdout
    assert abs(float(r.stdout.split()[-1]) - want) <= 1e-12 * want
