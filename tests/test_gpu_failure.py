"""Failure detection without faulting the GPU: a bounded device wait that is
made to run out reports EMU_ERR_TIMEOUT through the status word and leaves
the context usable; host-side fault injection: EMU_FAULT=alloc turns
workspace allocation into EMU_ERR_ALLOC while a caller-owned workspace still
works, EMU_FAULT=launch makes every fused GEMM launch fail on the host, and
EMU_FAULT=zero, scan, norm or split every launch of that step before it
(EMU_ERR_CUDA, C untouched, context intact)."""
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

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_bounded_wait_times_out_and_context_survives(orc):
    h = emu.Handle(0)
    emu.check(emu.emu_selftest_wait(h.h, 2_000_000, None))  # ~1 ms at 2 GHz
    assert h.status() == 6  # EMU_ERR_TIMEOUT, read and cleared
    assert h.status() == 0
    A, B = synth.gemm_pair(70, 50, 90, 1.0, 3)
    C = emu.dgemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), scheme="I", p=5, handle=h)
    assert np.array_equal(C.cpu().numpy(), orc.emu_I(A, B, 5))
    h.close()


CHILD = r"""
import sys, ctypes, torch
sys.path.insert(0, %r)
import paper_2606_25453_gb300 as emu
h = emu.Handle(0)
A = torch.ones((64, 64), dtype=torch.float64, device="cuda")
try:
    emu.dgemm(A, A, scheme="I", p=4, handle=h)
    print("no-error")
except emu.EmuError as e:
    print("code", e.code)
sz = ctypes.c_size_t()
emu.check(emu.emu_workspace_size(1, 64, 64, 64, 4, 0, ctypes.byref(sz)))
ws = torch.empty(sz.value + 256, dtype=torch.uint8, device="cuda")
emu.check(emu.emu_set_workspace(h.h, ws.data_ptr(), sz.value))
C = emu.dgemm(A, A, scheme="I", p=4, handle=h)
torch.cuda.synchronize()
print("user-ws", float(C[0, 0]))
"""


def test_alloc_fault_injection():
    env = dict(os.environ, EMU_FAULT="alloc")
    r = subprocess.run([sys.executable, "-c", CHILD % ROOT], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert "code 5" in r.stdout  # EMU_ERR_ALLOC
    assert "user-ws 64.0" in r.stdout


CHILD_LAUNCH = r"""
import sys, torch
sys.path.insert(0, %r)
import paper_2606_25453_gb300 as emu
h = emu.Handle(0)
A = torch.ones((64, 64), dtype=torch.float64, device="cuda")
for scheme, p in (("I", 4), ("I_F8", 8), ("II", 10)):
    C = torch.full((64, 64), 7.0, dtype=torch.float64, device="cuda")
    try:
        emu.dgemm(A, A, C, scheme=scheme, p=p, handle=h)
        print(scheme, "no-error")
    except emu.EmuError as e:
        torch.cuda.synchronize()
        print(scheme, "code", e.code, "untouched", bool((C == 7.0).all()), "|", str(e))
try:
    emu.zgemm(A.to(torch.complex128), A.to(torch.complex128), nm=8, handle=h)
except emu.EmuError as e:
    print("Z code", e.code)
print("status", h.status(), "ctx", float((A @ A)[0, 0]))
"""


def test_launch_fault_injection():
    # EMU_FAULT=launch: each fused GEMM launch fails on the host side after
    # the scan and split were enqueued; the caller gets EMU_ERR_CUDA with
    # the runtime's text, C is not written, nothing faults on the device,
    # and the context stays usable
    env = dict(os.environ, EMU_FAULT="launch")
    r = subprocess.run([sys.executable, "-c", CHILD_LAUNCH % ROOT], env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
    for scheme in ("I", "I_F8", "II"):
        assert "%s code 4 untouched True" % scheme in r.stdout, r.stdout
    assert "unspecified launch failure" in r.stdout
    assert "Z code 4" in r.stdout
    assert "status 0 ctx 64.0" in r.stdout


CHILD_STEP = r"""
import sys, torch
sys.path.insert(0, %r)
import paper_2606_25453_gb300 as emu
h = emu.Handle(0)
A = torch.ones((64, 64), dtype=torch.float64, device="cuda")
At = A.t()

def case(name, fn, C):
    try:
        fn(C)
        code = 0
    except emu.EmuError as e:
        code = e.code
    torch.cuda.synchronize()
    print(name, "code", code, "untouched", bool((C == 7.0).all()), flush=True)

def full(dtype=torch.float64, **kw):
    return torch.full((64, 64), 7.0, dtype=dtype, **(kw or {"device": "cuda"}))

for scheme, p in (("I", 4), ("I", 12), ("I_F8", 8), ("II", 10), ("II_NORM", 10)):
    case("d_%%s_%%d" %% (scheme, p), lambda C: emu.dgemm(A, A, C, scheme=scheme, p=p, handle=h), full())
    case("dcol_%%s_%%d" %% (scheme, p), lambda C: emu.dgemm(At, At, C.t(), scheme=scheme, p=p, handle=h), full())
    Z = A.to(torch.complex128)
    case("z_%%s_%%d" %% (scheme, p), lambda C: emu.zgemm(Z, Z, C, nm=p, p=p, scheme=scheme, handle=h), full(torch.complex128))
    F = A.float()
    case("s_%%s_%%d" %% (scheme, p), lambda C: emu.sgemm(F, F, C, scheme=scheme, p=p, handle=h), full(torch.float32))
    H = A.cpu().pin_memory()
    case("host_%%s_%%d" %% (scheme, p), lambda C: emu.dgemm_host(H, H, C, scheme=scheme, p=p, handle=h),
         full(pin_memory=True))
S = torch.cuda.current_stream().cuda_stream
case("noalloc_I", lambda C: emu.check(emu.emu_dgemm_noalloc(0, 64, 64, 64, 1.0, A.data_ptr(), 64, A.data_ptr(), 64, 0.0,
                                                            C.data_ptr(), 64, 4, None, S)), full())
for scheme in ("I", "II"):
    case("auto_" + scheme, lambda C: emu.dgemm_auto(A, A, 1e-10, handle=h, scheme=scheme, C=C), full())
E = torch.zeros(64, dtype=torch.int32, device="cuda")
X = torch.empty(1 << 16, dtype=torch.int8, device="cuda")
for name, fn in (("I", lambda: emu.emu_split_I(h.h, 0, 0, 64, 64, A.data_ptr(), 64, 4, X.data_ptr(), E.data_ptr(), S)),
                 ("F8", lambda: emu.emu_split_F8(h.h, 0, 0, 64, 64, A.data_ptr(), 64, 4, X.data_ptr(), E.data_ptr(), S)),
                 ("II", lambda: emu.emu_split_II(h.h, 0, 0, 64, 64, 64, A.data_ptr(), 64, 4, X.data_ptr(), E.data_ptr(), S))):
    print("split_" + name, "code", fn(), flush=True)
print("status", h.status(), "ctx", float((A @ A)[0, 0]))
"""


@pytest.mark.parametrize("engine", ["", "mma"])
@pytest.mark.parametrize("step", ["zero", "scan", "norm", "split"])
def test_step_fault_injection(step, engine):
    # a step whose launch fails must end the call with EMU_ERR_CUDA: the
    # kernels after it would run on what an earlier call left in the workspace
    env = dict(os.environ, EMU_FAULT=step)
    if engine:
        env.update(EMU_I_ENGINE=engine, EMU_II_ENGINE=engine, EMU_F8_ENGINE=engine)
    r = subprocess.run([sys.executable, "-c", CHILD_STEP % ROOT], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    lines = [x.split() for x in r.stdout.splitlines()]
    assert ["status", "0", "ctx", "64.0"] in lines, r.stdout
    seen = 0
    for x in lines:
        if x[1] != "code":
            continue
        # who runs the step at all: norm scaling alone has sums of squares; the
        # chunks of a product in host memory and the lone splits start with a
        # memset, and the selector's own kernel zeroes for Scheme I
        has = {"norm": "NORM" in x[0] or x[0] == "auto_II",
               "zero": not (x[0].startswith(("split", "host")) or x[0] == "auto_I") or "NORM" in x[0],
               "scan": True, "split": True}[step]
        if x[0].startswith("host_II") and engine == "mma":
            has = has or step == "zero"  # the INT8 engine takes the whole product
        assert x[2] == ("4" if has else "0"), (step, x)
        if has and not x[0].startswith("split"):
            assert x[4] == "True", (step, x)
        seen += has
    assert seen >= 5
