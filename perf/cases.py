"""The library's work as its users call it, one case per kind of call.

Every case is one emulated matrix product (or one batch of them) through the
public binding, on operands drawn like the method's own evaluation:
a_ij = (u - 0.5) exp(phi g), u ~ U(0, 1), g ~ N(0, 1).  A user's program
keeps a handle and its output buffers; inputs are new.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2606_25453_gb300 as emu
from paper_2606_25453_gb300 import selector

DEV = "cuda"
# the costliest case any draw may reach: m n k p (p + 1) of dgemm_I_8192
_LARGEST = 8192 ** 3 * 72


def listed():
    return [
        # the smallest configured product: a single launch-bound call, as in
        # a loop over small systems
        {"name": "dgemm_I_256", "op": "gemm", "dtype": "f64", "scheme": "I", "p": 7, "m": 256, "n": 256, "k": 256,
         "phi": 0.5, "layout": "row", "alpha": 1.0, "beta": 0.0},
        # the benchmark's product: FP64-accurate slices at n = 8192
        {"name": "dgemm_I_8192", "op": "gemm", "dtype": "f64", "scheme": "I", "p": 8, "m": 8192, "n": 8192, "k": 8192,
         "phi": 0.5, "layout": "row", "alpha": 1.0, "beta": 0.0},
        # a BLAS caller's update C = alpha A B + beta C, column-major, no
        # dimension a multiple of a tile
        {"name": "dgemm_I_ragged", "op": "gemm", "dtype": "f64", "scheme": "I", "p": 6, "m": 1531, "n": 2013,
         "k": 3007, "phi": 2.0, "layout": "col", "alpha": -0.75, "beta": 0.5},
        # FP32 target: four slices
        {"name": "sgemm_I_4096", "op": "gemm", "dtype": "f32", "scheme": "I", "p": 4, "m": 4096, "n": 4096, "k": 4096,
         "phi": 0.5, "layout": "row", "alpha": 1.0, "beta": 0.0},
        # FP64 accuracy through the moduli at the benchmark's size
        {"name": "dgemm_II_8192", "op": "gemm", "dtype": "f64", "scheme": "II", "p": 16, "m": 8192, "n": 8192,
         "k": 8192, "phi": 0.5, "layout": "row", "alpha": 1.0, "beta": 0.0},
        # norm scaling on a mid-sized ragged update (rank-k update of a solver)
        {"name": "dgemm_II_norm_ragged", "op": "gemm", "dtype": "f64", "scheme": "II_NORM", "p": 14, "m": 2905,
         "n": 1777, "k": 803, "phi": 1.0, "layout": "row", "alpha": 1.5, "beta": -0.5},
        # complex128 by 3M at its configured size
        {"name": "zgemm_II_8192", "op": "gemm", "dtype": "c128", "scheme": "II", "p": 16, "m": 8192, "n": 8192,
         "k": 8192, "phi": 1.0, "layout": "row", "alpha": 1.0, "beta": 0.0},
        # complex64 by 3M, column-major with odd sizes
        {"name": "cgemm_II_ragged", "op": "gemm", "dtype": "c64", "scheme": "II", "p": 8, "m": 3001, "n": 2047,
         "k": 2500, "phi": 1.0, "layout": "col", "alpha": 1.0, "beta": 0.0},
        # FP64 accuracy with E4M3 slices on the FP8 tensor cores
        {"name": "dgemm_F8_4096", "op": "gemm", "dtype": "f64", "scheme": "I_F8", "p": 12, "m": 4096, "n": 4096,
         "k": 4096, "phi": 0.5, "layout": "row", "alpha": 1.0, "beta": 0.0},
        # a batch of uneven independent products in one call
        {"name": "grouped_512", "op": "grouped", "count": 512, "p": 6, "mn_max": 1024, "k_max": 2048, "phi": 1.0},
        # the tolerance-driven call: features, network, product, probe
        {"name": "auto_I_3000", "op": "auto", "scheme": "I", "m": 3000, "n": 2800, "k": 3200, "phi": 1.0,
         "tol": 1e-12},
        # operands and result in pinned host memory
        {"name": "host_I_4096", "op": "host", "scheme": "I", "p": 8, "m": 4096, "n": 4096, "k": 4096, "phi": 0.5},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _passes(c):
    """Slice products or moduli, in the unit of _LARGEST's p (p + 1)."""
    if c["scheme"] in ("I", "I_F8"):
        w = c["p"] * (c["p"] + 1)
    else:
        w = 2 * c["p"] * (3 if c.get("dtype") in ("c128", "c64") else 1)
    return w


def draw(rng):
    op = rng.choice(["gemm"] * 8 + ["grouped", "auto", "host"])
    if op == "grouped":
        return {"op": op, "count": _log_int(rng, 8, 512), "p": rng.randint(4, 8),
                "mn_max": _log_int(rng, 128, 1024), "k_max": _log_int(rng, 256, 2048),
                "phi": rng.choice([0.5, 1.0])}
    if op == "auto":
        return {"op": op, "scheme": rng.choice(["I", "II"]), "m": _log_int(rng, 256, 4096),
                "n": _log_int(rng, 256, 4096), "k": _log_int(rng, 256, 4096), "phi": rng.choice([0.5, 1.0, 2.0]),
                "tol": rng.choice([1e-8, 1e-12])}
    if op == "host":
        return {"op": op, "scheme": rng.choice(["I", "II"]), "p": rng.choice([7, 8]),
                "m": _log_int(rng, 256, 4096), "n": _log_int(rng, 256, 4096), "k": _log_int(rng, 256, 4096),
                "phi": 0.5}
    dtype = rng.choice(["f64"] * 5 + ["f32", "c128", "c64"])
    if dtype == "f64":
        scheme = rng.choice(["I", "I", "II", "II_NORM", "I_F8"])
        p = {"I": rng.randint(4, 8), "II": rng.randint(12, 20), "II_NORM": rng.randint(10, 18),
             "I_F8": rng.randint(8, 12)}[scheme]
    elif dtype == "f32":
        scheme = rng.choice(["I", "II"])
        p = rng.randint(3, 4) if scheme == "I" else rng.randint(6, 8)
    else:
        scheme = "II"
        p = rng.randint(12, 18) if dtype == "c128" else rng.randint(8, 10)
    # few slices or moduli are used where the exponent range is narrow
    phis = [0.5] if dtype == "f32" else [0.5, 1.0] if p < 6 or dtype == "c64" else [0.5, 1.0, 2.0]
    c = {"op": "gemm", "dtype": dtype, "scheme": scheme, "p": p, "m": _log_int(rng, 64, 8192),
         "n": _log_int(rng, 64, 8192), "k": _log_int(rng, 64, 8192), "phi": rng.choice(phis),
         "layout": rng.choice(["row", "row", "col"]), "alpha": 1.0, "beta": 0.0}
    if rng.random() < 0.3:
        c["alpha"], c["beta"] = -1.25, 0.5
    while c["m"] * c["n"] * c["k"] * _passes(c) > _LARGEST:
        c["k"] = c["k"] * 3 // 4
    return c


_TYPES = {"f64": torch.float64, "f32": torch.float32, "c128": torch.complex128, "c64": torch.complex64}


def _matrix(rows, cols, phi, gen, dtype, layout="row"):
    def real(r, c):
        u = torch.rand((r, c), generator=gen, device=DEV, dtype=torch.float64)
        g = torch.randn((r, c), generator=gen, device=DEV, dtype=torch.float64)
        return (u - 0.5) * torch.exp(phi * g)

    r, c = (rows, cols) if layout == "row" else (cols, rows)
    t = _TYPES[dtype]
    x = torch.complex(real(r, c), real(r, c)).to(t) if t.is_complex else real(r, c).to(t)
    return x if layout == "row" else x.t()


def _group_shapes(case):
    """The batch's shapes are the case's own; the seed draws the entries."""
    r = np.random.Generator(np.random.PCG64(case["count"]))

    def log_int(lo, hi):
        return int(round(float(np.exp(r.uniform(np.log(lo), np.log(hi))))))

    return [(log_int(32, case["mn_max"]), log_int(32, case["mn_max"]), log_int(64, case["k_max"]))
            for _ in range(case["count"])]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _pair(case, seed):
    gen = _gen(seed)
    dt, lay = case.get("dtype", "f64"), case.get("layout", "row")
    A = _matrix(case["m"], case["k"], case["phi"], gen, dt, lay)
    B = _matrix(case["k"], case["n"], case["phi"], gen, dt, lay)
    C0 = _matrix(case["m"], case["n"], 0.0, gen, dt, lay) if case.get("beta", 0.0) != 0.0 else None
    return A, B, C0


def _group_inputs(case, seed):
    gen, shapes = _gen(seed), _group_shapes(case)
    entries = _matrix(1, sum(m * k + k * n for m, n, k in shapes), case["phi"], gen, "f64").reshape(-1)
    A, B, at = [], [], 0
    for m, n, k in shapes:
        A.append(entries[at:at + m * k].view(m, k))
        at += m * k
        B.append(entries[at:at + k * n].view(k, n))
        at += k * n
    return shapes, entries, A, B


def prepare(case, seed):
    s = {"case": case, "h": emu.Handle(0)}
    if case["op"] == "grouped":
        shapes, s["entries"], A, B = _group_inputs(case, seed)
        s["C"] = torch.empty(sum(m * n for m, n, _ in shapes), dtype=torch.float64, device=DEV)
        C, at = [], 0
        for m, n, _ in shapes:
            C.append(s["C"][at:at + m * n].view(m, n))
            at += m * n
        s["descs"] = emu.grouped_descs(A, B, C)
        return s
    A, B, s["C0"] = _pair(case, seed)
    if case["op"] == "host":
        s["A"], s["B"] = A.cpu().pin_memory(), B.cpu().pin_memory()
        s["C"] = torch.empty((case["m"], case["n"]), dtype=torch.float64, pin_memory=True)
        return s
    s["A"], s["B"] = A, B
    if case.get("layout", "row") == "row":
        s["C"] = A.new_empty((case["m"], case["n"]))
    else:
        s["C"] = A.new_empty((case["n"], case["m"])).t()
    if case["op"] == "auto":
        selector.install_default(s["h"])
    return s


def run(s):
    c, h = s["case"], s["h"]
    if c["op"] == "grouped":
        emu.dgemm_grouped(s["descs"], p=c["p"], handle=h)
        return s["C"]
    if c["op"] == "host":
        return emu.dgemm_host(s["A"], s["B"], s["C"], scheme=c["scheme"],
                              p=c["p"] if c["scheme"] == "I" else 2 * c["p"], handle=h)
    if c["op"] == "auto":
        C, p, code = emu.dgemm_auto(s["A"], s["B"], c["tol"], handle=h, scheme=c["scheme"], C=s["C"])
        return {"C": C, "p": p, "status": code}
    if s["C0"] is not None:
        s["C"].copy_(s["C0"])
    if c["dtype"] == "c128":
        return emu.zgemm(s["A"], s["B"], s["C"], c["alpha"], c["beta"], nm=c["p"], scheme=c["scheme"], handle=h)
    fn = {"f64": emu.dgemm, "f32": emu.sgemm, "c64": emu.cgemm}[c["dtype"]]
    return fn(s["A"], s["B"], s["C"], c["alpha"], c["beta"], scheme=c["scheme"], p=c["p"], handle=h)


_SIZE = {"f64": 8, "f32": 4, "c128": 16, "c64": 8}


def work(case):
    if case["op"] == "grouped":
        shapes = _group_shapes(case)
        return {"bytes": sum(8.0 * (m * k + k * n + m * n) for m, n, k in shapes),
                "flops": sum(2.0 * m * n * k for m, n, k in shapes)}
    m, n, k = case["m"], case["n"], case["k"]
    dt = case.get("dtype", "f64")
    cols = 2 if case.get("beta", 0.0) != 0.0 else 1
    return {"bytes": float(_SIZE[dt]) * (m * k + k * n + cols * m * n),
            "flops": (8.0 if dt in ("c128", "c64") else 2.0) * m * n * k}


def exact(case, seed):
    if case["op"] == "grouped":
        _, _, A, B = _group_inputs(case, seed)
        return torch.cat([(a @ b).reshape(-1) for a, b in zip(A, B)])
    A, B, C0 = _pair(case, seed)
    wide = torch.complex128 if A.is_complex() else torch.float64
    C = A.to(wide) @ B.to(wide)
    if C0 is not None:
        C = case["alpha"] * C + case["beta"] * C0.to(wide)
    elif case["op"] == "gemm":
        C = case["alpha"] * C
    if case["op"] == "auto":
        return {"C": C, "p": None, "status": None}
    return C
