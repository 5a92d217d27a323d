"""The calls a user of this solver makes, as measurable cases.

Every case is a strictly diagonally dominant tridiagonal system (or a packed
batch of them) solved through a public entry point:

  solve    Plan.solve          one device-resident system
  batch    Plan.solve_batched  packed device-resident systems, one graph launch
  host     Plan.solve_host_async  one system in pinned host memory
  noalloc  tps_solve_noalloc   one device-resident system, no plan

Systems: a, c ~ U(-1, 1); b = |a| + |c| + U(1, 2), or for "ratio" > 0
b = ratio * max(|a| + |c|, 2^-20); d = A x_true with x_true ~ U(-1, 1).
All sizes are rows; fp64 arrays except dtype "f32".
"""
import ctypes
import math

import numpy as np
import torch

from paper_2501_05938_gb300 import binding

DEVICE = "cuda"


def listed():
    return [
        # the smallest ordinary call: a 1-D line of a small grid, latency only
        {"name": "solve_df_1k", "kind": "solve", "dtype": "f64_df", "n": 1000, "ratio": 0.0},
        # a caller that cannot allocate, inside a latency-bound loop
        {"name": "noalloc_f64_10k", "kind": "noalloc", "dtype": "f64", "n": 10007, "ratio": 0.0},
        # the plain method's small system (256 blocks of 256 rows)
        {"name": "solve_f64_65536", "kind": "solve", "dtype": "f64", "n": 65536, "ratio": 0.0},
        # mid sizes, which fit in the GPU's shared memory; odd and even
        {"name": "solve_df_800k", "kind": "solve", "dtype": "f64_df", "n": 800000, "ratio": 0.0},
        {"name": "solve_f32_1m", "kind": "solve", "dtype": "f32", "n": 1000003, "ratio": 0.0},
        # just past shared memory, ragged, weakly dominant
        {"name": "solve_df_3m_weak", "kind": "solve", "dtype": "f64_df", "n": 3000017,
         "ratio": 1.1},
        # the headline system, and the plain method at large size
        {"name": "solve_df_2p27", "kind": "solve", "dtype": "f64_df", "n": 1 << 27, "ratio": 0.0},
        {"name": "solve_f64_100m", "kind": "solve", "dtype": "f64", "n": 100000000, "ratio": 0.0},
        # uneven batches: the full one, and an ordinary one in single precision
        {"name": "batch_df_4096", "kind": "batch", "dtype": "f64_df", "count": 4096, "lo": 8.0,
         "hi": 20.0, "sizes_seed": 1004, "ratio": 0.0},
        {"name": "batch_f32_256", "kind": "batch", "dtype": "f32", "count": 256, "lo": 8.0,
         "hi": 17.0, "sizes_seed": 1005, "ratio": 0.0},
        # mixed-precision refinement of a batch of weakly dominant systems
        {"name": "batch_mixed_1024", "kind": "batch", "dtype": "mixed", "count": 1024, "lo": 10.0,
         "hi": 18.0, "sizes_seed": 1006, "ratio": 1.01},
        # a system that lives in host memory: upload, solve, download
        {"name": "host_df_2p24", "kind": "host", "dtype": "f64_df", "n": 1 << 24, "ratio": 0.0},
    ]


def _log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "batch", "host", "noalloc"])
    ratio = rng.choice([0.0, 0.0, 1.01, 1.1, 2.0])
    if kind == "solve":
        dtype = rng.choice(["f64_df", "f64_df", "f64", "f32", "mixed"])
        return {"kind": kind, "dtype": dtype, "n": _log_uniform(rng, 300, 1.3e8), "ratio": ratio}
    if kind == "batch":
        dtype = rng.choice(["f64_df", "f64", "f32", "mixed"])
        lo = rng.uniform(8.0, 10.0)
        return {"kind": kind, "dtype": dtype, "count": _log_uniform(rng, 16, 2000), "lo": lo,
                "hi": rng.uniform(lo + 1.0, 18.0), "sizes_seed": rng.randrange(1 << 30),
                "ratio": ratio}
    if kind == "host":
        return {"kind": kind, "dtype": rng.choice(["f64_df", "f64", "f32"]),
                "n": _log_uniform(rng, 1 << 16, 1 << 25), "ratio": ratio}
    return {"kind": kind, "dtype": rng.choice(["f64_df", "f64", "f32"]),
            "n": _log_uniform(rng, 300, 262144), "ratio": ratio}


def _offsets(case):
    """count + 1 offsets of a batch: sizes log-uniform in [2^lo, 2^hi]."""
    u = np.random.default_rng(case["sizes_seed"]).random(case["count"])
    sizes = np.floor(np.exp2(case["lo"] + (case["hi"] - case["lo"]) * u)).astype(np.int64)
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def _rows(case):
    return int(_offsets(case)[-1]) if case["kind"] == "batch" else case["n"]


def _system(case, seed):
    """a, b, c, d on the GPU in the case's I/O type; couplings that leave a
    system are zero."""
    n = _rows(case)
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)

    def uniform():
        return torch.rand(n, dtype=torch.float64, device=DEVICE, generator=g)

    a = uniform().mul_(2.0).sub_(1.0)
    c = uniform().mul_(2.0).sub_(1.0)
    if case["kind"] == "batch":
        off = torch.as_tensor(_offsets(case), device=DEVICE)
        a[off[:-1]] = 0.0
        c[off[1:] - 1] = 0.0
    a[0] = 0.0
    c[-1] = 0.0
    b = a.abs().add_(c.abs())
    if case["ratio"] > 0.0:
        b.clamp_(min=2.0 ** -20).mul_(case["ratio"])
    else:
        b.add_(uniform()).add_(1.0)
    x = uniform().mul_(2.0).sub_(1.0)
    d = b * x
    d[1:].addcmul_(a[1:], x[:-1])
    d[:-1].addcmul_(c[:-1], x[1:])
    if case["dtype"] == "f32":
        a, b, c, d = (t.float() for t in (a, b, c, d))
    return a, b, c, d


def prepare(case, seed):
    n = _rows(case)
    a, b, c, d = _system(case, seed)
    kind, dtype = case["kind"], case["dtype"]
    if kind == "host":
        arrays = []
        for t in (a, b, c, d):
            h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
            h.copy_(t)
            arrays.append(h)
        x = torch.empty(n, dtype=b.dtype, pin_memory=True)
        plan = binding.Plan(n, dtype=dtype, residency="host", flags=binding.TUNE_PREDICT)
        return {"kind": kind, "plan": plan, "args": (*arrays, x)}
    x = torch.empty_like(b)
    state = {"kind": kind, "args": (a, b, c, d, x)}
    if kind == "solve":
        state["plan"] = binding.Plan(n, dtype=dtype)
    elif kind == "batch":
        off = _offsets(case)
        state["plan"] = binding.Plan(n, dtype=dtype, batch_max=case["count"],
                                     flags=binding.TUNE_PREDICT | binding.GRAPH)
        state["host_offsets"] = off
        state["offsets"] = torch.as_tensor(off, device=DEVICE)
    else:
        fn = binding.lib().tps_solve_noalloc
        fn.argtypes = [ctypes.c_int32, ctypes.c_int64] + [ctypes.c_void_p] * 7
        fn.restype = ctypes.c_int
        state["fn"] = fn
        state["status"] = torch.zeros(1, dtype=torch.int32, device=DEVICE)
        state["dtype"] = binding.DTYPES[dtype]
    return state


def run(state):
    a, b, c, d, x = state["args"]
    kind = state["kind"]
    if kind == "solve":
        return state["plan"].solve(a, b, c, d, x)
    if kind == "batch":
        return state["plan"].solve_batched(state["offsets"], a, b, c, d, x,
                                           host_offsets=state["host_offsets"])
    if kind == "host":
        return state["plan"].solve_host_async(a, b, c, d, x)
    binding.check(state["fn"](state["dtype"], b.numel(), a.data_ptr(), b.data_ptr(), c.data_ptr(),
                              d.data_ptr(), x.data_ptr(), state["status"].data_ptr(),
                              torch.cuda.current_stream().cuda_stream), "tps_solve_noalloc")
    return {"x": x, "status": state["status"]}


def work(case):
    n = _rows(case)
    size = 4 if case["dtype"] == "f32" else 8
    extra = 8 * (case["count"] + 1) if case["kind"] == "batch" else 0
    # Thomas: 3 multiplications, 3 subtractions, 2 divisions a row, and a
    # multiplication and a subtraction on the way back
    return {"bytes": 5 * size * n + extra, "flops": 8 * n}


def tolerance(case):
    """About four times what each arithmetic differs from exact() over
    n = 3000 .. 5000001 and the dominance ratios of these cases.  "f64_df"
    carries about 46 bits, "mixed" is refined to fp64.  A weaker dominance
    conditions the rows with the smallest diagonals worse, which shows in
    the largest difference far more than in the 2-norm."""
    unit = {"f64": 1e-15, "mixed": 1e-15, "f64_df": 2.8e-14, "f32": 2.8e-7}[case["dtype"]]
    norm, most = {0.0: (1, 8), 2.0: (1, 8), 1.1: (2, 64), 1.01: (5, 480)}[case["ratio"]]
    return {"rel": norm * unit, "max": most * unit}


def exact(case, seed):
    """Parallel cyclic reduction in fp64 (Hockney 1965), stopped once no
    coupling is left."""
    a, b, c, d = (t.double() for t in _system(case, seed))
    n = b.numel()
    a[0] = 0.0
    c[-1] = 0.0
    s = 1
    while s < n:
        lo = a[s:] / b[:-s]
        up = c[:-s] / b[s:]
        nb, nd = b.clone(), d.clone()
        nb[s:] -= lo * c[:-s]
        nb[:-s] -= up * a[s:]
        nd[s:] -= lo * d[:-s]
        nd[:-s] -= up * d[s:]
        na, nc = torch.zeros_like(a), torch.zeros_like(c)
        na[s:] = -lo * a[:-s]
        nc[:-s] = -up * c[s:]
        del lo, up
        a, b, c, d = na, nb, nc, nd
        s *= 2
        if max(float((a / b).abs().max()), float((c / b).abs().max())) < 1e-40:
            break
    x = d / b
    if case["kind"] == "host":
        x = x.cpu()
    if case["kind"] == "noalloc":
        return {"x": x, "status": torch.zeros(1, dtype=torch.int32)}
    return x
