"""The on-chip solve (each CTA eliminates its rows in shared memory, one grid
barrier, the CTA interface system by parallel cyclic reduction, recovery on
chip; two chained launches, or a cooperative one as Stage 2 of fp32 solves)
against the CPU oracle, at its capacity edges, as the Stage 2 of larger
solves, inside a captured CUDA graph, and with its barrier wait made to run
out for all CTAs or for some."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2501_05938_gb300 import binding, synth

pytestmark = pytest.mark.gpu

F64_FWD, F64_RES = 1e-10, 1e-12
F32_FWD, F32_RES = 1e-5, 1e-5
SMS = 152
CAP = {"f64": SMS * 256 * 23, "f64_df": SMS * 256 * 23, "f32": SMS * 256 * 47,
       "mixed": SMS * 256 * 23}


def solve(plan, s, tdt):
    a, b, c, d = (torch.as_tensor(np.ascontiguousarray(s[k])).to(device="cuda", dtype=tdt)
                  for k in "abcd")
    x = torch.full_like(b, float("nan"))
    plan.solve(a, b, c, d, x)
    torch.cuda.synchronize()
    return x.cpu().numpy().astype(np.float64), plan.query()


def check(dtype, n, seed, expect_onchip):
    s = synth.system(seed, n)
    tdt = torch.float64
    if dtype == "f32":
        s, tdt = synth.to_f32(s), torch.float32
    x, info = solve(binding.Plan(n, dtype=dtype), s, tdt)
    assert info["status"] == 0
    assert info["onchip"] == expect_onchip, info
    a, b, c, d = (np.asarray(s[k], dtype=np.float64) for k in "abcd")
    ref = oracle.thomas(a, b, c, d)
    fwd, res = (F32_FWD, F32_RES) if dtype == "f32" else (F64_FWD, F64_RES)
    assert oracle.rel_forward_error(x, ref) <= fwd
    assert oracle.rel_residual(a, b, c, d, x) <= res
    return x


@pytest.mark.skipif(torch.cuda.is_available() and
                    torch.cuda.get_device_properties(0).multi_processor_count != SMS,
                    reason="capacity figures assume 152 SMs")
@pytest.mark.parametrize("dtype", ["f64", "f64_df", "f32", "mixed"])
def test_capacity_edges(dtype):
    cap = CAP[dtype]
    # the largest system, one more row (a merged one-row tail), then too big
    check(dtype, cap, 11, 1)
    check(dtype, cap + 1, 12, 1)
    check(dtype, cap + 2, 13, 2)


@pytest.mark.parametrize("dtype", ["f64", "f64_df", "f32"])
@pytest.mark.parametrize("n", [65, 66, 100, 769, 770, 1000, 4097, 65537, 300001])
def test_small_and_mid_sizes(dtype, n):
    check(dtype, n, 20 + n, 1)


def test_matches_the_multi_launch_path():
    n = 500001
    s = synth.system(5, n)
    xo, io = solve(binding.Plan(n, dtype="f64"), s, torch.float64)
    xm, im = solve(binding.Plan(n, dtype="f64", flags=binding.NO_ONCHIP), s, torch.float64)
    assert io["onchip"] == 1 and im["onchip"] == 0
    assert oracle.rel_forward_error(xo, xm) <= 1e-14


@pytest.mark.parametrize("dtype", ["f64_df", "f64"])
def test_reduced_system_on_chip(dtype):
    n = (1 << 22) + 3
    g = synth.system_device(31, n)
    for flags in (0, binding.GRAPH):
        x = torch.empty_like(g["b"])
        plan = binding.Plan(n, dtype=dtype, m=128, flags=flags)
        for _ in range(2):  # graph: capture, then replay
            x.zero_()
            plan.solve(g["a"], g["b"], g["c"], g["d"], x)
            torch.cuda.synchronize()
            info = plan.query()
            assert info["status"] == 0 and info["onchip"] == 2
            err = ((x - g["x_true"]).abs().max() / g["x_true"].abs().max()).item()
            assert err <= 1e-12


def test_batched_reduced_system_on_chip():
    sizes = synth.batch_sizes(77, 64, 10, 16)
    off = synth.offsets_from_sizes(sizes)
    n = int(off[-1])
    s = synth.system(78, n, offsets=off)
    a, b, c, d = (torch.as_tensor(s[k]).cuda() for k in "abcd")
    x = torch.empty_like(b)
    plan = binding.Plan(n, dtype="f64_df", batch_max=64, m=32)
    plan.solve_batched(torch.as_tensor(off, device="cuda"), a, b, c, d, x, host_offsets=off)
    torch.cuda.synchronize()
    info = plan.query()
    assert info["status"] == 0 and info["onchip"] == 2
    ref = oracle.thomas_batched(off, s["a"], s["b"], s["c"], s["d"])
    assert oracle.rel_forward_error(x.cpu().numpy(), ref) <= F64_FWD


def test_barrier_timeout_is_reported_and_the_gpu_stays_usable(monkeypatch):
    n = 100003
    s = synth.system(3, n)
    monkeypatch.setenv("TPS_TEST_ONCHIP_TIMEOUT", "1")
    plan = binding.Plan(n, dtype="f64")
    monkeypatch.delenv("TPS_TEST_ONCHIP_TIMEOUT")
    _, info = solve(plan, s, torch.float64)
    assert info["status_name"] == "TPS_ERR_TIMEOUT"
    # the context survives: the next solve on a normal plan is correct
    check("f64", n, 3, 1)


@pytest.mark.parametrize("dtype,n", [
    ("f64_df", 2304), ("f64_df", 2305), ("f64_df", 2306),      # one CTA of 256 blocks, then four
    ("f32", 5888), ("f32", 5889), ("f32", 5890),
    ("f64", 320), ("f64", 448), ("f64", 449), ("f64", 450),    # one CTA of 64 blocks, then two
    ("f64", 152 * 64 * 7), ("f64", 152 * 64 * 7 + 1), ("f64", 152 * 64 * 7 + 2),  # 64 or 128 blocks
    ("f64", 152 * 128 * 45 + 1), ("f64", 152 * 128 * 45 + 2),  # 128 or 256 blocks
    ("f64_df", 769 + 3), ("f64_df", 33 * 3 + 1), ("f32", 95), ("f64", 161),
])
def test_block_and_cta_edges(dtype, n):
    """The rules that choose the block length, the blocks per CTA and one CTA."""
    check(dtype, n, 7 + n, 1)


@pytest.mark.parametrize("dtype,ulp", [("f64", 2.0 ** -53), ("f64_df", 2.0 ** -46),
                                       ("f32", 2.0 ** -24)])
@pytest.mark.parametrize("n", [5000, 20011, 120001])
def test_couplings_that_do_not_decay(dtype, ulp, n):
    """a = c = -1, b = 2 + 1e-4: the couplings of the interface rows fall by
    e^-0.01 a row, so no few strides of the reduction settle them and every
    CTA reduces all of them.  The matrix's condition number is 4e4; a direct
    solve is off by a small multiple of that times the unit roundoff."""
    delta = 1e-4
    rng = np.random.default_rng(n)
    one = np.ones(n)
    a, c, b = -one, -one.copy(), (2.0 + delta) * one
    a[0] = c[-1] = 0.0
    if dtype == "f32":
        b = b.astype(np.float32).astype(np.float64)
    xt = rng.uniform(-1, 1, n)
    d = b * xt
    d[1:] += a[1:] * xt[:-1]
    d[:-1] += c[:-1] * xt[1:]
    s = {"a": a, "b": b, "c": c, "d": d}
    tdt = torch.float64
    if dtype == "f32":
        s, tdt = synth.to_f32(s), torch.float32
    x, info = solve(binding.Plan(n, dtype=dtype), s, tdt)
    assert info["status"] == 0 and info["onchip"] == 1, info
    ref = oracle.thomas(*(np.asarray(s[k], dtype=np.float64) for k in "abcd"))
    assert oracle.rel_forward_error(x, ref) <= 16 * (4.0 / delta) * ulp


@pytest.mark.parametrize("dtype", ["f64", "f64_df", "f32"])
@pytest.mark.parametrize("n", [6000, 100003, 800001])
def test_ctas_that_gave_up_are_done_again(dtype, n, monkeypatch):
    """The barrier waits for one CTA more than there are, so every CTA gives up
    and the second launch does it again; a solve after it, undisturbed, finds
    the counters as they should be."""
    monkeypatch.setenv("TPS_TEST_ONCHIP_GIVE_UP", "1")
    plan = binding.Plan(n, dtype=dtype)
    monkeypatch.delenv("TPS_TEST_ONCHIP_GIVE_UP")
    s = synth.system(33 + n, n)
    tdt = torch.float64
    if dtype == "f32":
        s, tdt = synth.to_f32(s), torch.float32
    x0, info0 = solve(binding.Plan(n, dtype=dtype), s, tdt)
    for _ in range(2):
        x, info = solve(plan, s, tdt)
        assert info["status"] == 0 and info["onchip"] == 1, info
        assert np.array_equal(x, x0)


@pytest.mark.parametrize("dtype,n", [("f64", 10007), ("f64_df", 40009), ("f64_df", 800001),
                                     ("f32", 40009), ("f32", 1000003)])
def test_barrier_that_opened_early(dtype, n, monkeypatch):
    """A count left at the barrier (by two solves on one plan at once, a misuse)
    lets CTAs read interface rows that others are still writing.  That solve
    is spoiled, but its warps stay together, the context survives, and the plan's
    next solve finds nothing of it."""
    monkeypatch.setenv("TPS_TEST_ONCHIP_RESIDUE", "1")
    plan = binding.Plan(n, dtype=dtype)
    monkeypatch.delenv("TPS_TEST_ONCHIP_RESIDUE")
    tdt = torch.float32 if dtype == "f32" else torch.float64
    one = np.ones(n)
    s = {"a": -one, "b": 2.01 * one, "c": -one.copy()}  # every CTA needs the others' rows
    rng = np.random.default_rng(n)
    for k in range(12):
        s["d"] = rng.uniform(-1, 1, n)
        x, info = solve(plan, s, tdt)
        if k > 0:
            x0, _ = solve(binding.Plan(n, dtype=dtype), s, tdt)
            assert info["status"] == 0 and info["onchip"] == 1, info
            assert np.array_equal(x, x0)


@pytest.mark.parametrize("dtype", ["f64", "f64_df", "f32"])
@pytest.mark.parametrize("n", [500, 6000, 10007, 100003, 800001])
def test_some_ctas_gave_up(dtype, n, monkeypatch):
    """Every second CTA gives up: some rows come from the first launch, some from
    the second, whose CTAs share them."""
    monkeypatch.setenv("TPS_TEST_ONCHIP_GIVE_UP", "2")
    plan = binding.Plan(n, dtype=dtype)
    monkeypatch.delenv("TPS_TEST_ONCHIP_GIVE_UP")
    s = synth.system(34 + n, n, kind=synth.KIND_RATIO, ratio=1.1)
    tdt = torch.float64
    if dtype == "f32":
        s, tdt = synth.to_f32(s), torch.float32
    x0, info0 = solve(binding.Plan(n, dtype=dtype), s, tdt)
    for _ in range(2):
        x, info = solve(plan, s, tdt)
        assert info["status"] == 0 and info["onchip"] == 1, info
        assert np.array_equal(x, x0)
