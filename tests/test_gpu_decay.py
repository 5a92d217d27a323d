"""Terms that decay along a block: what is left out once they are small must
not be missed by any unknown, judged per system and per component, not in the
norm of the whole array."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2501_05938_gb300 import binding

pytestmark = pytest.mark.gpu

ULP = {"f64": 2.0 ** -53, "f64_df": 2.0 ** -46, "f32": 2.0 ** -24}


def toeplitz(n, b):
    """a = c = -1 and a constant diagonal."""
    one = np.ones(n)
    return {"a": -one, "b": b * one, "c": -one.copy()}


def multiply(s, x):
    d = s["b"] * x
    d[1:] += s["a"][1:] * x[:-1]
    d[:-1] += s["c"][:-1] * x[1:]
    return d


def make_plan(n, dtype, checkpoints, monkeypatch, **kw):
    monkeypatch.setenv("TPS_TEST_CHECKPOINTS", "1" if checkpoints else "0")
    plan = binding.Plan(n, dtype=dtype, **kw)
    monkeypatch.delenv("TPS_TEST_CHECKPOINTS")
    return plan


def to_device(s, dtype):
    tdt = torch.float32 if dtype == "f32" else torch.float64
    return [torch.as_tensor(np.ascontiguousarray(s[k])).to("cuda", tdt) for k in "abcd"]


@pytest.mark.parametrize("checkpoints", [False, True])
@pytest.mark.parametrize("dtype", ["f64", "f64_df", "f32"])
@pytest.mark.parametrize("b", [2.2, 4.0])
@pytest.mark.parametrize("cut", [249, 255, 256, 3])
def test_packed_systems_do_not_couple(dtype, checkpoints, b, cut, monkeypatch):
    """Two systems whose solutions lie 1e10 (fp32: 1e15) apart, the boundary
    `cut` rows into a block, either one first: the error of each is that of
    its own solve (condition number (b + 2) / (b - 2), the constant 16 for the
    roundings of a row), and one whose right-hand side is zero is exactly 0."""
    m, big = 256, 1e15 if dtype == "f32" else 1e10
    off = np.array([0, 5 * m + cut, 12 * m + 40], dtype=np.int64)
    n = int(off[-1])
    cond = (b + 2.0) / (b - 2.0)
    for first, second in ((1.0, big), (big, 1.0), (0.0, big), (big, 0.0)):
        s = toeplitz(n, b)
        if dtype == "f32":
            s = {k: v.astype(np.float32).astype(np.float64) for k, v in s.items()}
        s["a"][off[:-1]] = s["c"][off[1:] - 1] = 0.0
        xt = np.random.default_rng(cut).uniform(-1, 1, n)
        xt[:off[1]] *= first
        xt[off[1]:] *= second
        s["d"] = multiply(s, xt)
        if dtype == "f32":
            s["d"] = s["d"].astype(np.float32).astype(np.float64)
        ref = oracle.thomas_batched(off, *(s[k] for k in "abcd"))
        plan = make_plan(n, dtype, checkpoints, monkeypatch, m=m, batch_max=2,
                         flags=binding.NO_ONCHIP)
        a, bb, c, d = to_device(s, dtype)
        x = torch.full_like(bb, float("nan"))
        plan.solve_batched(torch.as_tensor(off, device="cuda"), a, bb, c, d, x, host_offsets=off)
        torch.cuda.synchronize()
        assert plan.query()["status"] == 0
        x = x.double().cpu().numpy()
        for lo, hi, size in ((0, off[1], first), (off[1], n, second)):
            err = np.abs(x[lo:hi] - ref[lo:hi]).max()
            assert err <= 16 * cond * ULP[dtype] * np.abs(ref[lo:hi]).max(), (first, second, size)


# How far below the impulse a component keeps its relative accuracy: native
# fp64 to the format's end; double-float as long as a relation's pair is normal
# (2^-126 with 24 bits of its low part below), fp32 as long as the value is.
DEEP = {"f64": 2.0 ** -950, "f64_df": 2.0 ** -98, "f32": 2.0 ** -120}


def impulse_error(x, ref, peak, dtype):
    """Largest relative error among the components down to DEEP of the peak."""
    use = np.abs(ref) >= DEEP[dtype] * peak
    return (np.abs(x - ref)[use] / np.abs(ref)[use]).max()


@pytest.mark.parametrize("checkpoints", [False, True])
@pytest.mark.parametrize("dtype", ["f64", "f64_df", "f32"])
@pytest.mark.parametrize("m,tail,at", [(256, 0, 0), (256, 0, 1), (256, 0, 17), (256, 0, 100),
                                       (256, 0, 255), (250, 57, 3), (1000, 1, 0), (123, 40, 122)])
def test_impulse_is_resolved_far_below_its_peak(dtype, checkpoints, m, tail, at, monkeypatch):
    """One nonzero entry in d, `at` rows into a block: x falls by 2 + sqrt(3) a
    row on either side, with no cancellation anywhere, so every component has
    a small relative error (a few roundings a row: 4 n ulp with n the rows it
    has come).  Native fp64 is held to it downwards of the impulse; upwards it
    leaves out what reaches a block's first unknown over more than 2^-60."""
    n = m * 40 + tail
    s = toeplitz(n, 4.0)
    row, peak = 11 * m + at, 2.0 ** 60
    s["d"] = np.zeros(n)
    s["d"][row] = peak
    ref = oracle.thomas(*(s[k] for k in "abcd"))
    plan = make_plan(n, dtype, checkpoints, monkeypatch, m=m, flags=binding.NO_ONCHIP)
    a, b, c, d = to_device(s, dtype)
    x = torch.full_like(b, float("nan"))
    plan.solve(a, b, c, d, x)
    torch.cuda.synchronize()
    assert plan.query()["status"] == 0
    x = x.double().cpu().numpy()
    if dtype == "f64":
        up = ref[:row] >= 2.0 ** -50 * peak
        assert (np.abs(x - ref)[:row][up] <= 2.0 ** -44 * ref[:row][up]).all()
        x, ref = x[row:], ref[row:]
    assert impulse_error(x, ref, peak, dtype) <= 2048 * ULP[dtype]


@pytest.mark.parametrize("dtype,n", [("f64", 5000), ("f64", 20011), ("f64_df", 5000),
                                     ("f64_df", 100003), ("f32", 20011), ("f32", 300007)])
def test_impulse_on_chip(dtype, n):
    """The same on chip, where the interface rows of the CTAs around decide."""
    s = toeplitz(n, 4.0)
    peak = 2.0 ** 60
    for row in (n // 2, n // 3 + 5, 0, n - 1):
        s["d"] = np.zeros(n)
        s["d"][row] = peak
        ref = oracle.thomas(*(s[k] for k in "abcd"))
        plan = binding.Plan(n, dtype=dtype)
        a, b, c, d = to_device(s, dtype)
        x = torch.full_like(b, float("nan"))
        plan.solve(a, b, c, d, x)
        torch.cuda.synchronize()
        info = plan.query()
        assert info["status"] == 0 and info["onchip"] == 1, info
        assert impulse_error(x.double().cpu().numpy(), ref, peak, dtype) <= 2048 * ULP[dtype]
