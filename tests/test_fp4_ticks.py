"""A CPU model of the step kernel's stochastic E2M1 encode (e2m1_sr_ticks in
step_kernel.cuh): when s and s + ticks agree above bit 22, s >> 22 is the code
of every value of the interval.  Against the oracle's exact rule (and that
against the oracle itself), at random bits beside the decision, at the grid's
edges, near zero and past the saturation point."""
import numpy as np
import pytest

import oracle

F32, U32, F64 = np.float32, np.uint32, np.float64


def exact_code(x, r):
    """Magnitude code of x >= 0 (float64 holding binary32 values) with 32 random bits r, as the format defines it."""
    grid = np.array([0, 0.5, 1, 1.5, 2, 3, 4, 6], F64)
    a = np.minimum(x, 6.0)
    i = np.minimum(np.searchsorted(grid, a, side="right") - 1, 6)
    frac = (a - grid[i]) / (grid[i + 1] - grid[i])
    return i + (r.astype(F64) < np.floor(frac * 4294967296.0))


def kernel_ticks(xm, r):
    """e2m1_sr_ticks, operation by operation, in wrapping 32-bit words."""
    a = np.minimum(xm, F32(6.0))
    sub = a < F32(1.0)
    f = (a.astype(F64) + 1.0).astype(F32)  # 1 + a rounded down: step back where the rounded sum lies above it
    down = np.where(f.astype(F64) - 1.0 > a.astype(F64), np.nextafter(f, F32(0.0)), f)
    z = np.where(sub, down, a).view(U32)
    k = np.where(sub, U32((0x003FFFFF - 0x3F800000) & 0xFFFFFFFF),
                 U32((0x003FFFFF - 0x3F000000) & 0xFFFFFFFF))
    return z + k - (r >> U32(10))


def intervals(rng, n):
    """Smaller ends, widths in ticks and random bits."""
    edges = np.array([0, 0.5, 1, 1.5, 2, 3, 4, 5, 6, 8], F32)
    kind = rng.integers(0, 4, n)
    ends = np.where(kind == 0, rng.uniform(0, 8, n),
                    np.where(kind == 1, np.exp2(rng.uniform(-140, 0, n)),
                             rng.choice(edges, n) + rng.normal(0, 1, n) * np.exp2(rng.uniform(-26, -6, n))))
    xm = np.maximum(ends, 2.0 ** -149).astype(F32)
    ticks = np.where(rng.random(n) < 0.5, 264, np.ceil(260 + np.exp2(rng.uniform(1, 21, n)))).astype(U32)
    grid = np.array([0, 0.5, 1, 1.5, 2, 3, 4, 6], F64)
    a = np.minimum(xm.astype(F64), 5.9999995)
    i = np.searchsorted(grid, a, side="right") - 1
    thr = np.floor((a - grid[i]) / (grid[i + 1] - grid[i]) * 4294967296.0)
    near = thr + np.round(rng.normal(0, 1, n) * np.exp2(rng.uniform(0, 24, n)))
    r = np.where(rng.random(n) < 0.8, np.clip(near, 0, 4294967295), rng.integers(0, 1 << 32, n)).astype(U32)
    return xm, ticks, r


def test_model_of_the_exact_rule():
    rng = np.random.default_rng(1)
    xm, _, r = intervals(rng, 20000)
    assert (exact_code(xm.astype(F64), r) == (oracle.e2m1_sr(xm, r) & 7)).all()


@pytest.mark.parametrize("seed", range(4))
def test_certified_codes_hold_over_the_interval(seed):
    rng = np.random.default_rng(seed)
    xm, ticks, r = intervals(rng, 1 << 20)
    with np.errstate(over="ignore"):
        s = kernel_ticks(xm, r)
        sure = ((s ^ (s + ticks)) >> U32(22)) == 0
    code = (s >> U32(22)) & U32(7)
    width = (ticks.astype(F64) - 3.0) / 2.0 ** 23  # ticks >= (xM - xm) 2^23 + 3
    assert 0.2 < sure.mean() < 0.95  # the sample lies beside the decision, not all on one side of it
    for part in (0.0, rng.random(xm.size), 1.0):
        top = xm.astype(F64) + width * part
        x = top.astype(F32)
        x = np.where(x.astype(F64) > top, np.nextafter(x, F32(0.0)), x)  # inside the interval
        assert (exact_code(x.astype(F64), r)[sure] == code[sure]).all()
