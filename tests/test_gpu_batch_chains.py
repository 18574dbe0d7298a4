"""FP32 batch members off the resident groups sweep in chains of their own kernels, or
jointly when there are more than 24: every member as on its own handle (same
roundings, so to the bit), with different sweep counts, an in-plane field, members
that share a stream, and resident groups beside them."""
import numpy as np
import pytest

from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Batch, Solver

pytestmark = pytest.mark.gpu

LARGE = [
    dict(nx=96, ny=88, nz=50, diameter=80.0, n_mag=6, seed=71),
    dict(nx=85, ny=85, nz=60, diameter=77.0, n_mag=9, b0_kind="tanh", ramp_center=30.0, ramp_width=8.0, seed=72),
    dict(nx=75, ny=77, nz=90, diameter=60.0, n_mag=1, seed=73),
]
OTHERS = {
    "alone": [],
    "with_a_field": [dict(nx=90, ny=90, nz=52, diameter=80.0, n_mag=4, b0_kind="field", seed=74)],
    "with_groups": [dict(nx=24, ny=24, nz=40, diameter=16.0, n_mag=5, seed=75)],
    "with_small_ones": [dict(nx=40, ny=40, nz=20, diameter=30.0, n_mag=8, sweep_kernel="split", seed=76),
                          dict(nx=33, ny=35, nz=12, diameter=24.0, n_mag=3, sweep_kernel="split", seed=77)],
}


@pytest.mark.parametrize("others", sorted(OTHERS))
def test_chains_match_single_handles(others):
    ps = [W.small_pipe(Ha=20.0, Rm=2e-3, **kw) for kw in LARGE + OTHERS[others]]
    for p in ps:
        if p["b0_kind"] == "field":
            p["b0_field"] = W.six_magnet_field(p["nx"], p["ny"], p["diameter"])
    with Batch(ps) as B:
        assert B.info()["launches_per_step"] >= 2 * (6 + 9 + 1)
        steps = 4
        B.step(1)
        B.step(steps - 1)
        got = [B.member(i).state() for i in range(len(ps))]
    for i, p in enumerate(ps):
        with Solver(dict(p, sweep_kernel="split")) as s:
            s.step(steps)
            want = s.state()
        for a, b in zip(got[i], want):
            np.testing.assert_array_equal(a, b, err_msg=str(i))


@pytest.mark.parametrize("count", [20, 24, 25])
def test_many_marching_members(count):
    # more members than streams; as many as take chains; one more, which march jointly
    ps = [W.small_pipe(nx=12 + i % 3, ny=11, nz=3 + i % 4, diameter=7.0, n_mag=2 + i % 5, Ha=20.0, Rm=2e-3, seed=i,
                       sweep_kernel="split") for i in range(count)]
    with Batch(ps) as B:
        chains = sum(2 * p["n_mag"] for p in ps)
        assert (B.info()["launches_per_step"] == chains + 3) == (count <= 24)
        B.step(3)
        got = [B.member(i).state() for i in range(count)]
    for i in (0, 7, count - 1):
        with Solver(ps[i]) as s:
            s.step(3)
            want = s.state()
        for a, b in zip(got[i], want):
            np.testing.assert_array_equal(a, b, err_msg=str(i))
