"""The FP64 resident sweep kernels against the oracle at the sizes where their
layouts change: the 2-D cluster kernel (bands of rows over the CTAs of one
cluster: fewer rows than CTAs, one row, short and empty last bands, several
nodes per thread, markers between two bands) and the 3-D plane kernel (one to
five nodes per thread, one and two planes).

Tolerance 1e-12 (FP64 path): both evaluate the sweep with fused multiply-adds
in another order than the oracle, a few roundings of 1.1e-16 per sweep on a
contracting iteration."""
import numpy as np
import pytest

import oracle
from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Solver

pytestmark = pytest.mark.gpu

TOL = 1e-12


def rel(a, b):
    nb = np.linalg.norm(b)
    return np.linalg.norm(a - b) / nb if nb > 0 else np.linalg.norm(a)


def check(p, steps, kernel="resident"):
    o = oracle.Oracle(p)
    with Solver(dict(p, sweep_kernel=kernel)) as s:
        assert s.units["sweep_kernel"] == kernel
        s.step(steps)
        s.mag_sweeps(3)
        got = s.state()
    o.step(steps)
    o.mag_sweeps(3)
    for a, b in zip(got, o.state()):
        assert rel(a, b) <= TOL


PLANES = {
    "one_row": dict(nx=40, ny=1, geometry="none"),
    "three_rows": dict(nx=21, ny=3, geometry="none"),
    "fewer_rows_than_ctas": dict(nx=16, ny=11, diameter=6.5),
    "short_last_band": dict(nx=19, ny=17, diameter=12.5),
    "empty_bands": dict(nx=24, ny=33, diameter=27.3),
    "walls_on_nodes": dict(nx=64, ny=32, diameter=31.0),
    "several_nodes_per_thread": dict(nx=131, ny=61, diameter=52.6),
    "ring": dict(nx=35, ny=38, geometry="pipe", diameter=25.0),
}


@pytest.mark.parametrize("case", sorted(PLANES))
def test_cluster_kernel_matches_oracle(case):
    p = W.hartmann_channel_2d(**dict(dict(n_mag=37, perturb=0.02, seed=3, diameter=8.0, Ha=6.0), **PLANES[case]))
    check(p, 3)


BOXES = {
    "one_node_per_thread": dict(nx=17, ny=19, nz=5, diameter=12.0),
    "one_plane": dict(nx=24, ny=22, nz=1, diameter=16.0),
    "two_planes": dict(nx=24, ny=22, nz=2, diameter=16.0),
    "four_nodes_per_thread": dict(nx=58, ny=57, nz=3, diameter=50.0),
    "five_nodes_per_thread": dict(nx=67, ny=65, nz=2, geometry="none"),
    "ramp": dict(nx=33, ny=30, nz=6, diameter=24.0, b0_kind="tanh", ramp_center=3.0, ramp_width=1.5),
    "strict_qs": dict(nx=20, ny=18, nz=4, diameter=12.0, strict_qs=1),
}


@pytest.mark.parametrize("case", sorted(BOXES))
def test_plane_kernel_matches_oracle(case):
    check(W.small_pipe(precision="fp64", n_mag=25, **BOXES[case]), 3)


@pytest.mark.parametrize("case", ["4096_nodes", "above_4096_nodes"])
def test_planes_at_the_limit_of_shared_memory(case):
    # the IB tables in 16 bits, eight and nine or ten nodes per thread
    n = dict(zip(["4096_nodes", "above_4096_nodes"], [(64, 64), (65, 65)]))[case]
    check(W.small_pipe(nx=n[0], ny=n[1], nz=3, diameter=n[0] - 8.0, n_mag=9, precision="fp64", Ha=20.0, Rm=2e-3), 2)
