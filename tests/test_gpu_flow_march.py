"""The marching force and flow kernels against the oracle at the edges of their
tile (32 x 8 columns in FP32, 32 x 4 in FP64): ragged widths and heights, one to
seven planes, both lattices, both density schemes; and the 2-D node-parallel form
past one CTA.

A node's update sums some 30 terms of its neighbours: in FP32 a few roundings of
6e-8 of rho = 1 in drho and of u in m, so 2e-6 of the field is an order above; in
FP64 1e-13 likewise."""
import numpy as np
import pytest

import oracle
from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Solver

pytestmark = pytest.mark.gpu

SHAPES = [(33, 9, 1), (32, 16, 2), (31, 17, 3), (65, 12, 7), (18, 16, 40)]


def check(p, shape, precision):
    rng = np.random.default_rng(7)
    u = 0.02 * rng.standard_normal((3,) + shape)
    b = 0.01 * rng.standard_normal((3,) + shape)
    if p["dim"] == 2:
        u[2] = b[2] = 0.0
    rho = 1.0 + 0.001 * rng.standard_normal(shape)
    if precision == "fp32":
        u, b, rho = (a.astype(np.float32).astype(np.float64) for a in (u, b, rho))
    o = oracle.Oracle(dict(p, precision="fp64"))
    o.set_state(rho, u, b, t=3)
    o.step(1)
    with Solver(dict(p, precision=precision)) as s:
        s.set_state(rho, u, b, t=3)
        s.step(1)
        grho, gu, _ = s.state()
    orho, ou, _ = o.state()
    tol = 2e-6 if precision == "fp32" else 1e-13
    assert np.abs(grho - orho).max() <= tol
    assert np.linalg.norm(gu - ou) <= tol * np.linalg.norm(ou)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("q,scheme", [(19, "single_step"), (27, "single_step"), (19, "macroscopic")])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_flow_step_matches_oracle(shape, q, scheme, precision):
    nx, ny, nz = shape
    # (the macroscopic scheme wants tau >= 1: a low Reynolds number)
    p = W.small_pipe(nx=nx, ny=ny, nz=nz, diameter=float(min(nx, ny) - 3), n_mag=1, Ha=5.0, Rm=1e-2, perturb=0.0,
                     Re=0.5 if scheme == "macroscopic" else 100.0, force_amp=0.2, force_period=50.0, flow_q=q, flow_scheme=scheme, sweep_kernel="split")
    check(p, (nz, ny, nx), precision)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny", [(64, 32), (65, 9)])
def test_2d_flow_step_matches_oracle(nx, ny, precision):
    p = W.hartmann_channel_2d(nx=nx, ny=ny, diameter=float(ny - 1), n_mag=1)
    check(p, (1, ny, nx), precision)
