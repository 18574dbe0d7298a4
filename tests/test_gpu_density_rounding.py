"""The FP32 density of one step against the oracle: its sum over the neighbours must not
be rounded at the size of the momentum that whole planes hand over.

A neighbour's part is w (E - q), q = 3 rho c.u less the reference of the target, so that
only the products p = 3 rho c.u are rounded at the size of the momentum.  With u_z = 0.03
p is 0.09, its rounding 2^-27 / sqrt(12) rms, and the ten (D3Q27: eighteen) directions
with a z component leave sqrt(sum w^2) = 0.11 (0.12) of it: 2.6e-10.  The bound is twice
that, for the roundings of the small terms.  (Planes summed whole reach 0.015 in the sum:
14 additions of 2^-30 / sqrt(12) rms, 1e-9.)"""
import numpy as np
import pytest

import oracle
from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Batch, Solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["march", "gather"])
@pytest.mark.parametrize("q,scheme", [(19, "single_step"), (27, "single_step"), (19, "macroscopic")])
def test_density_of_a_step(q, scheme, form):
    nx, ny, nz = 37, 21, 14
    p = W.small_pipe(nx=nx, ny=ny, nz=nz, diameter=12.0, geometry="none", n_mag=1, Ha=1.0, Rm=1e-3, perturb=0.0,
                     Re=0.5 if scheme == "macroscopic" else 100.0, flow_q=q, flow_scheme=scheme, sweep_kernel="split")
    rng = np.random.default_rng(11)
    shape = (nz, ny, nx)
    u = 1e-3 * rng.standard_normal((3,) + shape)
    u[2] += 0.03
    rho = 1e-3 * rng.standard_normal(shape)
    u, rho = u.astype(np.float32).astype(np.float64), 1.0 + rho.astype(np.float32).astype(np.float64)
    o = oracle.Oracle(dict(p, precision="fp64"))
    o.set_state(rho, u, np.zeros_like(u), t=0)
    o.step(1)
    want = o.state()[0]
    if form == "march":
        with Solver(p) as s:
            s.set_state(rho, u, np.zeros_like(u), t=0)
            s.step(1)
            got = s.state()[0]
    else:  # a batch's planes gather
        with Batch([p]) as B:
            B.member(0).set_state(rho, u, np.zeros_like(u), t=0)
            B.step(1)
            got = B.member(0).state()[0]
    assert np.sqrt(np.mean((got - want) ** 2)) <= 5.2e-10
