"""The FP32 sweep on node pairs (one sweep per launch) against the oracle at the
edges of its tile: 32 x 16 nodes, a pair wide and two rows high per thread, odd
widths (8-byte pairs not aligned) and heights, one to three planes, a chunk's end.

A sweep is a contracting iteration with a few FP32 roundings of 6e-8 on terms of
the size of b and, where the applied field enters the flux, of 1: 1e-5 of b is two
orders above the rounding."""
import numpy as np
import pytest

import oracle
from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Solver

pytestmark = pytest.mark.gpu

SHAPES = [(32, 16, 4), (33, 17, 1), (31, 15, 2), (34, 31, 3), (63, 33, 5), (65, 32, 3), (17, 64, 2), (9, 9, 61)]


@pytest.mark.parametrize("field", ["uniform", "field"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_pair_sweep_matches_oracle(shape, field):
    nx, ny, nz = shape
    d = float(min(nx, ny) - 3)
    kw = dict(b0_field=W.six_magnet_field(nx, ny, d)) if field == "field" else {}
    p = W.small_pipe(nx=nx, ny=ny, nz=nz, diameter=d, b0_kind=field, n_mag=7, perturb=0.0, Ha=25.0, Rm=4e-3,
                     sweep_kernel="split", **kw)
    z, y, x = np.meshgrid(np.arange(float(nz)), np.arange(float(ny)), np.arange(float(nx)), indexing="ij")
    u = np.stack([0.01 * np.sin(2 * np.pi * y / ny), 0.02 * np.cos(2 * np.pi * x / nx),
                  0.03 + 0.01 * np.sin(2 * np.pi * z / nz)])
    rng = np.random.default_rng(5)
    b = 1e-3 * rng.standard_normal(u.shape)
    o = oracle.Oracle(dict(p, precision="fp64"))
    o.set_state(np.ones_like(x), u, b, t=0)
    o.mag_sweeps(5)
    with Solver(p) as s:
        assert s.units["sweep_kernel"] == "split"
        s.set_state(np.ones_like(x), u, b, t=0)
        s.mag_sweeps(5)
        gb = s.state()[2]
    ob = o.state()[2]
    assert np.linalg.norm(gb - ob) <= 1e-5 * np.linalg.norm(ob)
