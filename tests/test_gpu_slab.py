"""The slab kernel (all sweeps of a step in one launch, a slab of planes per
CTA) against the oracle at the sizes where its layout changes: one to five rows
per thread, odd and even widths, one and several planes per CTA, unequal slabs,
both forms of its exchange, its in-plane field.

It carries the applied field's part of the flux apart from that of b; each is a
contracting iteration with a few FP32 roundings of 6e-8 per sweep on terms of the
size of b, so 1e-5 of b is two orders above the rounding."""
import numpy as np
import pytest

import oracle
from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Solver

pytestmark = pytest.mark.gpu


def rel(a, b):
    nb = np.linalg.norm(b)
    return np.linalg.norm(a - b) / nb if nb > 0 else np.linalg.norm(a)


SINGLES = {
    "one_row_one_plane": dict(nx=20, ny=21, nz=1, diameter=14.0),
    "two_planes": dict(nx=21, ny=20, nz=2, diameter=14.0),
    "two_rows": dict(nx=43, ny=41, nz=5, diameter=34.0),
    "three_rows": dict(nx=55, ny=52, nz=4, diameter=46.0),
    "four_rows": dict(nx=71, ny=68, nz=3, diameter=60.0),
    "five_rows": dict(nx=81, ny=75, nz=3, diameter=66.0),
    "two_planes_per_cta": dict(nx=21, ny=22, nz=307, diameter=14.0, b0_kind="tanh", ramp_center=150.0, ramp_width=20.0),
    "three_planes_per_cta": dict(nx=32, ny=31, nz=320, diameter=24.0),
    "uneven_slabs_of_one_and_two": dict(nx=40, ny=38, nz=153, diameter=30.0),
    "in_plane_field": dict(nx=26, ny=25, nz=6, diameter=18.0, b0_kind="field"),
    "in_plane_field_counters": dict(nx=64, ny=62, nz=4, diameter=54.0, b0_kind="field"),
    "odd_periodic": dict(nx=19, ny=16, nz=6, diameter=8.0, geometry="none"),
    "channel": dict(nx=18, ny=21, nz=6, geometry="channel", diameter=15.5, b0_dir=(0.0, 1.0, 0.0)),
    "strict_qs": dict(nx=20, ny=18, nz=4, diameter=12.0, strict_qs=1),
    "accelerated": dict(nx=22, ny=20, nz=5, diameter=14.0, alpha=0.75),
}


@pytest.mark.parametrize("case", sorted(SINGLES))
def test_single_handle_matches_oracle(case):
    kw = dict(SINGLES[case])
    if kw.get("b0_kind") == "field":
        kw["b0_field"] = W.six_magnet_field(kw["nx"], kw["ny"], kw["diameter"])
    p = W.small_pipe(n_mag=21, perturb=0.0, Ha=25.0, Rm=4e-3, **kw)
    z, y, x = np.meshgrid(np.arange(float(p["nz"])), np.arange(float(p["ny"])), np.arange(float(p["nx"])), indexing="ij")
    u = np.stack([0.01 * np.sin(2 * np.pi * y / p["ny"]), 0.02 * np.cos(2 * np.pi * x / p["nx"]),
                  0.03 + 0.01 * np.sin(2 * np.pi * z / p["nz"])])
    o = oracle.Oracle(dict(p, precision="fp64"))
    o.set_state(np.ones_like(x), u, np.zeros_like(u), t=0)
    o.mag_sweeps(40)
    o.step(2)
    with Solver(p) as s:
        assert s.units["sweep_kernel"] == "resident"
        s.set_state(np.ones_like(x), u, np.zeros_like(u), t=0)
        s.mag_sweeps(40)
        s.step(2)
        _, gu, gb = s.state()
    _, ou, ob = o.state()
    assert rel(gu, ou) <= 1e-5 and rel(gb, ob) <= 1e-5, (rel(gu, ou), rel(gb, ob))
