"""The planner's choice between the slab kernel and the split sweep, where one plane
per CTA does not fit: by what each costs on the domain, which for slabs depends on
the rows per thread and for the split sweep on how the planes fill the device."""
import pytest

from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Solver

pytestmark = pytest.mark.gpu

# measured slab / split, us per sweep (or per step of n_mag sweeps), on 152 SMs
SPLIT = [
    dict(nx=57, ny=57, nz=245),                                # 16.6 / 15.1
    dict(nx=57, ny=57, nz=153),                                # 16.4 / 11.6
    dict(nx=55, ny=55, nz=200),                                # 15.4 / 12.7
    dict(nx=54, ny=54, nz=153),                                # 13.5 / 9.8
    dict(nx=53, ny=53, nz=200, geometry="none"),               # 11.6 / 8.8
    dict(nx=59, ny=59, nz=245, geometry="none"),               # 13.6 / 10.4
    dict(nx=37, ny=37, nz=153, geometry="none"),               # 6.3 / 5.4
    dict(nx=20, ny=300, nz=40, b0_kind="field", diameter=12.0),  # 13.2 / 8.4
    dict(nx=55, ny=55, nz=200, b0_kind="field"),               # 15.4 / 14.1
    dict(nx=40, ny=40, nz=192, n_mag=3),                       # 73 / 49 a step
    dict(nx=24, ny=24, nz=300, n_mag=1),                       # 32 / 22 a step
    dict(nx=64, ny=64, nz=128, n_mag=1, b0_kind="field"),      # 62 / 41 a step
]
SLAB = [
    dict(nx=54, ny=54, nz=304),                                # 13.6 / 15.1
    dict(nx=53, ny=53, nz=304),                                # 13.7 / 16.2
    dict(nx=41, ny=41, nz=200),                                # 8.6 / 9.9
    dict(nx=40, ny=40, nz=192),                                # 7.7 / 8.5
    dict(nx=32, ny=32, nz=400),                                # 7.0 / 8.7
    dict(nx=24, ny=24, nz=300),                                # 2.9 / 6.2
    dict(nx=24, ny=24, nz=300, geometry="none"),               # 2.1 / 3.3
    dict(nx=64, ny=64, nz=128, b0_kind="field"),               # 7.1 / 10.8
    dict(nx=24, ny=24, nz=300, n_mag=24),
    dict(nx=40, ny=40, nz=192, n_mag=40),
]


@pytest.mark.parametrize("kw,slab", [(k, False) for k in SPLIT] + [(k, True) for k in SLAB], ids=str)
def test_route_by_cost(kw, slab):
    import torch

    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the cases' fill is counted for 152 SMs")
    kw = dict(dict(n_mag=270, diameter=float(min(kw["nx"], kw["ny"]) - 8)), **kw)
    if kw.get("b0_kind") == "field":
        kw["b0_field"] = W.six_magnet_field(kw["nx"], kw["ny"], kw["diameter"])
    with Solver(W.small_pipe(**kw)) as s:
        plan = s.plan()
    assert (plan["kernel"] == "k_sweeps_slab") == slab, plan
