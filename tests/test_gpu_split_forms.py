"""The two forms of the FP32 pair sweep: a row a thread on small domains, two on
large ones, each against the oracle at the edges of its tile (32 x 8 and 32 x 16
nodes; test_gpu_pair_sweep.py's shapes are small ones), and the plan that chooses
between them: a domain that does not fill the device is cut into short chunks, so
that a CTA's planes, one after the other, do not set the time.

Tolerance as in test_gpu_pair_sweep.py: a contracting iteration with a few FP32
roundings of 6e-8 per sweep."""
import numpy as np
import pytest

import oracle
from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Solver

pytestmark = pytest.mark.gpu

ONE = [(32, 8, 4), (31, 9, 2), (34, 23, 3), (65, 24, 1)]
TWO = [(33, 17, 420), (63, 33, 330), (34, 31, 500), (64, 32, 440), (9, 9, 1900)]


@pytest.mark.parametrize("field", ["uniform", "field"])
@pytest.mark.parametrize("shape,rows", [(s, 1) for s in ONE] + [(s, 2) for s in TWO], ids=str)
def test_form_matches_oracle(shape, rows, field):
    nx, ny, nz = shape
    d = float(min(nx, ny) - 3)
    kw = dict(b0_field=W.six_magnet_field(nx, ny, d)) if field == "field" else {}
    p = W.small_pipe(nx=nx, ny=ny, nz=nz, diameter=d, b0_kind=field, n_mag=7, perturb=0.0, Ha=25.0, Rm=4e-3,
                     sweep_kernel="split", **kw)
    z, y, x = np.meshgrid(np.arange(float(nz)), np.arange(float(ny)), np.arange(float(nx)), indexing="ij")
    u = np.stack([0.01 * np.sin(2 * np.pi * y / ny), 0.02 * np.cos(2 * np.pi * x / nx),
                  0.03 + 0.01 * np.sin(2 * np.pi * z / nz)])
    b = 1e-3 * np.random.default_rng(5).standard_normal(u.shape)
    o = oracle.Oracle(dict(p, precision="fp64"))
    o.set_state(np.ones_like(x), u, b, t=0)
    o.mag_sweeps(3)
    with Solver(p) as s:
        plan = s.plan()
        if field == "uniform" or nx % 2 == 0:  # (odd widths in an in-plane field: one node a thread)
            assert plan["kernel"] == "k_sweep_march_pair" and plan["rows"] == rows
        s.set_state(np.ones_like(x), u, b, t=0)
        s.mag_sweeps(3)
        gb = s.state()[2]
    ob = o.state()[2]
    assert np.linalg.norm(gb - ob) <= 1e-5 * np.linalg.norm(ob)


@pytest.mark.parametrize("shape", [(24, 24, 96), (40, 40, 60), (40, 40, 192), (48, 48, 128), (64, 64, 128),
                                   (41, 41, 150), (96, 96, 40), (101, 101, 20), (128, 128, 16)], ids=str)
def test_small_domains_are_cut_into_short_chunks(shape):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nx, ny, nz = shape
    with Solver(W.small_pipe(nx=nx, ny=ny, nz=nz, diameter=float(nx - 8), sweep_kernel="split")) as s:
        plan = s.plan()
    assert plan["planes"] == 1 or plan["ctas"] >= 2 * sms, plan


@pytest.mark.parametrize("shape", [(33, 35, 40), (99, 99, 64), (24, 24, 152), (24, 24, 153), (41, 41, 300)], ids=str)
def test_ib_pass_waits_where_the_planes_have_an_sm_each(shape):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nx, ny, nz = shape
    with Solver(W.small_pipe(nx=nx, ny=ny, nz=nz, diameter=float(nx - 8), sweep_kernel="split")) as s:
        assert s.plan()["ib_early"] == (nz > sms)


def test_large_domains_keep_two_rows():
    with Solver(W.pipe_ramp_96x96x512(sweep_kernel="split")) as s:
        plan = s.plan()
    assert plan["rows"] == 2 and plan["planes"] >= 16, plan
