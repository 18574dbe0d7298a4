"""Every form of the slab kernel against the oracle, each case checked to run it: one to
five rows per thread (more than three read S from memory, more than two exchange by
counters instead of messages), one to three planes per CTA, all slabs equal or the last of
one plane less, a single slab, no wall, in-plane and ramped fields, the strict and the
accelerated sweep.  And its messages, whose sequence numbers are of 16 bits, across their
wrap.

Tolerance as in test_gpu_slab.py: a contracting iteration with a few FP32 roundings of
6e-8 per sweep on terms of the size of b."""
import numpy as np
import pytest

import oracle
from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Batch, Solver

pytestmark = pytest.mark.gpu


def sms():
    import torch

    return torch.cuda.get_device_properties(0).multi_processor_count


# (rows, planes per CTA, box: planes as a function of the SM count)
CASES = {
    "one_slab": (1, 1, dict(nx=20, ny=21, nz=lambda n: 1)),
    "rows1": (1, 1, dict(nx=24, ny=21, nz=lambda n: 5)),
    "rows1_odd": (1, 1, dict(nx=21, ny=20, nz=lambda n: 2)),
    "rows1_two_planes": (1, 2, dict(nx=24, ny=23, nz=lambda n: 2 * n, b0_kind="tanh")),
    "rows1_two_and_one": (1, 2, dict(nx=21, ny=22, nz=lambda n: n + 1, b0_kind="tanh")),
    "rows1_three_planes": (1, 3, dict(nx=22, ny=20, nz=lambda n: 2 * n + 3)),
    "rows1_no_wall": (1, 1, dict(nx=24, ny=20, nz=lambda n: 6, geometry="none")),
    "rows1_strict": (1, 1, dict(nx=20, ny=18, nz=lambda n: 4, strict_qs=1)),
    "rows1_accelerated": (1, 1, dict(nx=22, ny=20, nz=lambda n: 5, alpha=0.75)),
    "rows1_channel": (1, 1, dict(nx=18, ny=21, nz=lambda n: 6, geometry="channel", diameter=15.5, b0_dir=(0.0, 1.0, 0.0))),
    "rows1_in_plane": (1, 1, dict(nx=26, ny=25, nz=lambda n: 6, b0_kind="field")),
    "rows2_odd": (2, 1, dict(nx=47, ny=40, nz=lambda n: 6)),
    "rows2_two_planes": (2, 2, dict(nx=32, ny=31, nz=lambda n: n + 40, b0_kind="tanh")),
    "rows2_odd_accelerated": (2, 1, dict(nx=41, ny=43, nz=lambda n: 3, alpha=0.75)),
    "rows3_odd": (3, 1, dict(nx=57, ny=56, nz=lambda n: 5, b0_kind="tanh")),
    "rows3_no_wall": (3, 1, dict(nx=57, ny=55, nz=lambda n: 4, geometry="none")),
    "rows3_strict": (3, 1, dict(nx=57, ny=54, nz=lambda n: 3, strict_qs=1)),
    "rows3_in_plane": (3, 1, dict(nx=64, ny=62, nz=lambda n: 60, b0_kind="field")),
    "rows3_two_planes": (3, 2, dict(nx=40, ny=40, nz=lambda n: 2 * n, b0_kind="tanh")),
    "rows3_two_and_one": (3, 2, dict(nx=40, ny=40, nz=lambda n: n + 1, b0_kind="tanh")),
    "rows3_three_planes": (3, 3, dict(nx=36, ny=35, nz=lambda n: 2 * n + 5)),
    "rows4_odd": (4, 1, dict(nx=71, ny=72, nz=lambda n: 4)),
    "rows4_two_planes": (4, 2, dict(nx=49, ny=49, nz=lambda n: 2 * n, b0_kind="tanh")),
    "rows4_two_and_one": (4, 2, dict(nx=49, ny=48, nz=lambda n: 2 * n - 1, b0_kind="tanh")),
    "rows4_in_plane": (4, 1, dict(nx=72, ny=72, nz=lambda n: 100, b0_kind="field")),
    "rows5_odd": (5, 1, dict(nx=71, ny=90, nz=lambda n: 5, b0_kind="tanh")),
    "rows5_two_planes": (5, 2, dict(nx=55, ny=55, nz=lambda n: 2 * n, b0_kind="tanh")),
    "rows5_two_and_one": (5, 2, dict(nx=55, ny=55, nz=lambda n: 2 * n - 1, b0_kind="tanh")),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_form_matches_oracle(case):
    rows, planes, kw = CASES[case]
    kw = dict(kw, nz=kw["nz"](sms()))
    kw.setdefault("diameter", float(min(kw["nx"], kw["ny"]) - 7))
    if kw.get("b0_kind") == "field":
        kw["b0_field"] = W.six_magnet_field(kw["nx"], kw["ny"], kw["diameter"])
    if kw.get("b0_kind") == "tanh":
        kw.update(ramp_center=kw["nz"] / 2.0, ramp_width=max(1.0, kw["nz"] / 16.0))
    p = W.small_pipe(n_mag=60, perturb=0.0, Ha=25.0, Rm=4e-3, **kw)
    z, y, x = np.meshgrid(np.arange(float(p["nz"])), np.arange(float(p["ny"])), np.arange(float(p["nx"])), indexing="ij")
    # (a short wave in z: a plane taken for its neighbour shows)
    u = np.stack([0.01 * np.sin(2 * np.pi * y / p["ny"]) + 0.005 * np.cos(2 * np.pi * z / min(p["nz"], 7)),
                  0.02 * np.cos(2 * np.pi * x / p["nx"]), 0.03 + 0.01 * np.sin(2 * np.pi * z / min(p["nz"], 5))])
    o = oracle.Oracle(dict(p, precision="fp64"))
    o.set_state(np.ones_like(x), u, np.zeros_like(u), t=0)
    o.mag_sweeps(23)
    o.step(1)
    with Solver(p) as s:
        plan = s.plan()
        assert plan["kernel"] == "k_sweeps_slab" and (plan["rows"], plan["planes"]) == (rows, planes), plan
        s.set_state(np.ones_like(x), u, np.zeros_like(u), t=0)
        s.mag_sweeps(23)
        s.step(1)
        _, gu, gb = s.state()
    _, ou, ob = o.state()
    for g, w in ((gu, ou), (gb, ob)):
        assert np.linalg.norm(g - w) <= 1e-5 * np.linalg.norm(w)


@pytest.mark.parametrize("shape", [(71, 72, 10), (70, 72, 10), (33, 31, 6)], ids=str)
def test_few_sweeps_stay_with_one_plane_per_cta(shape):
    # (below 24 sweeps a step the slab kernel's start does not pay)
    nx, ny, nz = shape
    with Solver(W.small_pipe(nx=nx, ny=ny, nz=nz, diameter=float(min(nx, ny) - 7), n_mag=23)) as s:
        assert s.plan()["kernel"] == "k_sweeps_resident"


MSG = dict(nx=20, ny=20, nz=6, diameter=14.0, n_mag=40, Ha=20.0, Rm=1e-3)


def states(s):
    rng = np.random.default_rng(3)
    shape = (MSG["nz"], MSG["ny"], MSG["nx"])
    for _ in range(2):
        yield np.ones(shape), 0.02 * rng.standard_normal((3,) + shape), 0.01 * rng.standard_normal((3,) + shape)


def sweeps(s, state, n):
    s.set_state(*state)
    s.mag_sweeps(n)
    return s.state()[2]


def test_message_numbers_wrap_inside_a_launch():
    with Solver(W.small_pipe(**MSG)) as s, Solver(W.small_pipe(**MSG)) as fresh:
        assert s.plan()["kernel"] == "k_sweeps_slab" and s.plan()["rows"] <= 2
        a, b = states(s)
        sweeps(s, a, 65536 - 41)
        np.testing.assert_array_equal(sweeps(s, b, 83), sweeps(fresh, b, 83))


def test_stale_messages_are_not_taken_for_new_ones():
    # two sweeps leave messages in both slots; single ones, each a launch, use the first
    # only, 65534 of them bring the numbers of the second back
    with Solver(W.small_pipe(**MSG)) as s, Solver(W.small_pipe(**MSG)) as fresh:
        a, b = states(s)
        sweeps(s, a, 2)
        for _ in range(65534):
            s.mag_sweeps(1)
        np.testing.assert_array_equal(sweeps(s, b, 5), sweeps(fresh, b, 5))


def test_group_messages_wrap():
    ps = [W.small_pipe(nx=20, ny=18, nz=9 + i, diameter=12.0, n_mag=270, Ha=20.0, Rm=1e-3, seed=5 + i) for i in range(2)]
    steps = 65536 // 270 + 3
    with Batch(ps) as B:
        info = B.info()
        assert info["resident_instances"] == 2 and info["resident_groups"] > 2
        B.step(steps)
        got = [B.member(i).state() for i in range(2)]
    for p, g in zip(ps, got):
        with Solver(dict(p, sweep_kernel="split")) as s:
            s.step(steps)
            want = s.state()
        for x, y in zip(g, want):
            np.testing.assert_array_equal(x, y)
