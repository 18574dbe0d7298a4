"""Chains are for steps whose graph stays small: members with very many sweeps march
jointly, one launch per sweep for all of them, and give what single handles give."""
import numpy as np
import pytest

from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Batch, Server, Solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_mag,chains", [(16384, True), (16385, False)])
def test_members_of_many_sweeps(n_mag, chains):
    ps = [W.small_pipe(nx=12, ny=11, nz=2, diameter=7.0, n_mag=n_mag, Ha=20.0, Rm=1e-3, seed=i, sweep_kernel="split")
          for i in range(2)]
    with Batch(ps) as B:
        assert B.info()["launches_per_step"] == (4 if chains else 2) * n_mag + 3
        B.step(1)
        got = B.member(1).state()
    with Solver(ps[1]) as s:
        s.step(1)
        want = s.state()
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("chunk", [1, 5])
def test_served_marching_requests_match_single_handles(chunk):
    # (one chunk of one step: the joint march; five: chains)
    ps = [W.small_pipe(nx=14 + i, ny=13, nz=5, diameter=8.0, n_mag=3 + i, Ha=20.0, Rm=2e-3, seed=i,
                       sweep_kernel="split") for i in range(3)]
    with Server(hbm_budget_bytes=1 << 30, chunk_steps=chunk) as S:
        ids = [S.submit(p, tol=1e-12, max_steps=2 * chunk, keep_fields=True) for p in ps]
        left = set(ids)
        while left:
            S.run()
            left -= {r["id"] for r in S.poll()}
        got = [S.fields(i) for i in ids]
    for p, g in zip(ps, got):
        with Solver(p) as s:
            s.step(2 * chunk)
            want = s.state()
        for a, b in zip(g, want):
            np.testing.assert_array_equal(np.reshape(a, b.shape), b)
