"""Handles and batches of different sizes side by side: what a later, smaller one
asks of a kernel both use leaves the earlier, larger one as it was."""
import numpy as np
import pytest

from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Batch, Solver

pytestmark = pytest.mark.gpu

KINDS = {
    "split": (dict(sweep_kernel="split"), 60, 24),
    "split_fp64": (dict(sweep_kernel="split", precision="fp64"), 60, 24),
    "fused": (dict(sweep_kernel="fused"), 64, 24),
    "resident_even": (dict(sweep_kernel="resident"), 64, 48),
    "resident_odd": (dict(sweep_kernel="resident"), 47, 41),
    "resident_fp64": (dict(sweep_kernel="resident", precision="fp64"), 48, 24),
}


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_a_later_smaller_handle_leaves_a_larger_one_running(kind):
    kw, large, small = KINDS[kind]
    make = lambda n: Solver(W.small_pipe(nx=n, ny=n, nz=6, diameter=n - 8.0, n_mag=30, **kw))
    with make(large) as s:
        s.step(2)
        want = s.state()
    with make(large) as s, make(small) as t:
        t.step(1)
        s.step(2)
        got = s.state()
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("kernel", ["split", "auto"])
def test_a_later_smaller_batch_leaves_a_larger_one_running(kernel):
    make = lambda n: Batch([W.small_pipe(nx=n, ny=n, nz=6, diameter=n - 8.0, n_mag=30, sweep_kernel=kernel)])
    with make(64) as A:
        A.step(2)
        want = A.member(0).state()
    with make(64) as A, make(24) as B:
        B.step(1)
        A.step(2)
        got = A.member(0).state()
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
