"""Smallest-first admission knows the planes that only the resident kernel's large
shared-memory stride holds."""
import pytest

from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Server

pytestmark = pytest.mark.gpu


def running(ps):
    with Server(hbm_budget_bytes=8 << 30, chunk_steps=1, admit="smallest") as S:
        for p in ps:
            S.submit(p, tol=1e-12, max_steps=2)
        return S.run()


def test_planes_above_the_small_stride():
    # 74 x 74 = 5476 nodes with a short wall beside small pipes: one launch holds them all
    ps = [W.small_pipe(nx=16, ny=16, nz=8, diameter=10.0, n_mag=3, seed=i) for i in range(2)]
    ps.append(W.small_pipe(nx=74, ny=74, nz=6, diameter=8.0, n_mag=3))
    assert running(ps) == (3, 0)


def test_what_no_stride_holds_still_waits():
    ps = [W.small_pipe(nx=16, ny=16, nz=8, diameter=10.0, n_mag=3, seed=i) for i in range(2)]
    ps.append(W.small_pipe(nx=90, ny=90, nz=6, diameter=80.0, n_mag=3))
    assert running(ps) == (2, 1)


def test_what_the_large_stride_holds_is_counted_there():
    # as many planes of 74 x 74 as the device has SMs, one a group, leave no room
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ps = [W.small_pipe(nx=74, ny=74, nz=sms // 2, diameter=8.0, n_mag=3, seed=i) for i in range(2)]
    assert running(ps) == (2, 0)
    assert running(ps + [W.small_pipe(nx=74, ny=75, nz=sms // 2, diameter=8.0, n_mag=3)]) == (2, 1)
