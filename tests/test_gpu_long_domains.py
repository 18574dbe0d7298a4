"""Steps on domains that are long in y or z: more tiles of rows, or more
chunks of planes, than the 65535 CTAs of a grid's second and third dimension.

One step from a noisy state against the oracle; tolerances as in
test_gpu_flow_march.py (a node's update sums some 30 terms of its neighbours)."""
import numpy as np
import pytest

from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Batch
from tests.test_gpu_flow_march import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,shape", [
    ("fp32", (2, 1, 65535 * 32 + 41)), ("fp64", (1, 2, 65535 * 32 + 41)),  # chunks are of at most 32 planes
    ("fp32", (2, 65535 * 8 + 9, 1)), ("fp64", (3, 65535 * 4 + 9, 2)),      # tiles are of 8 and 4 rows
], ids=["planes_fp32", "planes_fp64", "rows_fp32", "rows_fp64"])
def test_long_domain_matches_oracle(precision, shape):
    nx, ny, nz = shape
    p = W.small_pipe(nx=nx, ny=ny, nz=nz, diameter=8.0, geometry="none", n_mag=1, Ha=5.0, Rm=1e-2, perturb=0.0,
                     force_amp=0.2, force_period=50.0, sweep_kernel="split")
    check(p, (nz, ny, nx), precision)


def test_batch_member_of_more_rows_than_a_chains_grid_holds():
    # chains have tiles of 16 rows at most: this member marches jointly, at rest but for
    # its force, and is uniform like its domain
    p = W.small_pipe(nx=2, ny=65535 * 16 + 17, nz=1, diameter=8.0, geometry="none", n_mag=2, Ha=5.0, Rm=1e-2,
                     perturb=0.0, sweep_kernel="split")
    with Batch([p]) as B:
        B.step(2)
        u = B.member(0).state()[1]
    assert np.abs(u[2]).min() > 0 and np.ptp(u[2]) <= 1e-6 * np.abs(u[2]).max()
