"""Force and flow on domains that are long in y or z: more tiles of rows, or more
chunks of planes, than the 65535 CTAs of a grid's second and third dimension.

One step from a noisy state against the oracle; tolerances as in
test_gpu_flow_march.py (a node's update sums some 30 terms of its neighbours)."""
import pytest

from paper_2211_09370_gb300 import workloads as W
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
