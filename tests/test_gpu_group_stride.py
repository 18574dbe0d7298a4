"""The resident group kernel at its two shared-memory strides: as many planes of
27 x 27 nodes as only the larger one holds (eight a group instead of seven), end
planes exchanged between groups of unequal size, against the marching sweep.

Both form every node's value by the same roundings, so they agree to the bit."""
import numpy as np
import pytest

from paper_2211_09370_gb300 import workloads as W
from paper_2211_09370_gb300._lib import Batch, Solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("planes", [7, 8])
def test_groups_of_seven_and_eight_planes(planes):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nz = sms * planes // 4 - 2 * planes - 3  # four pipes: more than sms groups at one plane less
    ps = [W.small_pipe(nx=27, ny=27, nz=nz, diameter=19.0, n_mag=5, Re=100.0 + 20 * i, Ha=20.0, Rm=1e-3,
                       b0_kind="tanh" if i % 2 else "uniform", ramp_center=nz / 2.0, ramp_width=9.0, seed=61 + i)
          for i in range(4)]
    with Batch(ps) as B:
        info = B.info()
        assert info["resident_instances"] == 4
        B.step(2)
        got = [B.member(i).state() for i in range(4)]
    for i, p in enumerate(ps):
        with Solver(dict(p, sweep_kernel="split")) as s:
            s.step(2)
            want = s.state()
        for a, b in zip(got[i], want):
            np.testing.assert_array_equal(a, b, err_msg=str(i))
