"""The benchmark names the kernel that runs and hashes the sources it is made of."""
import ctypes as C
import os
import re

import pytest

import bench
from paper_2211_09370_gb300 import _lib
from paper_2211_09370_gb300.build import CSRC


class Handle:
    def __init__(self, route, kernel, planes):
        self.units = {"sweep_kernel": route, "n_mag": 7}
        self._plan = {"kernel": kernel, "ctas": 1, "threads": 1, "rows": 0, "planes": planes}

    def plan(self):
        return self._plan


@pytest.mark.parametrize("route,kernel,launches,per_launch", [
    ("resident", "k_sweeps_resident", 4, 7), ("resident", "k_sweeps_slab", 4, 7), ("resident", "k_sweeps_resident64", 4, 7),
    ("resident", "k_sweeps_cluster64", 4, 7), ("fused", "k_sweep_fused", 10, 1), ("split", "k_sweep_march_pair", 17, 1),
    ("split", "k_sweep_march", 17, 1), ("planes", "k_sweep_ib", 10, 1)])
def test_label_names_the_kernel_that_runs(route, kernel, launches, per_launch):
    n, name, sweeps = bench.sweep_kernel_info(Handle(route, kernel, 1), {"precision": "fp64"})
    assert (n, sweeps) == (launches, per_launch)
    assert name.startswith(kernel + "<")


def test_every_kernel_of_a_handle_is_in_the_source_hash():
    # files whose kernels a single handle launches: those qslbm_launch.cuh includes
    with open(os.path.join(CSRC, "qslbm_launch.cuh")) as f:
        used = {n for n in re.findall(r'#include "(qslbm_\w+\.cuh)"', f.read())}
    assert used | {"qslbm_launch.cuh"} == set(bench.KERNEL_SOURCES)


def test_plan_names_every_kernel_of_the_header():
    with open(os.path.join(os.path.dirname(CSRC), os.pardir, "include", "qslbm.h")) as f:
        src = f.read()
    names = {int(v): c for v, c in re.findall(r"#define QSLBM_KERNEL_\w+ (\d+)\s*/\* (\w+)", src)}
    assert names == _lib.SWEEP_PLAN_KERNEL
    assert C.sizeof(_lib.qslbm_sweep_plan_t) == 24
    L = _lib.load()
    assert L.qslbm_sweep_plan(None, None) == _lib.EINVAL
