"""bench.py's count of the library's kernels per step, against launches counted on a GPU with 152 SMs (a launch
list of one step of each set), and its sizes against the sources they follow."""
import os
import re
import sys
from types import SimpleNamespace

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from paper_0912_1786_gb300.workloads import Params  # noqa: E402

ALONE = dict(gravity=0, adaptive_softening=0)
COUNTED = [
    # n, gas, parameters, systems, kernels
    (1000, 1000, {}, 1, 20),
    (49152, 16381, {}, 1, 36),
    (68000, 34000, {}, 1, 36),
    (400000, 100000, {}, 1, 70),
    (70001, 70001, {}, 1, 30),
    (70001, 70001, dict(sph_scheme=1), 1, 33),
    (70001, 70001, dict(balsara=1), 1, 29),
    (110001, 70001, dict(balsara=1, visc_form=1), 1, 37),
    (70001, 0, dict(sph=0), 1, 32),
    (80001, 0, dict(sph=0), 1, 30),
    (70001, 0, dict(sph=0, periodic_mask=7), 1, 28),
    (95000, 95000, dict(periodic_mask=6, **ALONE), 1, 29),
    (43225, 43225, {}, 7, 32),
]


@pytest.mark.parametrize("n,n_gas,params,nsys,kernels", COUNTED)
def test_launches_per_step(n, n_gas, params, nsys, kernels):
    import bench
    w = SimpleNamespace(n=n, n_gas=n_gas, params=Params(**params), sys_offsets=None if nsys == 1 else range(nsys + 1))
    assert bench.launches_per_step(w) == kernels


def test_sizes_follow_the_sources():
    import bench
    csrc = os.path.join(ROOT, "paper_0912_1786_gb300", "csrc")
    text = {f: open(os.path.join(csrc, f)).read() for f in ("tree.cu", "lengths.cu", "evol_internal.cuh")}
    num = lambda f, name: int(re.search(name + r"\s*=?\s*(\d+)", text[f])[1])
    assert bench.RANK_MAX == num("tree.cu", "int RANK_MAX")
    assert bench.FUSED_MAX == num("evol_internal.cuh", "define EVOL_SORT_FUSED_MAX")
    assert bench.LISTS_MIN == num("lengths.cu", "int LISTS_MIN")
    assert bench.SCAN_ONE_MAX == (num("tree.cu", "int SCAN_ONE_MAX") * num("tree.cu", "int SC_THREADS") *
                                  num("tree.cu", "int SC_ITEMS"))
