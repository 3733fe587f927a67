"""h of gas whose smoothing lengths are far below the finest cells (side / 2^21 of the root cube), where the
cube reaches a thousand units to one side and the gas lies at coordinates near zero: a difference between a
gas coordinate and the cube's corner is rounded by as much as the kernels reach.

A length differs from the oracle's by the rounding of FP32 distances and sums (about 1e-7, and a few times
that where most of the kernel sum is the particle's own term); a neighbour that is not found changes it by
1e-4 or more.  The bound is 1e-5 on every particle."""
import numpy as np
import pytest

import oracle
from paper_0912_1786_gb300 import workloads as W

from gpu_common import run_gpu

pytestmark = pytest.mark.gpu


def _clump_over_a_cell_boundary(L, n_nei=32.0):
    """Gas of uniform density with lengths of about L on both sides of a boundary of finest cells along x, in
    the order of x; two other particles set the corner and the side of the cube, 2048."""
    f = np.float32
    corner = f(-1000.0) - f(5 * 2.0 ** -14)
    cell = 2048.0 / 2 ** 21
    edge = float(corner) + 1024000 * cell                    # -3.05e-4
    # gas on both sides of the edge, well inside a cell along y and z (edges there: multiples of 9.8e-4)
    lx, lyz = 2.0e-4, 1.2e-4
    n = int(lx * lyz ** 2 * n_nei / (4.0 / 3.0 * np.pi * (2.0 * L) ** 3))
    rng = np.random.default_rng(11)
    x = np.sort(edge + rng.uniform(-0.5 * lx, 0.5 * lx, n))
    y, z = (3.0e-4 + rng.uniform(0.0, lyz, n) for _ in range(2))
    far = [(corner, f(-1000.0), f(-1000.0)), (f(1000.0), f(0.0), f(0.0))]
    pos = [np.concatenate([a, [p[k] for p in far]]).astype(f) for k, a in enumerate((x, y, z))]
    one = np.ones(n + 2, f)
    p = W.Params(n_nei_sph=n_nei, gravity=0, adaptive_softening=0)
    return W.Workload("clump", *pos, 0 * one, 0 * one, 0 * one, one / (n + 2), one, f(L) * one, f(L) * one,
                      n_gas=n, params=p)


@pytest.mark.parametrize("L", [1.5e-5, 2.5e-5])
def test_lengths_below_the_finest_cells(L):
    w = _clump_over_a_cell_boundary(L)
    g = run_gpu(w, check=False)
    assert g["status"] == 0
    o = oracle.force_step(w, idx=np.zeros(1, np.int64))
    ng = w.n_gas
    assert np.abs(g["h"][:ng] / o["h"][:ng] - 1.0).max() < 1e-5
