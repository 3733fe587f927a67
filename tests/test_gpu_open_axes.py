"""Axes that are not periodic take no length: whatever periodic_lo and periodic_hi hold there (an unbounded
axis written as infinities, bounds whose difference overflows, unset values), results are those of finite
bounds, bit for bit."""
import dataclasses

import numpy as np
import pytest

from paper_0912_1786_gb300 import workloads as W

from gpu_common import run_gpu

pytestmark = pytest.mark.gpu

BOUNDS = {"infinite": (-np.inf, np.inf), "overflow": (-3.0e38, 3.0e38), "unset": (np.nan, np.nan)}
OUT = ("h", "rho", "P", "omega", "zeta", "ax", "ay", "az", "dudt")


def _slab():
    # x open, y and z periodic
    w = W.shock_tube(left=(25, 5, 5), right=(15, 3, 3), jitter=0.25)
    w.vx[:] = np.where(w.x < 0.5, 0.2, -0.2).astype(np.float32)
    return w, (0,)


def _open_gas():
    # SPH alone, no periodic axis
    w = W.evrard_sphere(700, seed=5, sigma_v=0.1)
    w.params = dataclasses.replace(w.params, gravity=0, adaptive_softening=0)
    return w, (0, 1, 2)


@pytest.mark.parametrize("api", ["step", "phases"])
@pytest.mark.parametrize("make", [_slab, _open_gas])
@pytest.mark.parametrize("bounds", BOUNDS)
def test_bounds_of_open_axes_are_not_read(bounds, make, api):
    w, open_axes = make()
    lo, hi = list(w.params.periodic_lo), list(w.params.periodic_hi)
    ref = run_gpu(w, check=False, api=api)
    assert ref["status"] == 0
    for a in open_axes:
        lo[a], hi[a] = BOUNDS[bounds]
    got = run_gpu(w, dataclasses.replace(w.params, periodic_lo=tuple(lo), periodic_hi=tuple(hi)), check=False, api=api)
    assert got["status"] == 0
    for k in OUT:
        assert np.array_equal(got[k], ref[k]), k
    assert np.any(ref["dudt"] != 0)
