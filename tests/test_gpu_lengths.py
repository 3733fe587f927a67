"""The length solves at the sizes where their blocks, chunks and lists end: h, eps and the sums at them
against the FP64 oracle.

The solves converge to the root of the same equation, so a length differs from the oracle's by the FP32
rounding of the distances and of the sums over some fifty neighbours (about 1e-7), far below the bounds the
force step is specified to (gpu_common: median 1e-5, 99th percentile 1e-4)."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_0912_1786_gb300 import workloads as W

from gpu_common import assert_tol, run_gpu

pytestmark = pytest.mark.gpu

GAS = ("h", "rho", "omega", "zeta")
ALL = ("eps", "ups", "X")


def _compare(w, names, p=None, offsets=None):
    g = run_gpu(w, p, check=False)
    assert g["status"] == 0
    o = oracle.force_step(w, params=p)
    for k in names:
        ref = o[k][: w.n_gas] if k in GAS else o[k]
        assert_tol(k, g[k][: len(ref)], ref, scale=_scale(k, w.m[: len(ref)]))


def _scale(k, m):
    # zeta = sum m (3 w + u w') / (3 sum w): a difference of terms of the order of the mass
    return m if k == "zeta" else None


@pytest.mark.parametrize("n", [61, 127, 128, 129, 1000, 4097, 30011])
@pytest.mark.parametrize("group", [0, 1, 16, 32])
def test_all_gas_sizes(n, group):
    _compare(W.evrard_sphere(n, seed=n, sigma_v=0.1, params=W.Params(leaf_size=8, length_group=group)), GAS + ALL)


@pytest.mark.parametrize("n_dm,n_gas,leaf", [(9000, 100, 8), (5000, 2501, 16), (50021, 17011, 32), (90001, 40003, 64)])
def test_gas_among_other_particles(n_dm, n_gas, leaf):
    # the gas lists of the h solve; from 65,536 particles on the super-groups' leaf lists, with wide leaves
    # also the block shape with more candidates
    _compare(W.hernquist_gas(n_dm, n_gas, seed=n_dm, params=W.Params(leaf_size=leaf)), GAS + ALL)


@pytest.mark.parametrize("factor", [0.2, 6.0])
@pytest.mark.parametrize("n", [2000, 70001])
def test_poor_starting_lengths(n, factor):
    w = W.periodic_box(n, seed=5, n_gas=n // 2, sigma_v=0.1)
    w.params = dataclasses.replace(w.params, gravity=0, adaptive_softening=0)
    w.h = np.ascontiguousarray(w.h * np.float32(factor))
    _compare(w, GAS)
    v = W.evrard_sphere(n, seed=6)
    v.h = np.ascontiguousarray(v.h * np.float32(factor))
    v.eps = np.ascontiguousarray(v.eps * np.float32(factor))
    _compare(v, GAS + ALL)


@pytest.mark.parametrize("nnei", [20.0, 110.0])
def test_neighbour_numbers_beyond_the_short_lists(nnei):
    # 110 neighbours: gathers above the four-way lists' room fall to the whole warp's list
    p = W.Params(leaf_size=8, n_nei_sph=nnei, n_nei_grav=nnei)
    _compare(W.evrard_sphere(9001, seed=9, params=p), GAS + ALL, p)


@pytest.mark.parametrize("n,group", [(9000, 0), (9000, 8), (20000, 16)])
def test_balls_of_far_outliers(n, group):
    # a small sphere without an edge: the balls of the outermost particles hold more than their lists do
    _compare(W.plummer(n, seed=7, params=W.Params(theta=0.6, n_nei_grav=32.0, sph=0, length_group=group)), ALL)


def test_many_small_systems():
    # blocks whose particles belong to several systems
    import torch
    from paper_0912_1786_gb300 import evol as E
    from paper_0912_1786_gb300.device import DeviceSet
    sizes = [70, 71, 64, 200, 65, 90, 77]
    parts = [W.evrard_sphere(k, seed=k) for k in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)])
    cat = {f: np.concatenate([getattr(q, f) for q in parts]) for f in parts[0].arrays()}
    w = W.Workload("systems", **cat, n_gas=int(off[-1]), params=parts[0].params, sys_offsets=off)
    ds = DeviceSet(w)
    ctx = E.evol_create(w.n, torch.cuda.current_stream().cuda_stream)
    try:
        E.evol_step_batched(ctx, off, ds.particles, ds.params, ds.outputs)
        E.evol_sync(ctx)
        g = ds.numpy()
    finally:
        E.evol_destroy(ctx)
    for k, q in enumerate(parts):
        o = oracle.force_step(q)
        for f in GAS + ALL:
            ref = o[f][: q.n_gas]
            assert_tol(f, g[f][off[k]: off[k + 1]], ref, scale=_scale(f, q.m))
