"""The force walk of sets that do not fill the chip, whose groups are walked in parts: results against the
FP64 oracle without check mode (which walks whole groups), at sizes around the ends of groups and of
super-groups and around the largest set that is split, for each form of the walk.  Tolerances as
gpu_common: the parts change the order of a few additions only."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_0912_1786_gb300 import workloads as W

from gpu_common import acc, assert_tol, run_gpu

pytestmark = pytest.mark.gpu


def _compare(w, p=None, precision=0, gas=True):
    g = run_gpu(w, p, check=False, precision=precision)
    assert g["status"] == 0
    o = oracle.force_step(w, params=p)
    assert_tol("acc", acc(g), np.stack([o["ax"], o["ay"], o["az"]], 1), scale=o["aabs"])
    if (p or w.params).gravity:
        assert_tol("pot", g["pot"], o["pot"])
    if gas:
        assert_tol("dudt", g["dudt"][: w.n_gas], o["dudt"][: w.n_gas], scale=o["duabs"][: w.n_gas])
    return g, o


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [61, 255, 256, 257, 1000, 4097, 30011, 58367, 58401])
def test_gravity_and_sph(n, precision):
    _compare(W.evrard_sphere(n, seed=n, sigma_v=0.1), precision=precision)


@pytest.mark.parametrize("n", [97, 6007, 40009])
def test_gravity_alone(n):
    w = W.evrard_sphere(n, seed=n)
    _compare(w, dataclasses.replace(w.params, sph=0), gas=False)


@pytest.mark.parametrize("a,b", [(7, 5), (21, 13)])
def test_sph_alone_periodic(a, b):
    w = W.shock_tube(left=(5 * a, a, a), right=(5 * b, b, b), jitter=0.25)
    rng = np.random.default_rng(3)
    w.vx, w.vy, w.vz = (np.ascontiguousarray(rng.normal(0, 0.1, w.n), np.float32) for _ in range(3))
    _compare(w)


@pytest.mark.parametrize("n", [300, 9001])
def test_dissipation_variants(n):
    w = W.with_dissipation(W.evrard_sphere(n, seed=n), seed=2, sigma_v=0.1, visc_form=1, balsara=1, variable_alpha=1,
                           conduction=1)
    g, o = _compare(w)
    for k in ("dalpha", "dalpha_u"):
        assert_tol(k, g[k][: w.n_gas], o[k][: w.n_gas], scale=np.full(w.n_gas, np.median(np.abs(o[k][: w.n_gas]))))


def test_several_systems_share_super_groups():
    # super-groups of two systems have no lists: the first part of their groups walks alone
    import torch
    from paper_0912_1786_gb300 import evol as E
    from paper_0912_1786_gb300.device import DeviceSet
    sizes = [301, 77, 500, 64, 1003]
    parts = [W.evrard_sphere(k, seed=k, sigma_v=0.1) for k in sizes]
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
        sl = slice(off[k], off[k + 1])
        assert_tol("acc", acc(g)[sl], np.stack([o["ax"], o["ay"], o["az"]], 1), scale=o["aabs"])
