"""Every particle of a length solve, and of a walk in parts, against the FP64 oracle, over the routes that a
particle can take: the last ones of a set, lists that overflow, leaf lists of super-groups with the velocity
divergence and with active lists, both shapes of block, one solve for h and eps on periodic axes.

Bounds on every particle, not on a percentile.  A length is the root of n L^3 = eta^3 over FP32 distances and
sums of some fifty terms, each right to a few 6e-8; the root carries a few times the sum's error where most of
the sum is the particle's own term, so 1e-5.  A sum of the walk is at most a few thousand terms of relative
error 6e-7 (a reciprocal square root cubed), added in blocks of 64 whose totals are rounded once each: 1e-5 of
the sum of their magnitudes, for particles none of whose decisions the oracle took within gpu_common's
EXPLAIN_MARGIN of its threshold (an FP32 decision can differ there, by a node's whole expansion error)."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_0912_1786_gb300 import workloads as W

from gpu_common import EXPLAIN_MARGIN, acc, assert_tol, report

pytestmark = pytest.mark.gpu

LEN_TOL = 1e-5
SUM_TOL = 1e-5
NONE = np.zeros(1, np.int64)          # one particle's forces: only the lengths are wanted


def _step(w, p=None, steps=1):
    import torch
    from paper_0912_1786_gb300 import build, evol as E
    from paper_0912_1786_gb300.device import DeviceSet
    build.build()
    ds = DeviceSet(w, p or w.params)
    ctx = E.evol_create(w.n, torch.cuda.current_stream().cuda_stream)
    try:
        for _ in range(steps):
            E.evol_step(ctx, ds.particles, ds.params, ds.outputs)
            assert E.evol_sync(ctx, raise_on_error=False) == 0
        g = ds.numpy()
        g["counters"] = E.evol_get_counters(ctx)
        if w.alpha is not None:
            g["diss"] = E.evol_get_debug(ctx, E.EVOL_DBG_DISS, np.float32).reshape(5, w.n).astype(np.float64)
    finally:
        E.evol_destroy(ctx)
    return g


def _every_length(w, g, o, names=("h", "eps")):
    for k in names:
        ref = o[k][: w.n_gas] if k == "h" else o[k]
        err = np.abs(g[k][: len(ref)] / ref - 1.0)
        report({"quantity": k + "_every", "n": int(len(ref)), "max": float(err.max())})
        assert err.max() < LEN_TOL, (k, int(err.argmax()), float(err.max()))


@pytest.mark.parametrize("n", [61, 129, 257, 1025, 4097, 30011])
def test_every_particle_of_a_set(n):
    w = W.evrard_sphere(n, seed=n, sigma_v=0.1)
    g, o = _step(w), oracle.force_step(w)
    _every_length(w, g, o)
    clear = o["margin"] > EXPLAIN_MARGIN
    assert clear.mean() > 0.9
    for name, d, scale in (("acc", np.linalg.norm(acc(g) - np.stack([o["ax"], o["ay"], o["az"]], 1), axis=1), o["aabs"]),
                           ("dudt", np.abs(g["dudt"] - o["dudt"]), o["duabs"])):
        err = (d / scale)[clear]
        report({"quantity": name + "_every", "n": int(len(err)), "max": float(err.max())})
        assert err.max() < SUM_TOL, (name, float(err.max()))


@pytest.mark.parametrize("n,group", [(9000, 0), (20000, 8)])
def test_far_outliers(n, group):
    # balls of the outermost particles that hold more than their lists do, and walks of their own
    w = W.plummer(n, seed=7, params=W.Params(theta=0.6, n_nei_grav=32.0, sph=0, length_group=group))
    g, o = _step(w), oracle.force_step(w, idx=NONE)
    _every_length(w, g, o, ("eps",))
    assert g["counters"][17] > 0 and g["counters"][18] > 0


@pytest.mark.parametrize("group", [2, 3, 4, 10, 15, 16, 24, 31])
def test_every_group_size_takes_the_leaf_lists(group):
    # 65,536 particles and more: an item of any size lies inside one quarter of a super-group
    n = 66001
    w = W.evrard_sphere(n, seed=10, params=W.Params(leaf_size=8, length_group=group))
    g, o = _step(w), oracle.force_step(w, idx=NONE)
    _every_length(w, g, o)
    # the queue's end: the items, each of four warps, and at most the grid's blocks, six per SM
    import torch
    per = 2 if group < 4 else 4 if group < 16 else 8
    items = -(-n // (4 * per))
    blocks = 6 * torch.cuda.get_device_properties(0).multi_processor_count
    assert items <= g["counters"][5] <= items + blocks


@pytest.mark.parametrize("n_gas", [65535, 65536])
def test_gas_lists_on_both_sides_of_the_line(n_gas):
    # the leaf lists of an h solve go by the number of gas particles, not by that of all particles
    w = W.hernquist_gas(20011, n_gas, seed=17)
    _every_length(w, _step(w), oracle.force_step(w, idx=NONE))


def _gas_of_a_halo(n):
    # h alone: the balls of the halo's outermost particles would hold more than the longest list
    w = W.hernquist_gas(n, n, seed=9)
    w.params = dataclasses.replace(w.params, gravity=0, adaptive_softening=0)
    return w


def _with_curl(n):
    return W.with_dissipation(W.evrard_sphere(n, seed=9), seed=3, sigma_v=0.1, balsara=1)


@pytest.mark.parametrize("nnei", [112.0, 113.0, 160.0])
@pytest.mark.parametrize("make", [lambda: W.evrard_sphere(9001, seed=9), lambda: _gas_of_a_halo(9001), lambda: _with_curl(9001)])
def test_many_neighbours(make, nnei):
    # from 113 on particles are solved by whole warps, with lists of twice the length
    w = make()
    w.params = dataclasses.replace(w.params, n_nei_sph=nnei, n_nei_grav=nnei)
    g = _step(w, steps=2)
    _every_length(w, g, oracle.force_step(w, idx=NONE), ("h", "eps") if w.params.gravity else ("h",))
    if nnei > 113:
        # near its root a particle's list is made once, not first a shorter one that overflows
        assert g["counters"][20] + g["counters"][21] < 1.1 * w.n_gas


@pytest.mark.parametrize("n", [3001, 70001])
def test_one_solve_for_both_lengths_on_periodic_axes(n):
    w = W.periodic_box(n, seed=8, n_gas=n, sigma_v=0.1)
    w.params = dataclasses.replace(w.params, n_nei_grav=w.params.n_nei_sph)
    g, o = _step(w), oracle.force_step(w, idx=NONE)
    assert g["counters"][24] == g["counters"][25] == g["counters"][3]      # one solve served both
    _every_length(w, g, o)
    for k in ("rho", "omega", "ups", "X"):
        assert_tol(k, g[k], o[k])


def test_wide_blocks_in_one_solve_for_both_lengths():
    # a halo and a sphere, all of it gas: more candidates than the blocks of four warps hold
    w = W.hernquist_gas(40009, 30007, seed=12, params=W.Params(leaf_size=8, length_group=16))
    w.n_gas, w.u = w.n, np.full(w.n, 0.05, np.float32)
    g, o = _step(w), oracle.force_step(w, idx=NONE)
    # the queue's end: items of 64 particles and the grid's blocks, fewer than there are items of 32
    assert g["counters"][5] < w.n // 32
    _every_length(w, g, o)
    for k in ("rho", "omega", "ups", "X"):
        assert_tol(k, g[k], o[k])


@pytest.mark.parametrize("make", [lambda: W.evrard_sphere(70001, seed=13), lambda: W.hernquist_gas(40009, 35017, seed=13)])
def test_divergence_and_curl_with_leaf_lists(make):
    w = W.with_dissipation(make(), seed=3, sigma_v=0.1, visc_form=1, balsara=1, variable_alpha=1, conduction=1)
    ng = w.n_gas
    g, o = _step(w), oracle.force_step(w, idx=W.sample_indices(ng, 500))
    _every_length(w, g, o)
    # sums that cancel: on the scale of the flow's gradients around the particle
    flow = np.abs(o["divv_h"][:ng]) + o["curlv_h"][:ng]
    for name, got, ref in (("divv_h", g["diss"][0, :ng], o["divv_h"][:ng]), ("curlv_h", g["diss"][1, :ng], o["curlv_h"][:ng])):
        assert_tol(name, got, ref, scale=flow)
    f = np.abs(g["diss"][2, :ng] - o["balsara_f"][:ng])
    assert np.median(f) < 1e-5 and f.max() < 1e-2
    ix = W.sample_indices(ng, 500)
    tau = w.params.alpha_tau * o["h"][ix] / o["vsig"][ix]
    st = o["state"]
    sc = np.abs(st["alpha"][ix] - w.params.alpha_min) / tau + w.params.alpha_source * st["f"][ix] * np.abs(o["divv_h"][ix])
    assert_tol("dalpha", g["dalpha"][ix], o["dalpha"][ix], scale=sc)


def _integrate(w, call):
    import torch
    from paper_0912_1786_gb300 import build, evol as E
    from paper_0912_1786_gb300.device import DeviceSet
    build.build()
    ds = DeviceSet(w)
    ctx = E.evol_create(w.n, torch.cuda.current_stream().cuda_stream)
    try:
        r = call(E, ctx, ds)
        assert E.evol_sync(ctx, raise_on_error=False) == 0
        st = {k: v.cpu().numpy().astype(np.float64) for k, v in ds.inp.items()}
        flow = E.evol_get_debug(ctx, E.EVOL_DBG_FLOW, np.float32).reshape(3, w.n).astype(np.float64)
        bins = E.evol_get_debug(ctx, E.EVOL_DBG_BINS, np.int64).reshape(2, w.n)
    finally:
        E.evol_destroy(ctx)
    return r, st, flow, bins


def _positions_track(st, o):
    err = np.linalg.norm(np.stack([st[k] - o[k] for k in "xyz"], 1), axis=1)
    report({"quantity": "positions", "median": float(np.median(err)), "max": float(err.max())})
    assert np.median(err) < 1e-6 and err.max() < 1e-4


def test_global_step_with_leaf_lists():
    w = W.evrard_sphere(70001, seed=14, sigma_v=0.1)
    ts = oracle.TimeStep(eta_acc=0.1, eta_courant=0.2, eta_u=0.2, dt_max=0.05)
    o = oracle.run(w, 1, ts)
    ip = dict(eta_acc=0.1, eta_courant=0.2, eta_u=0.2, dt_max=0.05)
    (t, _), st, flow, _ = _integrate(w, lambda E, c, ds: E.evol_run(c, ds.particles, ds.params, E.make_integrator(**ip),
                                                                   ds.outputs, 1))
    assert abs(t - o["dts"][0]) <= 2e-5 * o["dts"][0]
    _positions_track(st, o)
    for k, name in ((0, "divv_eps"), (1, "divv_h")):
        ref = o["last"][name]
        d = np.abs(flow[k] - ref) / np.sqrt(np.mean(ref ** 2))
        report({"quantity": name, "median": float(np.median(d)), "p99": float(np.percentile(d, 99))})
        assert np.median(d) <= 1e-5 and np.percentile(d, 99) <= 1e-4


def _scattered_hot(n, hot, seed):
    # a sphere of cool gas in which single particles, here and there, are hot and take short steps
    w = W.evrard_sphere(n, seed=seed, sigma_v=0.05)
    w.u[np.random.default_rng(seed).choice(n, hot, replace=False)] *= np.float32(400.0)
    return w


@pytest.mark.parametrize("gas_only", [True, False])
def test_individual_steps_of_a_scattered_few(gas_only):
    # leaf lists over the entries of an active list; its walk in parts, the first and last in whole groups
    n = 70001
    w = _scattered_hot(n, 300, 15)
    if not gas_only:
        d = W.hernquist_gas(n - 30000, 30000, seed=16)
        d.u[:300] *= np.float32(400.0)
        w = d
    dt_max = 2.0 ** -9              # one to two in a hundred take shorter steps, down to an eighth
    ts = oracle.TimeStep(eta_acc=0.1, eta_courant=0.2, eta_u=0.0, dt_max=dt_max)
    o = oracle.run_bins(w, 1, ts, oracle.Bins(max_bin=3, wake_factor=0.0))
    (_, stats), st, _, bins = _integrate(w, lambda E, c, ds: E.evol_run_bins(
        c, ds.particles, ds.params, E.make_bins(3, 0.0, eta_acc=0.1, eta_courant=0.2, eta_u=0.0, dt_max=dt_max,
                                                predict_lengths=0), ds.outputs, 1))
    report({"quantity": "bins", "gpu": stats, "oracle": o["stats"]})
    # no step decision within FP32 rounding of a boundary: the same timeline
    assert o["stats"]["step_margin"] > 5e-5 and o["stats"]["system_steps"] > 2
    assert stats[0] == o["stats"]["system_steps"] and stats[1] == o["stats"]["active_evaluations"]
    assert 0 < (stats[1] - 2 * n) / (stats[0] - 1) < 2000
    assert np.array_equal(bins[0], o["tb"]) and np.array_equal(bins[1], o["te"])
    _positions_track(st, o)
    _lengths_track(w, st, o["last"])


def _lengths_track(w, st, last):
    for k in ("h", "eps"):
        ref = last[k][: w.n_gas] if k == "h" else last[k]
        err = np.abs(st[k][: len(ref)] / ref - 1.0)
        report({"quantity": k + "_after", "p99": float(np.percentile(err, 99)), "max": float(err.max())})
        assert np.percentile(err, 99) < 1e-5
