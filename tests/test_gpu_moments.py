"""Node moments formed by eight lanes to a node: every node against FP64 sums over its particles, with leaves
smaller and larger than eight, massless nodes, coincident particles in a leaf at the deepest level, and a box
whose offset is much larger than its extent.

Bounds: a node's sums go through at most 8 additions in a lane, 3 across the lanes and 3 on each of up to 21
levels, about 75 roundings of 6e-8 relative to the terms: 5e-6 of M; with the products' own, 1e-5 of l for the
centre of mass (and one rounding of its coordinates) and for delta; the quadrupole's terms add up to less than
3 M l^2 and take the centre's error twice: 1e-4 of M l^2."""
import numpy as np
import pytest

from paper_0912_1786_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _set(n, offset, seed):
    r = np.random.default_rng(seed)
    x = r.normal(size=(n, 3))
    x[: n // 4] = 0.01 * x[: n // 4] + 0.7                      # a dense clump
    m = r.uniform(0.5, 1.5, n)
    m[x[:, 0] < -0.8] = 0.0                                     # whole cells without mass
    x[n - 5:] = x[n - 5]                                        # more in one place than a small leaf holds
    return (x + offset).astype(np.float32), m.astype(np.float32)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("offset", [0.0, 1000.0])
@pytest.mark.parametrize("n,leaf", [(9, 1), (33, 8), (1000, 7), (5000, 9), (40000, 24), (40000, 64), (200000, 3)])
def test_every_node(n, leaf, offset, precision):
    import torch
    from paper_0912_1786_gb300 import build, evol as E
    from paper_0912_1786_gb300.device import DeviceSet

    build.build()
    x, m = _set(n, offset, n + leaf)
    zero, one = np.zeros(n, np.float32), np.ones(n, np.float32)
    w = W.Workload("moments", x=x[:, 0].copy(), y=x[:, 1].copy(), z=x[:, 2].copy(), vx=zero, vy=zero, vz=zero, m=m,
                   u=zero, h=one, eps=one, n_gas=0, params=W.Params(sph=0, adaptive_softening=0, leaf_size=leaf))
    ds = DeviceSet(w, w.params, precision=precision)
    ctx = E.evol_create(n, torch.cuda.current_stream().cuda_stream)
    try:
        E.evol_build_tree(ctx, ds.particles, ds.params)
        assert E.evol_sync(ctx, raise_on_error=False) == 0
        perm = E.evol_get_debug(ctx, E.EVOL_DBG_PERM, np.int32)
        cube = E.evol_get_debug(ctx, E.EVOL_DBG_CUBE, np.float64)
        nd = E.evol_get_debug(ctx, E.EVOL_DBG_NODES, np.int32)
        nn = nd.size // 5
        begin, end, level = nd.reshape(5, nn)[:3]
        g = E.evol_get_debug(ctx, E.EVOL_DBG_MOMENTS, np.float32).reshape(nn, 20).astype(np.float64)
    finally:
        E.evol_destroy(ctx)
    xs, ms = x[perm].astype(np.float64), m[perm].astype(np.float64)
    lo = np.array([xs[b:e].min(0) for b, e in zip(begin, end)])
    hi = np.array([xs[b:e].max(0) for b, e in zip(begin, end)])
    assert np.array_equal(g[:, 11:14], lo) and np.array_equal(g[:, 14:17], hi)

    def over_nodes(v):
        c = np.concatenate([np.zeros((1,) + v.shape[1:], np.longdouble), np.cumsum(v, 0, dtype=np.longdouble)])
        return (c[end] - c[begin]).astype(np.float64)

    # about the middle of the set, so that the differences of prefix sums keep their digits
    y = xs - offset
    M = over_nodes(ms)
    S = over_nodes(ms[:, None] * y)
    full = M > 1e-9
    com = np.where(full[:, None], S / np.where(full, M, 1.0)[:, None], 0.5 * (lo + hi) - offset)
    l = cube[3] * 0.5 ** level
    cell = np.floor((lo - cube[:3]) / l[:, None])               # lower corner's cell
    cell = np.minimum(cell, 2.0 ** level[:, None] - 1)
    centre = cube[:3] + (cell + 0.5) * l[:, None] - offset
    delta = np.sqrt(((com - centre) ** 2).sum(1))
    P = over_nodes(ms[:, None, None] * y[:, :, None] * y[:, None, :])
    P = P - M[:, None, None] * com[:, :, None] * com[:, None, :]
    tr = np.trace(P, axis1=1, axis2=2)
    Q = np.stack([3 * P[:, 0, 0] - tr, 3 * P[:, 1, 1] - tr, 3 * P[:, 2, 2] - tr, 3 * P[:, 0, 1], 3 * P[:, 0, 2],
                  3 * P[:, 1, 2]], 1)
    assert np.abs(g[:, 0] - M).max() <= 5e-6 * M.max() and np.all(np.abs(g[:, 0] - M) <= 5e-6 * M + 1e-12 * M.max())
    away = np.abs(com + offset) * 6e-8 + 1e-5 * l[:, None] + 1e-12
    assert np.all(np.abs(g[:, 1:4] - offset - com) <= away)
    assert np.all(np.abs(g[:, 10] - delta) <= 2e-5 * l + 1e-12)
    assert np.all(np.abs(g[:, 4:10] - np.where(full[:, None], Q, 0.0)) <= 1e-4 * (M * l * l)[:, None] + 1e-11)
