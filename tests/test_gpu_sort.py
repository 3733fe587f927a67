"""The tree's order: keys and permutation of every form of the sort against a stable numpy sort, bit for bit, at
sizes around the ends of its tiles and around the sizes where one form takes over from the next, with distinct
and with many equal keys, for one system and for several."""
import numpy as np
import pytest

from paper_0912_1786_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _spread(v):
    out = np.zeros_like(v)
    for b in range(21):
        out |= ((v >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b)
    return out


def _keys(x):
    """Morton keys of one system's positions, in double as the oracle has them."""
    lo = x.min(0).astype(np.float64)
    ext = float((x.max(0).astype(np.float64) - lo).max())
    side = 2.0 ** np.ceil(np.log2(ext * (1 + 2.0 ** -20))) if ext > 0 else 1.0
    q = np.clip(np.floor((x.astype(np.float64) - lo) * (2.0 ** 21 / side)), 0, 2 ** 21 - 1).astype(np.uint64)
    return (_spread(q[:, 0]) << np.uint64(2)) | (_spread(q[:, 1]) << np.uint64(1)) | _spread(q[:, 2])


def _positions(n, cells, seed):
    r = np.random.default_rng(seed)
    if cells:
        return (r.integers(0, cells, (n, 3)) / cells).astype(np.float32)
    return (r.normal(size=(n, 3)) * np.array([1.0, 0.3, 1e-3]) + np.array([3.0, -1e-3, 40.0])).astype(np.float32)


def _check(offs, cells, seed, x=None):
    import torch
    from paper_0912_1786_gb300 import build, evol as E
    from paper_0912_1786_gb300.device import DeviceSet

    build.build()
    n = offs[-1]
    x = x if x is not None else np.concatenate([_positions(b - a, cells, seed + k) for k, (a, b) in enumerate(zip(offs[:-1], offs[1:]))])
    zero = np.zeros(n, np.float32)
    one = np.ones(n, np.float32)
    w = W.Workload("sort", x=x[:, 0].copy(), y=x[:, 1].copy(), z=x[:, 2].copy(), vx=zero, vy=zero, vz=zero, m=one,
                   u=zero, h=one, eps=one, n_gas=0, params=W.Params(theta=0.5, sph=0, adaptive_softening=0))
    ds = DeviceSet(w, w.params)
    ctx = E.evol_create(n, torch.cuda.current_stream().cuda_stream)
    try:
        if len(offs) > 2:
            E.evol_step_batched(ctx, offs, ds.particles, ds.params, ds.outputs)
        else:
            E.evol_build_tree(ctx, ds.particles, ds.params)
        assert E.evol_sync(ctx, raise_on_error=False) == 0
        keys = E.evol_get_debug(ctx, E.EVOL_DBG_KEYS, np.uint64)
        perm = E.evol_get_debug(ctx, E.EVOL_DBG_PERM, np.int32)
    finally:
        E.evol_destroy(ctx)
    for a, b in zip(offs[:-1], offs[1:]):
        k = _keys(x[a:b])
        order = np.argsort(k, kind="stable")
        assert np.array_equal(perm[a:b] - a, order)
        assert np.array_equal(keys[a:b], k[order])


@pytest.mark.parametrize("cells", [0, 4])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 1023, 1025, 2048, 12287, 12288, 12289, 14336, 131071, 131072, 131073,
                               300001])
def test_one_system(n, cells):
    _check([0, n], cells, n)


@pytest.mark.parametrize("cells", [0, 4])
@pytest.mark.parametrize("systems,size", [(2, 33), (300, 37), (300, 50), (257, 509), (700, 200), (3, 2999), (3, 9000)])
def test_several_systems(systems, size, cells):
    # sizes differ: every third system is a single particle
    sizes = [1 if k % 3 == 2 else size + k % 5 for k in range(systems)]
    _check([0] + [int(v) for v in np.cumsum(sizes)], cells, systems)


@pytest.mark.parametrize("low", [0.0, 1e-9, -1e-9, 1e-25, -1e-25, 1e-43, 0.3, -7.7, 1e6])
@pytest.mark.parametrize("size", [1.0, 3.7e-6, 2.5e9, 1e-36, 1e30])
def test_cell_edges(low, size):
    # positions on and next to the edges of cells, with corners that the differences to them round away in
    # float, in double, or not at all: the keys are formed in float arithmetic but must be those of double
    r = np.random.default_rng(int(abs(np.log(size)) * 10))
    lo = np.float32(low)
    t = (r.integers(0, 2 ** 21, (4000, 3)) / 2.0 ** 21 * size).astype(np.float32)
    t[:1500] += lo                                             # edges counted from the corner
    step = r.integers(-1, 2, t.shape)
    x = np.where(step > 0, np.nextafter(t, np.float32(np.inf)), np.where(step < 0, np.nextafter(t, lo), t))
    x = np.maximum(x, lo).astype(np.float32)
    x[0] = lo
    x[1] = lo + np.float32(size)
    _check([0, len(x)], 0, 0, x)
