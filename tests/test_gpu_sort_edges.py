"""Tree build at the edges of its kernels: the counting sort of few particles and
the radix sort beside it, scans in one block and in three kernels, small chop
tiles, and a radix sort whose keys are in order already.  Keys, order, nodes and
groups are whole numbers and must equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1909_07439_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    from paper_1909_07439_gb300 import build, native
    build.build()
    native.load()
    ctx = native.sph_create(1 << 16, 0)
    yield native, ctx, torch
    native.sph_destroy(ctx)


def _build(native, ctx, s):
    p = native.sph_params_default()
    native.sph_build_tree(ctx, s.c, p)
    native.sph_sync(ctx)
    return p


def _check_tree(native, ctx, p, sk):
    nodes, groups = native.sph_get_tree(ctx)
    ch = oracle.chop(sk, p.n_leaf)
    for f in ("level", "first", "count", "nchild"):
        assert np.array_equal(nodes[f], getattr(ch, f)), f
    cg = oracle.chop(sk, p.n_group)
    term = cg.nchild == 0
    assert np.array_equal(groups["first"], np.sort(cg.first[term]))
    assert np.array_equal(groups["count"], cg.count[term][np.argsort(cg.first[term])])


# warp, chop tile, rank tile, one-block scan and counting-sort limits
@pytest.mark.parametrize("dups", [False, True])
@pytest.mark.parametrize("n", [31, 32, 33, 255, 256, 257, 1023, 1024, 1025, 8191, 8192, 8193, 2048 * 5,
                               2048 * 5 + 1, 40000])
def test_order_and_tree_at_edges(lib, n, dups):
    native, ctx, torch = lib
    from paper_1909_07439_gb300 import DeviceState
    w = inputs.unit_sphere(n, seed=n)
    if dups:  # equal keys keep their input order
        w.pos[n // 3: n // 3 + min(n // 2, 90), :3] = w.pos[0, :3]
    keys = oracle.morton_keys(w.pos)
    order = oracle.sort_order(keys)
    s = DeviceState.from_arrays(w.pos, w.vel, w.h)
    p = _build(native, ctx, s)
    assert np.array_equal(s.numpy("perm").astype(np.int64), order)
    assert np.array_equal(s.numpy("keys").view(np.uint64), keys[order])
    assert np.array_equal(s.numpy("pos"), w.pos[order])
    _check_tree(native, ctx, p, keys[order])


@pytest.mark.parametrize("size", [3, 20, 40])
def test_radix_sort_of_shared_top_bits(lib, size):
    # above the counting sort's limit: the fix-up of runs of equal top bits,
    # and with more than 32 of them the passes over all 64 bits
    native, ctx, torch = lib
    from paper_1909_07439_gb300 import DeviceState
    n = 20000
    w = inputs.unit_sphere(n, seed=size)
    rng = np.random.default_rng(size)
    at = rng.permutation(n)[: (n // (2 * size)) * size].reshape(-1, size)
    w.pos[at[:, 1:], :3] = (w.pos[at[:, :1], :3] +
                            rng.uniform(-1e-6, 1e-6, at[:, 1:].shape + (3,)).astype(np.float32))
    keys = oracle.morton_keys(w.pos)
    order = oracle.sort_order(keys)
    s = DeviceState.from_arrays(w.pos, w.vel, w.h)
    p = _build(native, ctx, s)
    assert np.array_equal(s.numpy("perm").astype(np.int64), order)
    _check_tree(native, ctx, p, keys[order])


# (0, 1): lanes of one warp; (31, 32), (255, 256): over the edge of a warp and
# of a block; the last pair, and a pair far apart
@pytest.mark.parametrize("swap", [None, (0, 1), (31, 32), (255, 256), (-2, -1), (5, -3)])
@pytest.mark.parametrize("n", [8193, 30011])
def test_keys_in_order_already(lib, n, swap):
    native, ctx, torch = lib
    from paper_1909_07439_gb300 import DeviceState
    w = inputs.unit_sphere(n, seed=3)
    w.pos[100:140, :3] = w.pos[100, :3]
    o = oracle.sort_order(oracle.morton_keys(w.pos))
    if swap:
        a, b = swap
        o[a], o[b] = o[b], o[a]
    pos, vel, h = w.pos[o], w.vel[o], w.h[o]
    keys = oracle.morton_keys(pos)
    order = oracle.sort_order(keys)
    assert (swap is None) == np.array_equal(order, np.arange(n))
    s = DeviceState.from_arrays(pos, vel, h)
    p = _build(native, ctx, s)
    assert np.array_equal(s.numpy("perm").astype(np.int64), order)
    assert np.array_equal(s.numpy("vel"), vel[order])
    _check_tree(native, ctx, p, keys[order])


@pytest.mark.parametrize("swap", [None, (4095, 4096), (4998, 4999), (5000, 5001), (9000, 9001)])
def test_batch_in_order_already(lib, swap):
    # the order is (instance, key): neighbours over an instance's end are in
    # order whatever their keys
    native, ctx, torch = lib
    from paper_1909_07439_gb300 import DeviceState
    off = np.array([0, 5000, 6000, 11000], np.int64)
    w = inputs.unit_sphere(int(off[-1]), seed=9)
    want = np.empty(w.n, np.int64)
    for a, b in zip(off[:-1], off[1:]):
        o = a + oracle.sort_order(oracle.morton_keys(w.pos[a:b]))
        w.pos[a:b], w.vel[a:b], w.h[a:b] = w.pos[o], w.vel[o], w.h[o]
    if swap:
        i, j = swap
        w.pos[[i, j]] = w.pos[[j, i]]
    for a, b in zip(off[:-1], off[1:]):
        want[a:b] = a + oracle.sort_order(oracle.morton_keys(w.pos[a:b]))
    s = DeviceState.from_arrays(w.pos, w.vel, w.h)
    dt = torch.zeros(3, dtype=torch.float32, device="cuda")
    native.sph_batch_evaluate(ctx, s.c, torch.as_tensor(off, device="cuda"), 3, native.sph_params_default(), dt)
    torch.cuda.synchronize()
    assert np.array_equal(s.numpy("perm").astype(np.int64), want)
    assert np.array_equal(s.numpy("pos"), w.pos[want])
