"""Trees in contexts of their own size: below 22 particles the scanned node counts
(22 levels) are more numerous than the particles.  Whole numbers, equal to the
oracle's, twice from the same context."""
import numpy as np
import pytest

import oracle
from paper_1909_07439_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [1, 16])
@pytest.mark.parametrize("n", [1, 2, 7, 21, 22, 23])
def test_tree_in_a_context_of_its_own_size(n, leaf):
    from paper_1909_07439_gb300 import DeviceState, build, native
    build.build()
    native.load()
    ctx = native.sph_create(n, 0)
    try:
        w = inputs.unit_sphere(n, seed=n)
        keys = oracle.morton_keys(w.pos)
        order = oracle.sort_order(keys)
        ch, cg = oracle.chop(keys[order], leaf), oracle.chop(keys[order], 8)
        term = cg.nchild == 0
        p = native.sph_params_default(n_leaf=leaf)
        s = DeviceState.from_arrays(w.pos, w.vel, w.h)
        for _ in range(2):
            native.sph_build_tree(ctx, s.c, p)
            native.sph_sync(ctx)
            assert np.array_equal(s.numpy("perm").astype(np.int64), order)
            assert np.array_equal(s.numpy("pos"), w.pos[order])
            nodes, groups = native.sph_get_tree(ctx)
            for f in ("level", "first", "count", "nchild"):
                assert np.array_equal(nodes[f], getattr(ch, f)), f
            assert np.array_equal(groups["first"], np.sort(cg.first[term]))
            assert np.array_equal(groups["count"], cg.count[term][np.argsort(cg.first[term])])
    finally:
        native.sph_destroy(ctx)
