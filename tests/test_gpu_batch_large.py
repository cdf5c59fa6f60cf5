"""A batch so large that a warp of the per-instance reductions (box, Courant step)
combines several rounds of 32 particles, over instance ends anywhere in them.  Keys
and order are whole numbers and follow from each instance's box; the step is a
minimum, so it is that of the returned h and vsigmax."""
import numpy as np
import pytest

import oracle
from paper_1909_07439_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# ends inside a round, at its edge, several in one round and several rounds apart
SIZES = [100003, 9, 31, 17, 32, 33, 8, 60001, 95, 97, 2049, 12, 12, 12, 120011, 64, 50021, 10]


def test_boxes_and_steps_of_a_large_batch():
    from paper_1909_07439_gb300 import DeviceState, build, native
    build.build()
    native.load()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    off = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    n = int(off[-1])
    assert n > 2 * 32 * 8 * 4 * sms     # three rounds a warp
    parts = [inputs.unit_sphere(k, seed=i) for i, k in enumerate(SIZES)]
    pos, vel, h = (np.concatenate([getattr(w, f) for w in parts]) for f in ("pos", "vel", "h"))
    for i, (a, b) in enumerate(zip(off[:-1], off[1:])):
        pos[a:b, :3] += np.float32(i)   # boxes that differ
    s = DeviceState.from_arrays(pos, vel, h)
    dt = torch.zeros(len(SIZES), dtype=torch.float32, device="cuda")
    ctx = native.sph_create(n, 0)
    try:
        p = native.sph_params_default()
        native.sph_batch_evaluate(ctx, s.c, torch.as_tensor(off, device="cuda"), len(SIZES), p, dt)
        native.sph_sync(ctx)
    finally:
        native.sph_destroy(ctx)
    perm, keys = s.numpy("perm").astype(np.int64), s.numpy("keys").view(np.uint64)
    own = np.float32(0.3) * (s.numpy("h") / s.numpy("vsigmax"))
    for i, (a, b) in enumerate(zip(off[:-1], off[1:])):
        k = oracle.morton_keys(pos[a:b])
        order = oracle.sort_order(k)
        assert np.array_equal(perm[a:b], a + order), i
        assert np.array_equal(keys[a:b], k[order]), i
        assert abs(float(dt[i]) / float(own[a:b].min()) - 1) <= 2.0 ** -22, i   # two roundings
