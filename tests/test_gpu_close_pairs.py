"""drho/dt of the density pass where one close pair decides it.

A particle at rest whose only moving neighbour sits q = r / h of 2e-4 to 2e-3 away:
drho/dt = m (v . d / r) C f'(q) / (h^4 Omega) of that pair alone, so f' near 0 must
keep its relative precision.  Compared at the returned h and Omega: some 25
roundings of 2^-24 from the positions to the result, 1.5e-6."""
import numpy as np
import pytest

from oracle import adjoint_ref as R
from paper_1909_07439_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("scale", [1.0, 0.7])   # 0.7: h leaves its list pad, tree walks
@pytest.mark.parametrize("kernel,hfact", [(R.M4, 1.2), (R.WC6, 1.3)])
def test_density_rate_of_a_close_pair(kernel, hfact, scale):
    from paper_1909_07439_gb300 import DeviceState, build, native
    build.build()
    native.load()
    w = inputs.unit_sphere(6000, seed=2, hfact=hfact)
    far = np.nonzero(np.linalg.norm(w.pos[:, :3], axis=1) < 0.8)[0]
    at = [far[0]]
    for i in far:   # well apart: each has one moving neighbour
        if np.linalg.norm(w.pos[at, :3] - w.pos[i, :3], axis=1).min() > 0.35:
            at.append(i)
    at = np.array(at)
    assert len(at) >= 10
    rng = np.random.default_rng(1)
    e = rng.normal(size=(len(at), 3))
    e /= np.linalg.norm(e, axis=1, keepdims=True)
    q = np.geomspace(2e-4, 2e-3, len(at))
    x = w.pos[at].copy()
    x[:, :3] += (q * w.h[at])[:, None].astype(np.float32) * e.astype(np.float32)
    d = w.pos[at, :3].astype(np.float64) - x[:, :3]
    r = np.linalg.norm(d, axis=1)
    v = (0.3 * d / r[:, None]).astype(np.float32)
    w.vel[:, :3] = 0
    vel = w.vel[at].copy()
    vel[:, :3] = v
    s = DeviceState.from_arrays(np.concatenate([w.pos, x]), np.concatenate([w.vel, vel]),
                                np.float32(scale) * np.concatenate([w.h, w.h[at]]))
    ctx = native.sph_create(s.n, 0)
    try:
        p = native.sph_params_default(kernel=kernel, hfact=hfact)
        native.sph_build_tree(ctx, s.c, p)
        native.sph_density(ctx, s.c, p)
        native.sph_sync(ctx)
    finally:
        native.sph_destroy(ctx)
    h, om, got = (s.in_original_order(f)[at].astype(np.float64) for f in ("h", "omega", "drhodt"))
    df = R.kern(torch.tensor(r / h, dtype=torch.float64), kernel)[1].numpy()
    want = x[:, 3].astype(np.float64) * (-(v.astype(np.float64) * d).sum(1) / r) * R.C_NORM[kernel] * df / (h ** 4 * om)
    off = np.abs(got / want - 1).max()
    print(f"kernel {kernel} scale {scale}: drho/dt of a close pair off by {off:.1e}")
    assert off < 1.5e-6
