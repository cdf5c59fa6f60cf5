"""Evaluations whose neighbour lists do not fit: more neighbours than the kernels'
usual hfact gives.  Every batch walks the tree, with tiles of 128 to 384 entries, and
past those the lists are summed piece by piece.  Same bars as the other parity tests:
h and rho 1e-5 relative, Omega 1e-5 and accelerations 1e-4 of the largest."""
import numpy as np
import pytest

import oracle
from paper_1909_07439_gb300 import inputs

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

M4, M6, WC6 = 0, 1, 2


# 1.25 (4/3) pi (R 1.03 hfact)^3 entries expected: 154, 187, 225, 267, 361, 557; 267,
# 633; 314, 557
@pytest.mark.parametrize("kernel,hfact", [(M4, 1.5), (M4, 1.6), (M4, 1.7), (M4, 1.8), (M4, 1.99), (M4, 2.3),
                                          (M6, 1.2), (M6, 1.6), (WC6, 1.9), (WC6, 2.3)])
@pytest.mark.parametrize("tile", [0, 64])
def test_evaluation_with_many_neighbours(kernel, hfact, tile):
    from paper_1909_07439_gb300 import DeviceState, build, native
    build.build()
    native.load()
    w = inputs.unit_sphere(3001, seed=17, sigma_v=0.3, hfact=hfact)
    x, v, m, u = (a.astype(np.float64) for a in (w.pos[:, :3], w.vel[:, :3], w.pos[:, 3], w.vel[:, 3]))
    hf = float(np.float32(hfact))
    d = oracle.density(x, v, m, w.h, hfact=hf, kernel=kernel)
    f = oracle.force(x, v, m, u, d.h, d.rho, d.omega, gamma=float(np.float32(5 / 3)), kernel=kernel)
    ctx = native.sph_create(w.n, 0)
    try:
        p = native.sph_params_default(kernel=kernel, hfact=hfact, tile=tile)
        s = DeviceState.from_arrays(w.pos, w.vel, w.h)
        native.sph_build_tree(ctx, s.c, p)
        native.sph_density(ctx, s.c, p)
        native.sph_force(ctx, s.c, p)
        native.sph_sync(ctx)
        st = native.sph_get_stats(ctx)
    finally:
        native.sph_destroy(ctx)
    assert st["density_rewalks"] > 0
    h, rho, om, dr, acc = (s.in_original_order(k).astype(np.float64) for k in ("h", "rho", "omega", "drhodt", "acc"))
    assert np.max(np.abs(h / d.h - 1)) < 1e-5
    assert np.max(np.abs(rho / d.rho - 1)) < 1e-5
    assert np.max(np.abs(om - d.omega)) < 1e-5 * np.max(np.abs(d.omega))
    assert np.max(np.abs(dr - d.drhodt)) < 1e-4 * np.max(np.abs(d.drhodt))
    assert np.max(np.abs(acc[:, :3] - f.acc)) < 1e-4 * np.max(np.abs(f.acc))
    assert np.max(np.abs(acc[:, 3] - f.dudt)) < 1e-4 * np.max(np.abs(f.dudt))
