"""max_h_iter bounds the whole solve of a particle, also where its batch is handed
from the neighbour lists to tree walks on the way (include/sph.h).

The sweeps that each particle needs come from the same bracketed Newton iteration in
64 bits on the CPU; with h_tol = 1e-4 and the last steps not near it the 32-bit solve
needs the same number."""
import numpy as np
import pytest

from oracle import adjoint_ref as R
from paper_1909_07439_gb300 import inputs

pytest.importorskip("torch")
import torch  # noqa: E402

TOL, HFACT = 1e-4, 1.2


def _sweeps(w, h):
    """Sweeps of the density sums until every particle's step is below TOL h, and the largest
    step of each sweep over TOL h."""
    x, m = w.pos[:, :3].astype(np.float64), w.pos[:, 3].astype(np.float64)
    r = np.linalg.norm(x[:, None] - x[None], axis=2)
    M, C = m * HFACT ** 3, R.C_NORM[R.M4]
    h, lo, hi = h.astype(np.float64), np.zeros(w.n), np.full(w.n, np.inf)
    done, need, most = np.zeros(w.n, bool), np.zeros(w.n, int), []
    for k in range(1, 60):
        q = r / h[:, None]
        f, df = (t.numpy() for t in R.kern(torch.tensor(q), R.M4))
        gt, gp = C * (m * f).sum(1) - M, 3 * M - C * (m * (3 * f + q * df)).sum(1)
        lo, hi = np.where(~done & (gt < 0), h, lo), np.where(~done & (gt >= 0), h, hi)
        hn = h * (1 - gt / gp)
        ok = (gp > 0) & (hn >= lo) & (hn <= hi) & (hn >= 0.5 * h) & (hn <= 2 * h)
        with np.errstate(invalid="ignore"):
            alt = np.where((lo > 0) & np.isfinite(hi), 0.5 * (lo + hi), np.where(gt < 0, 2 * h, 0.5 * h))
        hn = np.where(ok, hn, alt)
        step = np.abs(hn - h) / (TOL * h)
        most.append(step[~done].max())
        need[~done] = k
        done_now = step < 1
        h = np.where(done | done_now, h, hn)
        done |= done_now
        if done.all():
            return need, most
    raise AssertionError("no convergence")


def _case():
    w = inputs.unit_sphere(700, seed=6, hfact=HFACT)
    h = (0.6 * w.h).astype(np.float32)   # the first step leaves the lists' pad of 3 %
    return w, h


def test_the_case_is_decided():
    need, most = _sweeps(*_case())
    assert need.max() >= 5 and len(most) == need.max()
    # FP32 moves a step of 1e-4 h by some 1e-7 h, 0.1 %
    assert most[-1] < 0.9 and min(most[:-1]) > 1.1


@pytest.mark.gpu
@pytest.mark.parametrize("less", [0, 1, 2])
def test_cap_counts_the_updates_before_the_walks(less):
    from paper_1909_07439_gb300 import DeviceState, build, native
    build.build()
    native.load()
    w, h = _case()
    cap = int(_sweeps(w, h)[0].max()) - less
    ctx = native.sph_create(w.n, 0)
    try:
        p = native.sph_params_default(max_h_iter=cap, h_tol=TOL)
        s = DeviceState.from_arrays(w.pos, w.vel, h)
        native.sph_build_tree(ctx, s.c, p)
        native.sph_density(ctx, s.c, p)
        if less == 0:
            native.sph_sync(ctx)
            assert native.sph_get_stats(ctx)["density_rewalks"] > 0
        else:
            with pytest.raises(native.SphError, match="NOT_CONVERGED"):
                native.sph_sync(ctx)
    finally:
        native.sph_destroy(ctx)
