"""The backward of the differentiable evaluation (adjoint.evaluate): the state it
differentiates at, with lists, and its gradients where the tests of small, converged
clouds do not reach (the radix sort, a fixed number of Newton updates)."""
import numpy as np
import pytest

import oracle
from paper_1909_07439_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
from oracle import adjoint_ref as R  # noqa: E402

T = torch.float64
HFACT = {R.M4: 1.2, R.M6: 0.9, R.WC6: 1.3}


@pytest.fixture(scope="module")
def lib():
    from paper_1909_07439_gb300 import build, native
    build.build()
    native.load()
    ctx = native.sph_create(1 << 16, 0)
    yield native, ctx
    native.sph_destroy(ctx)


def _cloud(n, seed, kernel):
    w = inputs.unit_sphere(n, seed=seed, sigma_v=0.3, hfact=HFACT[kernel])
    rng = np.random.default_rng(seed)
    w.vel[:, 3] *= rng.uniform(0.5, 2.0, n).astype(np.float32)
    return w, rng.normal(size=(n, 4)).astype(np.float32)


def _evaluate(ctx, w, p):
    from paper_1909_07439_gb300.adjoint import evaluate
    pos, vel = (torch.tensor(a, device="cuda", requires_grad=True) for a in (w.pos, w.vel))
    al = torch.tensor(1.0, dtype=T, requires_grad=True)
    return pos, vel, al, evaluate(ctx, pos, vel, torch.tensor(w.h, device="cuda"), al, p)


# the rough h of a sphere's edge leaves the lists' pad in the forward pass; on both
# sides of the counting sort's limit
@pytest.mark.parametrize("n,kernel,iters", [(2003, R.M4, 0), (2003, R.M4, 3), (9001, R.WC6, 0), (9001, R.M6, 3)])
def test_backward_is_taken_at_the_forward_values(lib, monkeypatch, n, kernel, iters):
    native, ctx = lib
    from paper_1909_07439_gb300 import adjoint
    made, seen = [], {}

    class Recorded(adjoint.DeviceState):
        def __init__(self, *a, **k):
            super().__init__(*a, **k)
            made.append(self)

    force_bwd = native.sph_force_bwd

    def record(c, s, *a, **k):
        seen.update({f: getattr(made[-1], f)[:n].clone() for f in ("h", "rho", "omega")})
        return force_bwd(c, s, *a, **k)

    monkeypatch.setattr(adjoint, "DeviceState", Recorded)
    monkeypatch.setattr(native, "sph_force_bwd", record)
    w, g = _cloud(n, 5, kernel)
    p = native.sph_params_default(kernel=kernel, hfact=HFACT[kernel], density_iters=iters)
    _, _, _, out = _evaluate(ctx, w, p)
    order = made[0].perm[:n].long()
    before = native.sph_get_stats(ctx)
    assert before["density_rewalks"] > 0        # the case has batches that leave the pad
    torch.autograd.backward(out[3], torch.tensor(g, device="cuda"))
    after = native.sph_get_stats(ctx)  # since the call before
    for name, o in zip(("h", "rho", "omega"), out):
        assert torch.equal(seen[name], o.detach()[order]), name
    # only a particle without a list is walked (its list overflowed)
    assert after["list_overflows"] > 0 or after["density_rewalks"] == 0


@pytest.mark.parametrize("n,kernel,iters", [(9001, R.WC6, 0), (9001, R.M4, 0), (1500, R.M4, 7), (1500, R.M6, 7)])
def test_gradients_match_fp64_autograd(lib, n, kernel, iters):
    # seven Newton updates reach the root to rounding: the reference's
    native, ctx = lib
    w, g = _cloud(n, 21, kernel)
    p = native.sph_params_default(kernel=kernel, hfact=HFACT[kernel], density_iters=iters)
    pos, vel, al, out = _evaluate(ctx, w, p)
    gh = np.random.default_rng(3).normal(size=n).astype(np.float32)
    cot = [torch.tensor(gh, device="cuda")] * 3 + [torch.tensor(g, device="cuda")]
    torch.autograd.backward(out, cot)
    x, v, u = (torch.tensor(a, dtype=T, requires_grad=True) for a in (w.pos[:, :3], w.vel[:, :3], w.vel[:, 3]))
    m, hfact = torch.tensor(w.pos[:, 3], dtype=T), float(np.float32(HFACT[kernel]))
    d = oracle.density(w.pos[:, :3].astype(np.float64), w.vel[:, :3].astype(np.float64),
                       w.pos[:, 3].astype(np.float64), w.h, hfact=hfact, kernel=kernel)
    h = torch.tensor(d.h, dtype=T)
    i, j = R.pair_list(x.detach(), h, 1.01, kernel=kernel)
    # the derivatives of the root, at the values that the forward returned: 1 / sqrt|P_i - P_j|
    # of the conduction speed is large where a pair's pressures nearly agree
    root = R.density(x, m, h, i, j, hfact, kernel=kernel)
    h, rho, om = (r + (o.detach().cpu().double() - r.detach()) for r, o in zip(root, out))
    gamma = float(np.float32(5 / 3))
    acc = [torch.cat([a, b[:, None]], 1) for a, b in
           (R.force(x, v, u, m, h, rho, om, i, j, gamma=gamma, alpha=al_, kernel=kernel) for al_ in (0.0, 1.0))]
    torch.autograd.backward((h, rho, om, acc[1]), [torch.tensor(c, dtype=T) for c in (gh, gh, gh, g)])
    rel = lambda a, b: float((a.cpu().double() - b).norm() / b.norm())  # noqa: E731
    assert rel(pos.grad[:, :3], x.grad) < 1e-3
    assert rel(vel.grad[:, :3], v.grad) < 1e-3
    assert rel(vel.grad[:, 3], u.grad) < 1e-3
    # dL/dalpha = sum_i t_i, t_i = g_i . (A_i(1) - A_i(0)), A_i = (a_i, du_i/dt): terms
    # of both signs, so its error is held against their 2-norm: an h up to h_tol = 1e-6
    # off its root times the terms' sensitivity to their own and their neighbours' h
    # (some 5 each)
    t = (torch.tensor(g, dtype=T) * (acc[1] - acc[0])).sum(1).detach()
    off = abs(float(al.grad) - float(t.sum())) / float(t.norm())
    print(f"n {n} kernel {kernel} iters {iters}: dL/dalpha off by {off:.1e} of the terms' norm")
    assert off < 7e-6


def test_backward_again_and_through_saved_tensor_hooks(lib):
    native, ctx = lib
    w, g = _cloud(1200, 8, R.M4)
    p = native.sph_params_default()
    cot = torch.tensor(g, device="cuda")

    def grads(hooks, times):
        with hooks:
            pos, vel, al, out = _evaluate(ctx, w, p)
        out[0].mul_(2.0)    # the outputs are the caller's
        for k in range(times):
            for t in (pos, vel, al):
                t.grad = None
            torch.autograd.backward(out[3], cot, retain_graph=k + 1 < times)
        return pos.grad, vel.grad, al.grad

    plain = lambda t: t  # noqa: E731
    want = grads(torch.autograd.graph.saved_tensors_hooks(plain, plain), 1)
    for hooks, times in ((torch.autograd.graph.saved_tensors_hooks(plain, plain), 2),
                         (torch.autograd.graph.save_on_cpu(pin_memory=True), 1),
                         (torch.autograd.graph.saved_tensors_hooks(lambda t: t.double(), plain), 1)):
        got = grads(hooks, times)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        assert abs(float(got[2]) / float(want[2]) - 1) < 1e-12     # FP64 sum in any order
    with pytest.raises(TypeError):
        grads(torch.autograd.graph.saved_tensors_hooks(lambda t: t.cpu(), plain), 1)
