"""torch.autograd.Functions over libsph's differentiable forms.

``evaluate(ctx, pos, velu, h0, alpha, params)``: one evaluation (tree build,
density solve, force pass) returning h, rho, Omega and acc = (a, du/dt) in
the caller's particle order; its backward takes arbitrary cotangents of those
outputs and returns dL/dx, dL/d(v, u) and dL/dalpha_AV from the library's
adjoint kernels (sph_force_bwd, then sph_density_bwd through the h-rho
fixed point by the implicit-function theorem), taken at the forward's own h, rho
and Omega.  The backward rebuilds the tree and the neighbour lists, so the context
may be used for other work in between.

``rollout_loss(ctx, pos, velu, h, alpha, ...)`` returns the scalar loss
(mean squared density of probe particles after n_steps leapfrog steps) as a
torch tensor whose backward gives dL/d(velocities, internal energies) and
dL/dalpha_AV from the library's adjoint rollout (sph_rollout).

Marshalling only: the forward and backward sweeps run in libsph.
"""
from __future__ import annotations

import torch

from . import native
from .state import DeviceState


def _params(params, alpha):
    p = native.sph_params_default(**{k: getattr(params, k) for k, _ in params._fields_})
    p.alpha_av = float(alpha)
    return p


def _check_cuda_f32(**arrays):
    for name, t in arrays.items():
        if t.dtype != torch.float32 or not t.is_cuda:
            raise TypeError(f"{name} must be a float32 CUDA tensor")


def _state(pos, velu, h):
    """A fresh state with these particles."""
    s = DeviceState(pos.shape[0], device=pos.device, zero=False)
    s.pos[: s.n].copy_(pos.detach())
    s.vel[: s.n].copy_(velu.detach())
    s.h[: s.n].copy_(h.detach())
    return s


class _Evaluate(torch.autograd.Function):
    @staticmethod
    def forward(fctx, pos, velu, h0, alpha, handle, params):
        p = _params(params, alpha)
        s = _state(pos, velu, h0)
        native.sph_build_tree(handle, s.c, p)
        native.sph_density(handle, s.c, p)
        native.sph_force(handle, s.c, p)
        native.sph_sync(handle)
        perm = s.perm[: s.n].long()
        n = s.n
        out = []
        for f in ("h", "rho", "omega", "acc"):
            a = getattr(s, f)[:n]
            out.append(torch.empty_like(a).index_copy_(0, perm, a))   # curve order -> caller order
        # the inputs too: a change of theirs before the backward pass is an error;
        # the outputs' values in curve order and the order (16 bytes per particle)
        # are copies, so that the caller may change the outputs
        fctx.save_for_backward(pos, velu, h0, alpha, s.perm, s.h, s.rho, s.omega)
        fctx.handle, fctx.p = handle, p
        return tuple(out)

    @staticmethod
    def backward(fctx, gh, grho, gom, gacc):
        pos, velu, h0, alpha, perm, h, rho, omega = fctx.saved_tensors
        # the library takes raw pointers; a saved-tensor hook may return anything
        if not all(t.is_cuda for t in (pos, velu, perm, h, rho, omega)):
            raise TypeError("evaluate's saved tensors must be on the GPU")
        handle, p = fctx.handle, fctx.p
        n, dev = pos.shape[0], pos.device
        perm = perm.long()
        # The forward's tree and the lists of its h, rho and Omega, at which it is
        # differentiated: the state in the forward's curve order (the sort is the
        # identity), one sweep of the density pass that accepts any h (a Newton
        # step is at most h), so that no batch leaves the list pad, and the
        # forward's rho and Omega in place of that sweep's.  The adjoint passes
        # read nothing of a force pass.
        s = DeviceState(n, device=dev, zero=False)
        s.pos, s.vel = (t.detach().to(torch.float32).index_select(0, perm) for t in (pos, velu))
        s.h.copy_(h)
        q = _params(p, p.alpha_av)
        q.density_iters, q.h_tol = 0, 4.0
        native.sph_build_tree(handle, s.c, p)
        native.sph_density(handle, s.c, q)
        s.rho, s.omega = (t.to(torch.float32).contiguous() for t in (rho, omega))

        def to_curve(g, shape):
            return (torch.zeros(shape, dtype=torch.float32, device=dev) if g is None
                    else g.to(torch.float32).index_select(0, perm))

        gacc_c = to_curve(gacc, (n, 4))
        gpos_c, gvel_c = torch.empty((2, n, 4), dtype=torch.float32, device=dev)
        gh_f, grho_f, gom_f = torch.empty((3, n), dtype=torch.float32, device=dev)
        galpha = torch.zeros(1, dtype=torch.float64, device=dev)
        native.sph_force_bwd(handle, s.c, p, gacc_c, gpos_c, gvel_c, gh_f, grho_f, gom_f, galpha)
        for f, g in ((gh_f, gh), (grho_f, grho), (gom_f, gom)):
            if g is not None:
                f.add_(to_curve(g, (n,)))
        native.sph_density_bwd(handle, s.c, p, gh_f, grho_f, gom_f, gpos_c)
        native.sph_sync(handle)
        # the masses are constants of the problem: gpos_c's last column is zero
        gpos = torch.empty_like(gpos_c).index_copy_(0, perm, gpos_c)
        gvel = torch.empty_like(gvel_c).index_copy_(0, perm, gvel_c)
        return gpos, gvel, None, galpha.reshape(()).to(device=alpha.device, dtype=alpha.dtype), None, None


def evaluate(handle, pos, velu, h0, alpha, params):
    """One differentiable SPH evaluation (Eqs. 1-4 and 9-15).

    pos [n,4] (x, y, z, m), velu [n,4] (vx, vy, vz, u), h0 [n] (starting
    guess of the h-rho solve, not differentiated): float32 CUDA tensors;
    alpha: 0-dim tensor (alpha_AV); params: sph_params (alpha_av replaced by
    alpha); handle: a context with max_n >= n.  Returns (h, rho, Omega,
    acc) in the caller's order, acc [n,4] = (a xyz, du/dt); gradients flow to
    the positions, velocities, internal energies and alpha (masses get zero)."""
    _check_cuda_f32(pos=pos, velu=velu, h0=h0)
    if pos.shape != velu.shape or pos.shape[-1] != 4 or h0.shape != pos.shape[:1]:
        raise ValueError("pos and velu must be [n, 4] and h0 [n]")
    return _Evaluate.apply(pos, velu, h0, alpha, handle, params)


class _Rollout(torch.autograd.Function):
    @staticmethod
    def forward(fctx, velu, alpha, pos, h, handle, params, n_steps, ckpt, probes):
        p = _params(params, alpha)
        st = native.sph_state()
        st.n = pos.shape[0]
        st.pos, st.vel, st.h = pos.data_ptr(), velu.data_ptr(), h.data_ptr()
        need = velu.requires_grad or alpha.requires_grad
        g = torch.zeros_like(velu, memory_format=torch.contiguous_format) if need else None
        loss, ga = native.sph_rollout(handle, st, p, n_steps, ckpt, probes, probes.numel(), g)
        if need:
            fctx.save_for_backward(g)
            fctx.ga = ga
        return torch.tensor(loss, dtype=torch.float64, device=velu.device)

    @staticmethod
    def backward(fctx, gl):
        (g,) = fctx.saved_tensors
        s = gl.to(torch.float32)
        return (g * s, gl * fctx.ga, None, None, None, None, None, None, None)


def rollout_loss(handle, pos, velu, h, alpha, params, n_steps, ckpt, probes):
    """pos [n,4] (x,y,z,m), velu [n,4] (vx,vy,vz,u), h [n]: CUDA float32 tensors;
    alpha: 0-dim float64 tensor (alpha_AV); probes: CUDA int64 tensor.
    The library reads raw pointers, so every array must be a contiguous
    float32 CUDA tensor (velu is not copied: a copy would cut it off from
    autograd); anything else is rejected."""
    for name, t in (("pos", pos), ("velu", velu), ("h", h)):
        if t.dtype != torch.float32 or not t.is_cuda:
            raise TypeError(f"{name} must be a float32 CUDA tensor")
    if not velu.is_contiguous():
        raise ValueError("velu must be contiguous (pass velu.contiguous() as the leaf)")
    if pos.shape != velu.shape or pos.shape[-1] != 4 or h.shape != pos.shape[:1]:
        raise ValueError("pos and velu must be [n, 4] and h [n]")
    if probes.dtype != torch.int64 or not probes.is_cuda or not probes.is_contiguous():
        raise TypeError("probes must be a contiguous int64 CUDA tensor")
    return _Rollout.apply(velu, alpha, pos.contiguous(), h.contiguous(), handle, params,
                          n_steps, ckpt, probes)
