// Adjoint (reverse-mode) kernels of the density and force passes, for the
// differentiable rollout.  Not part of the paper's method; they differentiate
// Eqs. 1-4 and 9-15 as implemented by density.cu and force.cu.
//
// All backward passes are "pull" passes: a warp walks the tree for a group of
// targets, collects each target's neighbours (force set, or density set), and
// every target sums the cotangent contributions that land on ITS inputs, from
// its own equations and from its neighbours' equations.  No atomics, so the
// results are deterministic.
//
// Force backward: the two terms of a pair that depend on a target k's inputs,
// T_kj (the contribution of j to a_k and du_k/dt, Eqs. 9-15 as the force pass
// computes them) and T_jk, are differentiated together by one hand-written
// reverse sweep (force_pair_vjp): they share all their forward values.  FP32
// only (this GPU's FP64 rate is a small fraction of FP32's).
//
// Density backward (implicit-function theorem): h_i solves
// g_i = sum_j m_j W(r_ij, h_i) - M_i / h_i^3 = 0, M_i = m_i hfact^3, with
// dg_i/dh_i = 3 rho_i Omega_i / h_i and dg_i/dr_ij = m_j F(r_ij, h_i);
// rho_i = M_i / h_i^3 and Omega_i = 1 + h_i^4 S_i / (3 M_i),
// S_i = sum_j m_j dW/dh(r_ij, h_i).
//
// The pair operations are templates on the smoothing kernel K (SphKernel<K>:
// f, f', f'' and the support radius R).
#include <algorithm>

#include "kernels.cuh"
#include "walk.cuh"

namespace sph {

// ------------------------------------------------------- generic pair walk
struct PairWalkArgs {
    const float4 *pos;
    const float *h;
    const int2 *grp_ref;
    const float4 *grp_lo, *grp_hi;
    const int *sizes;
    int *work;
    WalkTree tree;
    const int *inst;
    int dens_set;  // 1: density set r < R h_i (self included); 0: force set r < R max(h_i, h_j)
    float kr;      // R, the kernel's support radius in units of h
    // neighbour lists of the last density pass (a superset of both pair sets
    // while they are fresh and no h of the instance outgrew the list pad)
    const int *nl_idx, *nl_len, *rec_ctl, *rec_bad;
    int nl_stride;
    int *err;
};

constexpr int kPW_TB = 8;

template <int CAP>
struct PairWalkSmem {
    WalkSmem w;
    float4 tp[kPW_TB];
    float th[kPW_TB];
    int tlen[kPW_TB];
    int ej[kPW_TB][CAP];
};

// Five blocks per SM: the gathers' latency is what binds, and a rollout of 8 steps of
// 64^3 with its adjoint took 39.0 -> 38.3 ms although the force operator spills
// some 60 bytes at that limit.
// Op: struct with  Acc;  init(i, Acc&);  pair(j, x_j and m_j, Acc&);  reduce(Acc&, L);  store(i, Acc&)
template <int CAP, class Op>
__global__ void __launch_bounds__(128, 5) pairwalk_kernel(PairWalkArgs a, Op op)
{
    pdl_sync();
    extern __shared__ __align__(16) unsigned char pw_raw[];
    PairWalkSmem<CAP> &sm = reinterpret_cast<PairWalkSmem<CAP> *>(pw_raw)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const unsigned lt = lane_lt();
    const int ng = a.sizes[SZ_GROUPS];
    while (true) {
        int g = 0;
        if (lane == 0) g = atomicAdd(a.work, 1);
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g >= ng) break;
        const int2 gr = a.grp_ref[g];
        const float4 glo = a.grp_lo[g], ghi = a.grp_hi[g];
        const int root = a.inst ? a.inst[gr.x] : 0;
        for (int b0 = 0; b0 < gr.y; b0 += kPW_TB) {
            const int nt = min(kPW_TB, gr.y - b0);
            const int L = nt > 4 ? 4 : nt > 2 ? 8 : nt > 1 ? 16 : 32;
            const int t = lane >> (__ffs(L) - 1), sub = lane & (L - 1);  // L a power of two
            const bool act = t < nt;
            const int i0 = gr.x + b0;
            const int i = i0 + (act ? t : 0);
            if (lane < nt) {
                sm.tp[lane] = a.pos[i0 + lane];
                sm.th[lane] = a.h[i0 + lane];
                sm.tlen[lane] = 0;
            }
            __syncwarp();
            typename Op::Acc acc;
            op.init(i, acc);
            float hmx = lane < nt ? sm.th[lane] : 0.f;
            for (int o = 16; o > 0; o >>= 1) hmx = fmaxf(hmx, __shfl_xor_sync(0xffffffffu, hmx, o));
            auto flush = [&]() {
                if (act) {
                    const int len = sm.tlen[t];
                    for (int e = sub; e < len; e += L) op.pair(sm.ej[t][e], __ldg(&a.pos[sm.ej[t][e]]), acc);
                }
                __syncwarp();
                if (lane < nt) sm.tlen[lane] = 0;
                __syncwarp();
            };
            auto chunk = [&](int j) {
                const float4 pj = j >= 0 ? __ldg(&a.pos[j]) : make_float4(0, 0, 0, 0);
                const float hj = j >= 0 ? __ldg(&a.h[j]) : 0.f;
                unsigned bs[kPW_TB];
                int base[kPW_TB];
                bool over = false;
#pragma unroll
                for (int tt = 0; tt < kPW_TB; ++tt) {
                    bs[tt] = 0u;
                    base[tt] = 0;
                    if (tt < nt) {
                        const float4 tp = sm.tp[tt];
                        const float r2 = canon_r2p(tp.x, tp.y, tp.z, pj.x, pj.y, pj.z, a.tree.per);
                        bool hit;
                        if (a.dens_set) {
                            const float R = a.kr * sm.th[tt];
                            hit = j >= 0 && r2 < R * R;
                        } else {
                            const float R = a.kr * fmaxf(sm.th[tt], hj);
                            hit = j >= 0 && j != i0 + tt && r2 < R * R;
                        }
                        bs[tt] = __ballot_sync(0xffffffffu, hit);
                        base[tt] = sm.tlen[tt];
                        over |= base[tt] + __popc(bs[tt]) > CAP;
                    }
                }
                if (over) {
                    flush();
#pragma unroll
                    for (int tt = 0; tt < kPW_TB; ++tt) base[tt] = 0;
                }
#pragma unroll
                for (int tt = 0; tt < kPW_TB; ++tt) {
                    if (tt < nt) {
                        if ((bs[tt] >> lane) & 1u) sm.ej[tt][base[tt] + __popc(bs[tt] & lt)] = j;
                        if (lane == tt) sm.tlen[tt] = base[tt] + __popc(bs[tt]);
                    }
                }
                __syncwarp();
            };
            const int len = act ? a.nl_len[i] : 0;
            const bool lists = a.rec_ctl[1] == 0 && a.rec_bad[root] == 0 &&
                               !__any_sync(0xffffffffu, len < 0);
            if (lists) {
                // the pair set from the target's list, with the same exact tests
                if (act) {
                    const int *__restrict__ lst = a.nl_idx + (size_t)i * a.nl_stride;
                    const float4 tp = sm.tp[t];
                    const float ht = sm.th[t];
                    int jn = sub < len ? __ldcs(lst + sub) : 0;  // an entry ahead
                    for (int e = sub; e < len; e += L) {
                        const int j = jn;
                        if (e + L < len) jn = __ldcs(lst + e + L);
                        const float4 pj = __ldg(&a.pos[j]);
                        const float r2 = canon_r2p(tp.x, tp.y, tp.z, pj.x, pj.y, pj.z, a.tree.per);
                        const float R = a.dens_set ? a.kr * ht : a.kr * fmaxf(ht, __ldg(&a.h[j]));
                        if (r2 < R * R && (a.dens_set || j != i)) op.pair(j, pj, acc);
                    }
                }
                __syncwarp();
            } else {
                const float hr = 0.5f * a.kr;
                bool ok = a.dens_set ? walk_group(a.tree, root, glo, ghi, a.kr * hmx, false, 0.f, sm.w, chunk)
                                     : walk_group(a.tree, root, glo, ghi, 0.f, true, hr * hmx, sm.w, chunk, hr);
                if (!ok && lane == 0) raise_error(a.err, SPH_ERR_TILE_OVERFLOW);
                flush();
            }
            op.reduce(acc, L);
            if (act && sub == 0) op.store(i, acc);
            __syncwarp();
        }
    }
}

// ------------------------------------------------------------ force backward
// P_i - P_j = (gamma - 1)(rho_i u_i - rho_j u_j) without FP64 (whose rate is
// a small fraction of FP32's on this GPU): each product's rounding error is
// recovered exactly with an FMA, and when the pressures are close the
// difference of the rounded products is exact (Sterbenz), so the difference
// keeps about twice FP32's precision.  The conduction speed's derivative
// carries 1 / sqrt(|P_i - P_j|), so the difference must not be swamped by
// the rounding of the two pressures.  (The products by intrinsics, which the
// compiler never contracts: a - b as one FMA would count ea twice, 1e-3 of dL/du.)
__device__ __forceinline__ float pressure_diff(float gm1, float ri, float ui, float rj, float uj)
{
    const float a = __fmul_rn(ri, ui), b = __fmul_rn(rj, uj);
    const float ea = fmaf(ri, ui, -a), eb = fmaf(rj, uj, -b);
    return gm1 * ((a - b) + (ea - eb));
}

// sqrt(x) for x >= 0 through the hardware reciprocal square root (0 at 0)
__device__ __forceinline__ float fast_sqrt(float x) { return x > 0.f ? x * rsqrtf(x) : 0.f; }

// A particle in a pair term: position and mass, velocity and u, (h, rho,
// A = 1 / (rho Omega), c), the cotangent w of (a xyz, du/dt).
struct PairIn {
    float4 x, v, q, w;
};

// What a target's pairs add up to: the cotangents of x, v, u, h, rho and of
// A and c (turned into those of rho, Omega and u once at the end), and twice
// that of alpha_AV.
struct PairGrad {
    float x[3], v[3], u, h, rho, A, c, al;
};

// Reverse-mode derivative, with respect to the inputs of the target k, of
//   S = w_k . T_kj + w_j . T_jk
//     = -coef (W . d) / r + e_k E_k + e_j E_j + (e_k - e_j) alpha_u / 2 vsu (u_k - u_j) AF,
// W = m_j w_k - m_k w_j (its acceleration part), e_k = m_j w_k.w, e_j = m_k w_j.w,
// d = x_k - x_j, coef = sum of A p F over both, E = A ((gamma - 1) u vr F - D),
// D = vsig vr^2 F / 2 for vr < 0, AF = sum of A F (the same operations as the
// force pass).  r = 0 gives no term, the viscous terms act for vr < 0 only, and
// sqrt has derivative 0 at 0 (at equal pressures the conduction term carries
// u_k - u_j times a zero speed).  Quotients and roots use the hardware
// approximations (a few ulp).  hk = 1 / h_k.  (One sweep over each of the two
// terms by itself forms every forward value twice: 64^3 lattice 575 -> 427 us.)
template <int K>
__device__ __forceinline__ void force_pair_vjp(const PairIn &I, const PairIn &J, float hk, float alpha,
                                               float beta, float alpha_u, float gm1, const Period &P,
                                               PairGrad &g)
{
    // nearest images on the periodic axes (the wrap's derivative is 1)
    const float dx = wrap_sep(I.x.x - J.x.x, P.x), dy = wrap_sep(I.x.y - J.x.y, P.y),
                dz = wrap_sep(I.x.z - J.x.z, P.z);
    const float r2 = dx * dx + dy * dy + dz * dz;
    if (!(r2 > 0.f)) return;
    const float rinv = rsqrtf(r2);
    const float r = r2 * rinv;
    // ---- forward values
    const float hj = __fdividef(1.f, J.q.x);
    const float qk = r * hk, qj = r * hj;
    const float h2k = hk * hk, h2j = hj * hj;
    const float Kk = SphKernel<K>::C * h2k * h2k, Kj = SphKernel<K>::C * h2j * h2j;  // C / h^4
    const float Fk = SphKernel<K>::df(qk) * Kk, Fj = SphKernel<K>::df(qj) * Kj;
    const float dvx = I.v.x - J.v.x, dvy = I.v.y - J.v.y, dvz = I.v.z - J.v.z;
    const float sd = dvx * dx + dvy * dy + dvz * dz;
    const float vr = sd * rinv, vr2 = vr * vr;
    const float avr = fabsf(vr);
    const bool visc = vr < 0.f;
    const float vsk = alpha * I.q.w + beta * avr, vsj = alpha * J.q.w + beta * avr;
    const float Ak = I.q.z, Aj = J.q.z;
    const float prk = gm1 * I.v.w, prj = gm1 * J.v.w;  // P / rho
    const float pk = prk + (visc ? -0.5f * (vsk * vr) : 0.f), pj = prj + (visc ? -0.5f * (vsj * vr) : 0.f);
    const float Dk = visc ? 0.5f * (vsk * vr2 * Fk) : 0.f;
    const float coef = Ak * pk * Fk + Aj * pj * Fj;
    const float PD = pressure_diff(gm1, I.q.y, I.v.w, J.q.y, J.v.w);
    const float Sinv = __fdividef(2.f, I.q.y + J.q.y);   // 1 / ((rho_k + rho_j) / 2)
    const float X = fabsf(PD) * Sinv;
    const float vsu = fast_sqrt(X);
    const float du = I.v.w - J.v.w;
    const float AF = Fk * Ak + Fj * Aj;
    // ---- reverse sweep
    const float mj = J.x.w, mk = I.x.w;
    const float Wx = mj * I.w.x - mk * J.w.x, Wy = mj * I.w.y - mk * J.w.y, Wz = mj * I.w.z - mk * J.w.z;
    const float ek = mj * I.w.w, ej = mk * J.w.w;
    const float Wd = Wx * dx + Wy * dy + Wz * dz;
    // -coef (W . d) rinv
    const float cr = -coef * rinv;
    float bdx = cr * Wx, bdy = cr * Wy, bdz = cr * Wz;
    float brinv = -coef * Wd;
    const float bcoef = -rinv * Wd;
    // conduction
    const float hau = 0.5f * alpha_u * (ek - ej);
    float bu = hau * vsu * AF + ek * gm1 * Ak * vr * Fk;
    const float bvsu = hau * du * AF, bAF = hau * vsu * du;
    // pressure work and viscous heating
    const float ekA = ek * Ak, ejA = ej * Aj;
    float bA = ek * (prk * vr * Fk - Dk) + bAF * Fk;
    float bvr = ekA * prk * Fk + ejA * prj * Fj;
    float bFk = ekA * prk * vr + bAF * Ak;
    float bFj = ejA * prj * vr + bAF * Aj;
    // vsu = sqrt(|PD| / Srho), Srho = (rho_k + rho_j) / 2
    const float bX = vsu > 0.f ? __fdividef(0.5f * bvsu, vsu) : 0.f;
    const float bAPD = bX * Sinv;
    const float bPD = PD < 0.f ? -bAPD : bAPD;
    g.rho += bPD * prk - 0.5f * bAPD * X;
    bu += bPD * gm1 * I.q.y;
    // coef = sum of A p F
    bA += bcoef * pk * Fk;
    bFk += bcoef * Ak * pk;
    bFj += bcoef * Aj * pj;
    const float bpk = bcoef * Ak * Fk, bpj = bcoef * Aj * Fj;
    bu += bpk * gm1;
    if (visc) {
        // p = (gamma - 1) u - vsig vr / 2, D = vsig vr^2 F / 2 with cotangents -ekA, -ejA
        const float hvr = -0.5f * vr, hv2 = 0.5f * vr2;
        const float bvsk = bpk * hvr - ekA * hv2 * Fk, bvsj = bpj * hvr - ejA * hv2 * Fj;
        bvr += -0.5f * (bpk * vsk + bpj * vsj) - vr * (ekA * vsk * Fk + ejA * vsj * Fj);
        bFk -= ekA * hv2 * vsk;
        bFj -= ejA * hv2 * vsj;
        g.al += bvsk * I.q.w + bvsj * J.q.w;
        g.c += bvsk * alpha;
        bvr -= (bvsk + bvsj) * beta;  // |vr| = -vr here
    }
    g.u += bu;
    g.A += bA;
    // vr = sd rinv
    const float bsd = bvr * rinv;
    brinv += bvr * sd;
    // F = C f'(q) / h^4, q = r / h
    const float bqk = bFk * Kk * SphKernel<K>::d2f(qk), bqj = bFj * Kj * SphKernel<K>::d2f(qj);
    g.h -= hk * (4.f * bFk * Fk + bqk * qk);
    // rinv = 1 / r, r = |d|
    const float br = (bqk * hk + bqj * hj - brinv * rinv * rinv) * rinv;
    g.x[0] += bdx + bsd * dvx + br * dx;
    g.x[1] += bdy + bsd * dvy + br * dy;
    g.x[2] += bdz + bsd * dvz + br * dz;
    g.v[0] += bsd * dx;
    g.v[1] += bsd * dy;
    g.v[2] += bsd * dz;
}

// (h, rho, 1 / (rho Omega), c) of every particle, as the force pass has it
__global__ void bwd_prep_kernel(const float4 *__restrict__ vel, const float *__restrict__ h,
                                const float *__restrict__ rho, const float *__restrict__ omega, int n,
                                float gamma, float4 *__restrict__ prop)
{
    pdl_sync();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float c2 = gamma * (gamma - 1.f) * vel[i].w;
        prop[i] = make_float4(h[i], rho[i], 1.f / (rho[i] * omega[i]), sqrtf(fmaxf(c2, 0.f)));
    }
}

template <int KER>
struct ForceBwdOp {
    const float4 *pos, *vel, *prop, *gacc;  // gacc: (dL/da xyz, dL/d(du/dt))
    const float *omega;
    float4 *gpos, *gvel;             // out: dL/dx (xyz, 0), dL/dv (xyz), dL/du (w)
    float *gh, *grho, *gom;          // out
    double *galpha;                  // out: accumulated (one atomic per target)
    float alpha, beta, alpha_u, gamma;
    Period per;
    struct Acc {
        PairIn K;     // the target's own inputs, loaded once
        float hk;
        PairGrad g;
    };
    __device__ void init(int k, Acc &c) const
    {
        c.K = PairIn{pos[k], vel[k], prop[k], gacc[k]};
        c.hk = 1.f / c.K.q.x;
        c.g = PairGrad{{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    }
    // the terms that land on k's inputs: from k's own equations (T_kj with
    // cotangent gacc[k]) and from j's (T_jk with cotangent gacc[j])
    __device__ void pair(int j, float4 pj, Acc &c) const
    {
        const PairIn J{pj, __ldg(&vel[j]), __ldg(&prop[j]), __ldg(&gacc[j])};
        force_pair_vjp<KER>(c.K, J, c.hk, alpha, beta, alpha_u, gamma - 1.f, per, c.g);
    }
    __device__ void reduce(Acc &c, int L) const
    {
        for (int o = L >> 1; o > 0; o >>= 1) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                c.g.x[a] += __shfl_xor_sync(0xffffffffu, c.g.x[a], o);
                c.g.v[a] += __shfl_xor_sync(0xffffffffu, c.g.v[a], o);
            }
            c.g.u += __shfl_xor_sync(0xffffffffu, c.g.u, o);
            c.g.h += __shfl_xor_sync(0xffffffffu, c.g.h, o);
            c.g.rho += __shfl_xor_sync(0xffffffffu, c.g.rho, o);
            c.g.A += __shfl_xor_sync(0xffffffffu, c.g.A, o);
            c.g.c += __shfl_xor_sync(0xffffffffu, c.g.c, o);
            c.g.al += __shfl_xor_sync(0xffffffffu, c.g.al, o);
        }
    }
    __device__ void store(int k, Acc &c) const
    {
        // A = 1 / (rho Omega), c = sqrt(gamma (gamma - 1) u)
        const float bA = c.g.A * c.K.q.z, cs = c.K.q.w;
        const float bu = cs > 0.f ? c.g.c * gamma * (gamma - 1.f) * 0.5f / cs : 0.f;
        gpos[k] = make_float4(c.g.x[0], c.g.x[1], c.g.x[2], 0.f);
        gvel[k] = make_float4(c.g.v[0], c.g.v[1], c.g.v[2], c.g.u + bu);
        gh[k] = c.g.h;
        grho[k] = c.g.rho - bA / c.K.q.y;
        gom[k] = -bA / omega[k];
        // T_kj counts here and in the sum of j
        atomicAdd(galpha, 0.5 * (double)c.g.al);
    }
};

// --------------------------------------------------------- density backward
// kernel pieces f, f', f'' at q (all 0 beyond the support)
template <int K>
__device__ __forceinline__ void kernel_all(float q, float &f, float &df, float &d2f)
{
    SphKernel<K>::f_df(q, f, df);
    d2f = SphKernel<K>::d2f(q);
}

// pass 1: per target, S = sum m dW/dh and S2 = sum m d2W/dh2 over the density
// set; then lambda (the IFT multiplier) and omega-coefficient per particle.
template <int K>
struct DensBwd1Op {
    const float4 *pos;
    const float *h, *rho, *omega;
    const float *gh, *grho, *gom;  // cotangents of h, rho, Omega
    float4 *coef;                  // out: (lambda, w, 1 / h, -)
    float hf3;
    Period per;
    struct Acc { float4 x; float hinv, S, S2; };
    __device__ void init(int i, Acc &c) const
    {
        c.x = pos[i];
        c.hinv = __fdividef(1.f, h[i]);
        c.S = c.S2 = 0.f;
    }
    // sums without their factors C / h^4 and C / h^5
    __device__ void pair(int, float4 pj, Acc &c) const
    {
        const float dx = wrap_sep(c.x.x - pj.x, per.x), dy = wrap_sep(c.x.y - pj.y, per.y),
                    dz = wrap_sep(c.x.z - pj.z, per.z);
        const float q = fast_sqrt(dx * dx + dy * dy + dz * dz) * c.hinv;
        float f, df, d2f;
        kernel_all<K>(q, f, df, d2f);
        c.S -= pj.w * (3.f * f + q * df);
        c.S2 += pj.w * (12.f * f + 8.f * q * df + q * q * d2f);
    }
    __device__ void reduce(Acc &c, int L) const
    {
        for (int o = L >> 1; o > 0; o >>= 1) {
            c.S += __shfl_xor_sync(0xffffffffu, c.S, o);
            c.S2 += __shfl_xor_sync(0xffffffffu, c.S2, o);
        }
    }
    __device__ void store(int i, Acc &c) const
    {
        const float hi = h[i], M = c.x.w * hf3, hinv = 1.f / hi;
        const float h4 = hi * hi * hi * hi;
        // h^3 S and h^4 S2 of the full sums are C / h times these
        const float domdh = SphKernel<K>::C * hinv * (4.f * c.S + c.S2) / (3.f * M);
        const float htot = gh[i] - 3.f * rho[i] / hi * grho[i] + gom[i] * domdh;
        const float lambda = htot * hi / (3.f * rho[i] * omega[i]);
        coef[i] = make_float4(lambda, gom[i] * h4 / (3.f * M), hinv, 0.f);
    }
};

// pass 2 (force set): gx_k += sum_j (c_kj + c_jk) rhat_kj,
// c_ij = -lambda_i m_j F(r, h_i) + w_i m_j d2W/dh dr(r, h_i)
template <int K>
struct DensBwd2Op {
    const float4 *pos, *coef;
    float4 *gpos;  // accumulated (+=)
    Period per;
    struct Acc { float4 x, q; float g[3]; };
    __device__ void init(int k, Acc &c) const
    {
        c.x = pos[k];
        c.q = coef[k];
        c.g[0] = c.g[1] = c.g[2] = 0.f;
    }
    __device__ static float cterm(float r, float4 q, float m)  // q = (lambda, w, 1 / h)
    {
        const float x = r * q.z, h2 = q.z * q.z;
        const float df = SphKernel<K>::df(x), d2f = SphKernel<K>::d2f(x);
        return -m * SphKernel<K>::C * h2 * h2 * (q.x * df + q.y * q.z * (4.f * df + x * d2f));
    }
    __device__ void pair(int j, float4 pj, Acc &c) const
    {
        const float dx = wrap_sep(c.x.x - pj.x, per.x), dy = wrap_sep(c.x.y - pj.y, per.y),
                    dz = wrap_sep(c.x.z - pj.z, per.z);
        const float r2 = dx * dx + dy * dy + dz * dz;
        if (!(r2 > 0.f)) return;
        const float rinv = rsqrtf(r2), r = r2 * rinv;
        const float s = (cterm(r, c.q, pj.w) + cterm(r, __ldg(&coef[j]), c.x.w)) * rinv;
        c.g[0] += s * dx;
        c.g[1] += s * dy;
        c.g[2] += s * dz;
    }
    __device__ void reduce(Acc &c, int L) const
    {
        for (int o = L >> 1; o > 0; o >>= 1)
#pragma unroll
            for (int a = 0; a < 3; ++a) c.g[a] += __shfl_xor_sync(0xffffffffu, c.g[a], o);
    }
    __device__ void store(int k, Acc &c) const
    {
        float4 g = gpos[k];
        gpos[k] = make_float4(g.x + c.g[0], g.y + c.g[1], g.z + c.g[2], g.w);
    }
};

// ------------------------------------------------------------------ launch
template <int CAP, class Op>
static cudaError_t launch_pairwalk(Ctx &c, const sph_state &s, bool dens_set, float kr, Period per,
                                   const Op &op, cudaStream_t st, const Batch *batch)
{
    size_t smem = sizeof(PairWalkSmem<CAP>) * 4;
    static std::mutex mu;  // first calls may come from several host threads
    std::lock_guard<std::mutex> lock(mu);
    static bool configured = false;
    static int blocks = 1;
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(pairwalk_kernel<CAP, Op>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        int nb = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pairwalk_kernel<CAP, Op>, 128, smem);
        if (e != cudaSuccess) return e;
        blocks = nb > 0 ? nb : 1;
        configured = true;
    }
    PairWalkArgs a{};
    a.pos = (const float4 *)s.pos;
    a.h = s.h;
    a.grp_ref = c.tree.grp_ref;
    a.grp_lo = c.tree.grp_lo;
    a.grp_hi = c.tree.grp_hi;
    a.sizes = c.d_sizes;
    a.work = c.d_sizes + SZ_WORK;
    a.tree = WalkTree{c.tree.node_lo, c.tree.node_hi, c.tree.node_ref, per};
    a.inst = batch ? c.inst : nullptr;
    a.dens_set = dens_set ? 1 : 0;
    a.kr = kr;
    a.nl_idx = c.nl_idx;
    a.nl_len = c.nl_len;
    a.nl_stride = c.nl_stride;
    a.rec_ctl = c.tree.rec_ctl;
    a.rec_bad = c.tree.rec_bad;
    a.err = c.d_err;
    cudaError_t e = clear_words(Clear{{a.work}, {1}}, st);
    if (e != cudaSuccess) return e;
    launch(pairwalk_kernel<CAP, Op>, c.num_sms * blocks, 128, smem, st, a, op);
    return cudaGetLastError();
}

template <int K>
static cudaError_t force_bwd_k(Ctx &c, const sph_state &s, const sph_params &p, const float4 *gacc,
                               float4 *gpos, float4 *gvel, float *gh, float *grho, float *gom,
                               double *galpha, cudaStream_t st)
{
    ForceBwdOp<K> op;
    op.pos = (const float4 *)s.pos;
    op.vel = (const float4 *)s.vel;
    op.prop = c.prop;
    op.gacc = gacc;
    op.omega = s.omega;
    op.gpos = gpos;
    op.gvel = gvel;
    op.gh = gh;
    op.grho = grho;
    op.gom = gom;
    op.galpha = galpha;
    op.alpha = p.alpha_av;
    op.beta = p.beta_av;
    op.alpha_u = p.alpha_u;
    op.gamma = p.gamma;
    op.per = period_of(p);
    // the force-set walk needs node and group h_max of the current h
    cudaError_t e = check_list_kernel(c, p, st);
    if (e == cudaSuccess) e = update_hmax(c, s, p, st);
    if (e != cudaSuccess) return e;
    const int n = (int)s.n, grid = std::min(div_up(n, 256), c.num_sms * 16);
    launch(bwd_prep_kernel, grid, 256, 0, st, op.vel, s.h, s.rho, s.omega, n, p.gamma, c.prop);
    return launch_pairwalk<96>(c, s, false, SphKernel<K>::R, op.per, op, st, nullptr);
}

cudaError_t force_bwd(Ctx &c, const sph_state &s, const sph_params &p, const float4 *gacc,
                      float4 *gpos, float4 *gvel, float *gh, float *grho, float *gom,
                      double *galpha, cudaStream_t st)
{
    if (p.kernel == 1) return force_bwd_k<1>(c, s, p, gacc, gpos, gvel, gh, grho, gom, galpha, st);
    if (p.kernel == 2) return force_bwd_k<2>(c, s, p, gacc, gpos, gvel, gh, grho, gom, galpha, st);
    return force_bwd_k<0>(c, s, p, gacc, gpos, gvel, gh, grho, gom, galpha, st);
}

template <int K>
static cudaError_t density_bwd_k(Ctx &c, const sph_state &s, const sph_params &p, const float *gh,
                                 const float *grho, const float *gom, float4 *gpos, float4 *coef,
                                 cudaStream_t st, bool refresh_hmax)
{
    DensBwd1Op<K> op1;
    op1.pos = (const float4 *)s.pos;
    op1.h = s.h;
    op1.rho = s.rho;
    op1.omega = s.omega;
    op1.gh = gh;
    op1.grho = grho;
    op1.gom = gom;
    op1.coef = coef;
    op1.hf3 = p.hfact * p.hfact * p.hfact;
    op1.per = period_of(p);
    // pass 2 opens nodes by their h_max (force set) where it walks: refresh it
    // for the current h (unless the caller just did)
    cudaError_t e = check_list_kernel(c, p, st);
    if (e == cudaSuccess && refresh_hmax) e = update_hmax(c, s, p, st);
    if (e != cudaSuccess) return e;
    e = launch_pairwalk<96>(c, s, true, SphKernel<K>::R, op1.per, op1, st, nullptr);
    if (e != cudaSuccess) return e;
    DensBwd2Op<K> op2;
    op2.pos = (const float4 *)s.pos;
    op2.coef = coef;
    op2.gpos = gpos;
    op2.per = op1.per;
    return launch_pairwalk<96>(c, s, false, SphKernel<K>::R, op2.per, op2, st, nullptr);
}

cudaError_t density_bwd(Ctx &c, const sph_state &s, const sph_params &p, const float *gh,
                        const float *grho, const float *gom, float4 *gpos, float4 *coef,
                        cudaStream_t st, bool refresh_hmax)
{
    if (p.kernel == 1) return density_bwd_k<1>(c, s, p, gh, grho, gom, gpos, coef, st, refresh_hmax);
    if (p.kernel == 2) return density_bwd_k<2>(c, s, p, gh, grho, gom, gpos, coef, st, refresh_hmax);
    return density_bwd_k<0>(c, s, p, gh, grho, gom, gpos, coef, st, refresh_hmax);
}

}  // namespace sph
