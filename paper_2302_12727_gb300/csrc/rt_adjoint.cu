// Reverse-mode derivative of n sub-cycles of the transport step (no counterpart in the
// thesis).  Given lambda = dL/dU(final) it returns dL/dU0 and dL/dL_src.
//
// One forward step is  U_inj = U + inj(L);  g = grad(U_inj);  Phi_kl = flux(U_inj, g);
// U~_i = U_inj,i - dt omega_i (sum_{k=i} Phi - sum_{l=i} Phi);  U'_i = U~_i sink_i.
// Its adjoint, for lambda' = dL/dU':
//   lambda~_i = lambda'_i sink_i,  mu_i = -dt omega_i lambda~_i,  Phibar_kl = mu_k - mu_l;
//   through the GLF flux (Eq. riemann-GLF), the M1 closure (Eq. eddington-group) and the
//   limited face states (Eq. rt-riemann-problem, Eq. rt-minmod: the derivative follows the
//   selected slope) to Ubar (direct) and gbar (through the gradients);
//   through the least-squares gradient (Eq. gradient), whose transpose is
//   Ubar_i -= sum_j d_ij . (gamma_i w(r_ij/H_i) + gamma_j w(r_ij/H_j)), gamma = omega Bp gbar;
//   the injection is additive, so lambda passes through and dL/dL_s,g += dt sum_e coef_e lambda_E.
// The fix-up E <- max(E, 0) is treated as inactive.
//
// The forward pass keeps the state every ckpt_every steps; the reverse pass recomputes each
// segment with the forward kernels (bitwise the same states) and walks it backwards.  Each
// pair's terms are evaluated once, in its canonical orientation (k < l), into slots that its
// two particles then sum, so the reductions are per particle, fixed-order and atomic-free.
#include "rt_pair.cuh"

namespace rt {

static inline unsigned nblk_(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// J(U)^T pb for the M1 flux contracted with A (m1_terms): U = (E, F), pb = dL/d(flux).  With
// e = cE, f = F/e, u = f.f, s = sqrt(4 - 3u) and g = 3/(2 + s) the flux rows are
// Pi = c e (a A + g (f.A) f), a = (s - 1)/3, and a' = -1/(2s), g' = g^2/(2s), so
//   d(p.Pi)/de = c [(a + u/s) p.A - (g + u g^2/s) (f.A)(p.f)]
//   d(p.Pi)/dF = c [(g^2 (f.A)(p.f) - p.A)/s f + g ((p.f) A + (f.A) p)];
// where |f| > 1 is clipped, Pi = c e (f.A) f / u.  f keeps every term scale-free; a clipped state
// with u beyond the range (E far below |F|, as at a front) takes F itself for f: Pi does not
// change, and d(p.Pi)/dF is e times what f gives.
template <class T>
__device__ __forceinline__ void m1_vjp(const T u4[4], T Ax, T Ay, T Az, T c, const T pb[4], T ub[4]) {
    ub[0] = T(0);
    ub[1] = pb[0] * Ax;
    ub[2] = pb[0] * Ay;
    ub[3] = pb[0] * Az;
    const T e = c * u4[0];
    if (!(e > tiny_<T>())) return;
    const T ie = rcp_fast(e);
    T fx = u4[1] * ie, fy = u4[2] * ie, fz = u4[3] * ie;
    T fA = fx * Ax + fy * Ay + fz * Az;
    const T pA = pb[1] * Ax + pb[2] * Ay + pb[3] * Az;
    T pf = pb[1] * fx + pb[2] * fy + pb[3] * fz;
    T u = fx * fx + fy * fy + fz * fz;
    T ce, cf, cg;   // d/de, and the coefficients of f and of (p.f) A + (f.A) p
    if (u > T(1)) {
        const bool far = !(u <= T(1) / tiny_<T>());     // 1/u below the normal numbers, or u infinite
        if (far) {
            fx = u4[1];
            fy = u4[2];
            fz = u4[3];
            fA = fx * Ax + fy * Ay + fz * Az;
            pf = pb[1] * fx + pb[2] * fy + pb[3] * fz;
            u = fx * fx + fy * fy + fz * fz;
        }
        cg = rcp_fast(u);
        ce = cg * fA * pf;
        if (far) cg *= e;
        cf = T(-2) * cg * ce;
    } else {
        T is;
        const T s = sqrt_fast(fma_rn(T(-3), u, T(4)), is);
        cg = T(3) * rcp_fast(T(2) + s);
        const T h = cg * fA * pf;             // g (f.A)(p.f)
        const T k = cg * h - pA;
        ce = (s - T(1)) * T(1.0 / 3.0) * pA - h - u * is * k;
        cf = is * k;
    }
    cg *= c;
    cf *= c;
    ub[0] = c * (c * ce);
    ub[1] += cf * fx + cg * (pf * Ax + fA * pb[1]);
    ub[2] += cf * fy + cg * (pf * Ay + fA * pb[2]);
    ub[3] += cf * fz + cg * (pf * Az + fA * pb[3]);
}

// which particle's slope the limiter chose: 1 for k, 2 for l, 0 for none (opposite signs or a
// zero slope); equal slopes count as l's, as in minmod_
template <class T>
__device__ __forceinline__ int slope_of(T dqk, T dql, T s) {
    return s == T(0) ? 0 : (fabs(dqk) < fabs(dql) ? 1 : 2);
}

// sink factor of particle p over one step
template <class T>
__device__ __forceinline__ T grey_sink(const FluxExtra<T>& x, int64_t p, T dt) {
    return x.alpha ? fmax_(T(1) - x.c * x.alpha[p] * dt, T(0)) : T(1);
}

// mu_i = -dt omega_i sink_i lambda_i for every component: the derivative of the loss with
// respect to the flux sum of particle i
template <class T>
__global__ void __launch_bounds__(256) k_adj_mu(PairArgs<T> a, FluxExtra<T> x, const T* __restrict__ lam,
                                                T* __restrict__ mu) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = t / a.G;
    if (i >= a.n) return;
    const T dt = (T)(*x.dt_dev);
    const T f = -dt * a.omega[i], sk = grey_sink(x, i, dt);
    T l[4];
    vload<4>(lam + 4 * t, l);
#pragma unroll
    for (int q = 0; q < 4; ++q) l[q] = f * (l[q] * sk);
    vstore<4>(mu + 4 * t, l);
}

// Adjoint of the flux of each unordered pair, once, by one thread, for the groups [g0, g0 + GC):
// the slot gets dL/dQ_k through the left state, dL/dQ_l through the right state and dL/ds of
// the slope (12 values a group), sel the particle whose slope each component took (2 bits
// each).  Evaluating the pair for each of its particles, as a kernel over rows does, costs
// twice the double instructions that bound it: 4.26 ms a step in double on 32,768 particles and
// two groups, against 0.53 ms for this pass and its gather.
template <class T, int GC>
__global__ void __launch_bounds__(128) k_adj_pair(PairArgs<T> a, T c, const T* __restrict__ mu,
                                                  const T* __restrict__ W, T* __restrict__ slots,
                                                  uint8_t* __restrict__ sel, int g0) {
    const int64_t slot = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (slot >= a.n_pairs) return;
    const int G = a.G, RS = 4 * G;
    const int2 kl = a.ends[slot];
    const int64_t i = kl.x, j = kl.y;
    PairGeo<T> p;
    T sk, sl;
    load_pair_geo(a, slot, i, j, c, p, sk, sl);
    const T wl = T(1) - p.wk;
#pragma unroll
    for (int g = 0; g < GC; ++g) {
        const int gg = g0 + g;
        T uk[4], ul[4], gk[12], gl[12], mk[4], ml[4], L[4], R[4];
        vload<4>(W + i * RS + 4 * gg, uk);
        vload<4>(W + j * RS + 4 * gg, ul);
        vload<12>(a.grad + i * 12 * G + 12 * gg, gk);
        vload<12>(a.grad + j * 12 * G + 12 * gg, gl);
        vload<4>(mu + i * RS + 4 * gg, mk);
        vload<4>(mu + j * RS + 4 * gg, ml);
        unsigned code = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const T dqk = gk[3 * q] * p.dx + gk[3 * q + 1] * p.dy + gk[3 * q + 2] * p.dz;
            const T dql = gl[3 * q] * p.dx + gl[3 * q + 1] * p.dy + gl[3 * q + 2] * p.dz;
            const T s = minmod_(dqk, dql);
            code |= (unsigned)slope_of(dqk, dql, s) << (2 * q);
            L[q] = fma_rn(p.wk, s, uk[q]);
            R[q] = fma_rn(-wl, s, ul[q]);
            mk[q] -= ml[q];
        }
        // half the surface: the central flux is the mean of the two states' fluxes
        T jL[4], jR[4], sb[4];
        m1_vjp(L, p.hx, p.hy, p.hz, c, mk, jL);
        m1_vjp(R, p.hx, p.hy, p.hz, c, mk, jR);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            jL[q] += p.diss * mk[q];
            jR[q] -= p.diss * mk[q];
            sb[q] = p.wk * jL[q] - wl * jR[q];
        }
        T* o = slots + (slot * GC + g) * 12;
        vstore<4>(o, jL);
        vstore<4>(o + 4, jR);
        vstore<4>(o + 8, sb);
        sel[slot * GC + g] = (uint8_t)code;
    }
}

// d = x_l - x_k of a slot: kept, or from the two positions
template <class T>
__device__ __forceinline__ void pair_sep(const PairArgs<T>& a, int64_t slot, int64_t k, int64_t l, T& dx, T& dy, T& dz) {
    if constexpr (std::is_same<T, double>::value) {
        if (a.pg) {
            const double* p = reinterpret_cast<const double*>(a.pg + slot);
            const double2 v = *reinterpret_cast<const double2*>(p);
            dx = v.x;
            dy = v.y;
            dz = p[2];
            return;
        }
    }
    const T* tag = nullptr;
    sep(a.sp, load_pos(tag, a.pos, k), load_pos(tag, a.pos, l), dx, dy, dz);
}

// Particle i's share of its slots, one thread per (particle, group): Ubar through its own
// states, gbar = sum of dL/ds d over the slots whose slope it gave, gamma = omega Bp gbar
template <class T, int GC>
__global__ void __launch_bounds__(128) k_adj_gather(PairArgs<T> a, FluxExtra<T> x, const T* __restrict__ lam,
                                                    const T* __restrict__ slots, const uint8_t* __restrict__ sel,
                                                    T* __restrict__ ubar, T* __restrict__ gam, int g0) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = t / GC;
    if (i >= a.n) return;
    const int g = (int)(t - i * GC), gg = g0 + g;
    const int G = a.G, RS = 4 * G;
    T ub[4], gb[4][3];
    vload<4>(lam + i * RS + 4 * gg, ub);
    const T sk = grey_sink(x, i, (T)(*x.dt_dev));
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        ub[q] *= sk;
        gb[q][0] = gb[q][1] = gb[q][2] = T(0);
    }
    auto add = [&](int64_t slot, int64_t k, int64_t l, int side) {
        T v[4], sb[4], dx, dy, dz;
        const T* o = slots + (slot * GC + g) * 12;
        vload<4>(o + 4 * (side - 1), v);
        vload<4>(o + 8, sb);
        const unsigned code = sel[slot * GC + g];
        pair_sep(a, slot, k, l, dx, dy, dz);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            ub[q] += v[q];
            const T b = ((code >> (2 * q)) & 3u) == (unsigned)side ? sb[q] : T(0);
            gb[q][0] += b * dx;
            gb[q][1] += b * dy;
            gb[q][2] += b * dz;
        }
    };
    const int64_t r0 = a.row_off[i], s0 = a.up_off[i], s1 = a.up_off[i + 1];
    const int nl = a.n_low[i];
    const int32_t* ls = a.low_slot + (r0 - s0);
#pragma unroll 2
    for (int e = 0; e < nl; ++e) add(ls[e], a.cols[r0 + e], i, 2);
#pragma unroll 2
    for (int64_t s = s0; s < s1; ++s) add(s, i, a.cols[r0 + nl + (s - s0)], 1);
    vstore<4>(ubar + i * RS + 4 * gg, ub);
    // gamma_i = omega_i Bp_i gbar_i (the gradient is omega_i Bp_i sum_j (Q_j - Q_i) w d, Bp symmetric)
    T Mi[6], out[12];
    const T om = a.omega[i];
#pragma unroll
    for (int k = 0; k < 6; ++k) Mi[k] = om * a.geo[8 * i + 2 + k];
#pragma unroll
    for (int q = 0; q < 4; ++q) sym_mv(Mi, gb[q][0], gb[q][1], gb[q][2], out[3 * q], out[3 * q + 1], out[3 * q + 2]);
    vstore<12>(gam + i * 12 * G + 12 * gg, out);
}

// Transpose of the gradient operator by pairs: v = d . (gamma_k w(r/H_k) + gamma_l w(r/H_l)) is
// what lambda_k loses and lambda_l gains; the gather below sums the slots in row order
template <class T, int GC>
__global__ void __launch_bounds__(128) k_adj_grad_pair(PairArgs<T> a, T c, const T* __restrict__ gam,
                                                       T* __restrict__ pairbuf, int g0) {
    const int64_t slot = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (slot >= a.n_pairs) return;
    const int G = a.G;
    const int2 kl = a.ends[slot];
    PairGeo<T> p;
    T sk, sl;
    load_pair_geo(a, slot, kl.x, kl.y, c, p, sk, sl);
    const T kx = sk * p.dx, ky = sk * p.dy, kz = sk * p.dz, lx = sl * p.dx, ly = sl * p.dy, lz = sl * p.dz;
#pragma unroll
    for (int g = 0; g < GC; ++g) {
        T gk[12], gl[12], v[4];
        vload<12>(gam + (int64_t)kl.x * 12 * G + 12 * (g0 + g), gk);
        vload<12>(gam + (int64_t)kl.y * 12 * G + 12 * (g0 + g), gl);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] = gk[3 * q] * kx + gk[3 * q + 1] * ky + gk[3 * q + 2] * kz + gl[3 * q] * lx + gl[3 * q + 1] * ly +
                   gl[3 * q + 2] * lz;
        vstore<4>(pairbuf + (slot * GC + g) * 4, v);
    }
}

template <class T, int GC>
__global__ void __launch_bounds__(128) k_adj_grad_gather(PairArgs<T> a, const T* __restrict__ ubar,
                                                         const T* __restrict__ pairbuf, T* __restrict__ lam_out,
                                                         int g0) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = t / GC;
    if (i >= a.n) return;
    const int g = (int)(t - i * GC);
    const int64_t o = i * 4 * a.G + 4 * (g0 + g);
    T acc[4], v[4];
    vload<4>(ubar + o, acc);
    const T* pb = pairbuf + 4 * g;
    const int64_t s0 = a.up_off[i], s1 = a.up_off[i + 1];
    const int nl = a.n_low[i];
    const int32_t* ls = a.low_slot + (a.row_off[i] - s0);
#pragma unroll 4
    for (int e = 0; e < nl; ++e) {
        vload<4>(pb + (int64_t)ls[e] * 4 * GC, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] += v[q];
    }
#pragma unroll 4
    for (int64_t s = s0; s < s1; ++s) {
        vload<4>(pb + s * 4 * GC, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] -= v[q];
    }
    vstore<4>(lam_out + o, acc);
}

// The same two stages without per-pair slots, for sets whose slots device memory does not hold
// (run_adjoint): one thread per (particle i, group) over i's whole row, every pair evaluated by
// both of its particles.
template <class T, int GC>
__global__ void __launch_bounds__(128) k_adj_flux(PairArgs<T> a, FluxExtra<T> x, const T* __restrict__ lam,
                                                  const T* __restrict__ W, T* __restrict__ ubar, T* __restrict__ gam,
                                                  int g0) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = t / GC;
    if (i >= a.n) return;
    const int gg = g0 + (int)(t - i * GC);
    const T* tag = nullptr;
    const int G = a.G, RS = 4 * G;
    const T dt = (T)(*x.dt_dev);
    const T sink_i = grey_sink(x, i, dt), om_i = a.omega[i];
    T li[4], mui[4], ub[4], gb[4][3];
    vload<4>(lam + i * RS + 4 * gg, li);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        li[q] *= sink_i;
        mui[q] = -dt * om_i * li[q];   // same expression as for the other particle below
        ub[q] = li[q];
        gb[q][0] = gb[q][1] = gb[q][2] = T(0);
    }
    const Pos<T> pi = load_pos(tag, a.pos, i);
    T gi8[8], ui[4], gri[12];
    vload<8>(a.geo + 8 * i, gi8);
    vload<4>(W + i * RS + 4 * gg, ui);
    vload<12>(a.grad + i * 12 * G + 12 * gg, gri);
    for (int64_t e = a.row_off[i]; e < a.row_off[i + 1]; ++e) {
        const int64_t j = a.cols[e];
        const bool ik = i < j;                     // i is the left state k
        const Pos<T> pj = load_pos(tag, a.pos, j);
        T gj8[8];
        vload<8>(a.geo + 8 * j, gj8);
        const T* gk8 = ik ? gi8 : gj8;
        const T* gl8 = ik ? gj8 : gi8;
        T dx, dy, dz;
        if (ik) sep(a.sp, pi, pj, dx, dy, dz);
        else sep(a.sp, pj, pi, dx, dy, dz);       // d = x_l - x_k
        PairGeo<T> p;
        T sk, sl;
        pair_geo(dx, dy, dz, gk8, gl8, x.c, p, sk, sl);
        const T wk = p.wk, wl = T(1) - p.wk;
        // mu of the other particle
        const T sink_j = grey_sink(x, j, dt), om_j = a.omega[j];
        T lj[4], uj[4], grj[12];
        vload<4>(lam + j * RS + 4 * gg, lj);
        vload<4>(W + j * RS + 4 * gg, uj);
        vload<12>(a.grad + j * 12 * G + 12 * gg, grj);
        const T* uk = ik ? ui : uj;
        const T* ul = ik ? uj : ui;
        const T* gk = ik ? gri : grj;
        const T* gl = ik ? grj : gri;
        T L[4], R[4], s[4];
        int sel[4];                          // 1: slope of k, 2: slope of l, 0: none
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            T dqk = gk[3 * q] * dx + gk[3 * q + 1] * dy + gk[3 * q + 2] * dz;
            T dql = gl[3 * q] * dx + gl[3 * q + 1] * dy + gl[3 * q + 2] * dz;
            s[q] = minmod_(dqk, dql);
            sel[q] = slope_of(dqk, dql, s[q]);
            L[q] = fma_rn(wk, s[q], uk[q]);
            R[q] = fma_rn(-wl, s[q], ul[q]);
        }
        T pb[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const T muj = -dt * om_j * (lj[q] * sink_j);
            const T muk = ik ? mui[q] : muj;
            const T mul = ik ? muj : mui[q];
            pb[q] = muk - mul;
        }
        T jL[4], jR[4];
        m1_vjp(L, p.hx, p.hy, p.hz, x.c, pb, jL);   // half the surface: the mean of the fluxes
        m1_vjp(R, p.hx, p.hy, p.hz, x.c, pb, jR);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const T Lb = jL[q] + p.diss * pb[q];
            const T Rb = jR[q] - p.diss * pb[q];
            const T sb = wk * Lb - wl * Rb;
            ub[q] += ik ? Lb : Rb;
            const bool mine = ik ? (sel[q] == 1) : (sel[q] == 2);
            if (mine) {
                gb[q][0] += sb * dx;
                gb[q][1] += sb * dy;
                gb[q][2] += sb * dz;
            }
        }
    }
    vstore<4>(ubar + i * RS + 4 * gg, ub);
    // gamma_i = omega_i Bp_i gbar_i (the gradient is omega_i Bp_i sum_j (Q_j - Q_i) w d, Bp symmetric)
    T Mi[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) Mi[k] = om_i * gi8[2 + k];
    T out[12];
#pragma unroll
    for (int q = 0; q < 4; ++q) sym_mv(Mi, gb[q][0], gb[q][1], gb[q][2], out[3 * q], out[3 * q + 1], out[3 * q + 2]);
    vstore<12>(gam + i * 12 * G + 12 * gg, out);
}

// transpose of the gradient operator: lambda_i = ubar_i - sum_j d_ij . (gamma_i w_i + gamma_j w_j),
// one thread per (particle i, group g0 + g of a chunk of GC)
template <class T, int GC>
__global__ void __launch_bounds__(128) k_adj_grad(PairArgs<T> a, const T* __restrict__ ubar,
                                                  const T* __restrict__ gam, T* __restrict__ lam_out, int g0) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = t / GC;
    if (i >= a.n) return;
    const int gg = g0 + (int)(t - i * GC);
    const T* tag = nullptr;
    const int G = a.G, RS = 4 * G;
    const Pos<T> pi = load_pos(tag, a.pos, i);
    const T iHi = a.geo[8 * i];
    T gi[12], acc[4];
    vload<12>(gam + i * 12 * G + 12 * gg, gi);
    vload<4>(ubar + i * RS + 4 * gg, acc);
    for (int64_t e = a.row_off[i]; e < a.row_off[i + 1]; ++e) {
        const int64_t j = a.cols[e];
        const Pos<T> pj = load_pos(tag, a.pos, j);
        T dx, dy, dz;
        sep(a.sp, pi, pj, dx, dy, dz);              // d_ij = x_j - x_i
        const T r = sqrt_(dx * dx + dy * dy + dz * dz);
        const T wi = spline_w_(r, iHi);
        const T wj = spline_w_(r, a.geo[8 * j]);
        T gj[12];
        vload<12>(gam + j * 12 * G + 12 * gg, gj);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const T vx = gi[3 * q] * wi + gj[3 * q] * wj;
            const T vy = gi[3 * q + 1] * wi + gj[3 * q + 1] * wj;
            const T vz = gi[3 * q + 2] * wi + gj[3 * q + 2] * wj;
            acc[q] -= dx * vx + dy * vy + dz * vz;
        }
    }
    vstore<4>(lam_out + i * RS + 4 * gg, acc);
}

// dL/dL_s,g += dt sum over the source's entries of (xi / V_target) lambda_E,g(target): one
// warp per (source, group); its lanes load 32 consecutive entries at a time and every lane adds
// their terms in entry order (the same sum in all lanes)
template <class T>
__global__ void k_adj_inject(const int64_t* __restrict__ src_off, const int32_t* __restrict__ e_gas,
                             const double* __restrict__ e_xi, const double* __restrict__ V, const T* __restrict__ lam,
                             int64_t S, int G, const double* __restrict__ dt_dev, double* dLdL) {
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= S * G) return;   // whole warps
    const int64_t s = w / G;
    const int g = (int)(w % G);
    const int64_t e0 = src_off[s], e1 = src_off[s + 1];
    double acc = 0.0;
    for (int64_t b = e0; b < e1; b += 32) {
        const int64_t e = b + lane;
        double q = 0.0, l = 0.0;
        if (e < e1) {
            const int64_t p = e_gas[e];
            q = e_xi[e] / V[p];
            l = (double)lam[p * 4 * G + 4 * g];
        }
        const int m = e1 - b < 32 ? (int)(e1 - b) : 32;
        for (int u = 0; u < m; ++u)
            acc = fma(__shfl_sync(0xffffffffu, q, u), __shfl_sync(0xffffffffu, l, u), acc);
    }
    if (lane == 0) dLdL[w] += *dt_dev * acc;
}

template <class T>
static void launch_adj_step(rt_ctx* c, cudaStream_t s, const T* lamN, const T* W, T* ub, T* gam, T* lamO,
                            bool has_alpha) {
    PairArgs<T> a = pair_args<T>(c);
    FluxExtra<T> x;
    x.wave = nullptr;   // GLF only
    x.alpha = has_alpha ? c->alpha_s.as<T>() : nullptr;
    x.alpha_g = nullptr;   // grey sink only
    x.acc = nullptr;
    x.inj = nullptr;
    x.dt_dev = c->dt_dev.as<double>();
    x.c = (T)c->cfg.c_red;
    x.clamp = 0;
    x.clamp_count = nullptr;
    const int G = c->cfg.n_groups;
    if (c->adj_slots.p) {
        T* mu = c->adj_x.as<T>();      // free between the forward steps
        T* slots = c->adj_slots.as<T>();
        uint8_t* sel = c->adj_sel.as<uint8_t>();
        T* pb = c->pairbuf.as<T>();
        const unsigned nbp = nblk_(std::max<int64_t>(a.n_pairs, 1), 128);
        k_adj_mu<T><<<nblk_(c->n * G, 256), 256, 0, s>>>(a, x, lamN, mu);
        ++c->launches;
        for (int g0 = 0; g0 < G; g0 += chunk_groups(G)) {
            const int gc = G - g0 < chunk_groups(G) ? G - g0 : chunk_groups(G);
            const unsigned nbg = nblk_(c->n * gc, 128);
#define RT_ADJ_PAIRS(GC_)                                                                      \
    k_adj_pair<T, GC_><<<nbp, 128, 0, s>>>(a, x.c, mu, W, slots, sel, g0);                      \
    k_adj_gather<T, GC_><<<nbg, 128, 0, s>>>(a, x, lamN, slots, sel, ub, gam, g0);             \
    k_adj_grad_pair<T, GC_><<<nbp, 128, 0, s>>>(a, x.c, gam, pb, g0);                           \
    k_adj_grad_gather<T, GC_><<<nbg, 128, 0, s>>>(a, ub, pb, lamO, g0);
            switch (gc) {
                case 1: RT_ADJ_PAIRS(1) break;
                case 2: RT_ADJ_PAIRS(2) break;
                case 3: RT_ADJ_PAIRS(3) break;
                default: RT_ADJ_PAIRS(4) break;
            }
#undef RT_ADJ_PAIRS
            c->launches += 4;
        }
        return;
    }
    for (int g0 = 0; g0 < G; g0 += chunk_groups(G)) {
        int gc = G - g0 < chunk_groups(G) ? G - g0 : chunk_groups(G);
        const unsigned nbg = nblk_(c->n * gc, 128);
        switch (gc) {
            case 1: k_adj_flux<T, 1><<<nbg, 128, 0, s>>>(a, x, lamN, W, ub, gam, g0); break;
            case 2: k_adj_flux<T, 2><<<nbg, 128, 0, s>>>(a, x, lamN, W, ub, gam, g0); break;
            case 3: k_adj_flux<T, 3><<<nbg, 128, 0, s>>>(a, x, lamN, W, ub, gam, g0); break;
            default: k_adj_flux<T, 4><<<nbg, 128, 0, s>>>(a, x, lamN, W, ub, gam, g0); break;
        }
    }
    for (int g0 = 0; g0 < G; g0 += chunk_groups(G)) {
        int gc = G - g0 < chunk_groups(G) ? G - g0 : chunk_groups(G);
        const unsigned nbg = nblk_(c->n * gc, 128);
        switch (gc) {
            case 1: k_adj_grad<T, 1><<<nbg, 128, 0, s>>>(a, ub, gam, lamO, g0); break;
            case 2: k_adj_grad<T, 2><<<nbg, 128, 0, s>>>(a, ub, gam, lamO, g0); break;
            case 3: k_adj_grad<T, 3><<<nbg, 128, 0, s>>>(a, ub, gam, lamO, g0); break;
            default: k_adj_grad<T, 4><<<nbg, 128, 0, s>>>(a, ub, gam, lamO, g0); break;
        }
    }
    c->launches += 2 * ((G + chunk_groups(G) - 1) / chunk_groups(G));
}

rt_status run_adjoint(rt_ctx* c, int n_sub, int k, bool has_src, bool has_alpha, const void* U0s,
                      const void* lam_final, void* lam0, double* dLdL) {
    const int G = c->cfg.n_groups;
    const int64_t n = c->n;
    const size_t ts = c->fp64 ? 8 : 4;
    const size_t S = (size_t)4 * G * n * ts;     // one state, bytes
    const int nck = (n_sub + k - 1) / k;
    const int kseg = k < n_sub ? k : n_sub;
    cudaStream_t st = c->stream;
    RT_TRY(ensure(c, c->ck, (size_t)nck * S, "adjoint checkpoints"));
    RT_TRY(ensure(c, c->seg, (size_t)kseg * S, "adjoint segment"));
    RT_TRY(ensure(c, c->adj_w, S, "adjoint"));
    RT_TRY(ensure(c, c->adj_x, S, "adjoint"));
    RT_TRY(ensure(c, c->adj_ub, S, "adjoint"));
    RT_TRY(ensure(c, c->adj_gam, 3 * S, "adjoint"));
    RT_TRY(ensure(c, c->adj_lam, S, "adjoint"));
    // slots of 12 values and a code byte per pair and group of a chunk, where they take no more
    // than half of the memory that is free
    const size_t pg = (size_t)std::max<int64_t>(c->n_directed / 2, 1) * (G < kMaxGC ? G : kMaxGC);
    if (c->adj_slots.bytes < pg * 12 * ts || c->adj_sel.bytes < pg) {
        size_t free_b = 0, total_b = 0;
        free_buf(c->adj_slots);
        free_buf(c->adj_sel);
        RT_CUDA(c, cudaMemGetInfo(&free_b, &total_b));
        if (pg * (12 * ts + 1) <= free_b / 2) {
            if (ensure(c, c->adj_slots, pg * 12 * ts, "adjoint slots") != RT_OK ||
                ensure(c, c->adj_sel, pg, "adjoint slots") != RT_OK) {
                c->err.clear();          // the stages without slots run
                free_buf(c->adj_slots);
                free_buf(c->adj_sel);
            }
        }
    }
    char* ck = c->ck.as<char>();
    char* seg = c->seg.as<char>();
    void* X = c->adj_x.p;
    void* W = c->adj_w.p;

    // forward pass with a checkpoint every k steps
    const int n_last = (nck - 1) * k;
    RT_CUDA(c, cudaMemcpyAsync(X, U0s, S, cudaMemcpyDeviceToDevice, st));
    for (int t = 0; t < n_sub; ++t) {
        if (t % k == 0) RT_CUDA(c, cudaMemcpyAsync(ck + (size_t)(t / k) * S, X, S, cudaMemcpyDeviceToDevice, st));
        // the last segment, the first to be walked back, is kept whole as it passes
        if (t > n_last) RT_CUDA(c, cudaMemcpyAsync(seg + (size_t)(t - n_last) * S, X, S, cudaMemcpyDeviceToDevice, st));
        if (t == n_sub - 1) break;      // the final state is not needed
        RT_TRY(launch_step(c, st, X, W, has_src, has_alpha));
        std::swap(X, W);
    }

    // reverse pass: lambda ping-pongs between the caller's final-lambda copy and adj_lam
    void* lamN = const_cast<void*>(lam_final);
    void* lamO = c->adj_lam.p;
    for (int m = nck - 1; m >= 0; --m) {
        const int n0 = m * k;
        const int len = (n_sub - n0) < k ? (n_sub - n0) : k;
        RT_CUDA(c, cudaMemcpyAsync(seg, ck + (size_t)m * S, S, cudaMemcpyDeviceToDevice, st));
        for (int t = 0; t + 1 < len && m < nck - 1; ++t) {
            RT_CUDA(c, cudaMemcpyAsync(c->adj_x.p, seg + (size_t)t * S, S, cudaMemcpyDeviceToDevice, st));
            RT_TRY(launch_step(c, st, c->adj_x.p, seg + (size_t)(t + 1) * S, has_src, has_alpha));
        }
        for (int t = len - 1; t >= 0; --t) {
            RT_CUDA(c, cudaMemcpyAsync(c->adj_w.p, seg + (size_t)t * S, S, cudaMemcpyDeviceToDevice, st));
            if (has_src) RT_TRY(launch_inject(c, st, c->adj_w.p));
            RT_TRY(launch_gradient(c, st, c->adj_w.p));
            if (c->fp64)
                launch_adj_step<double>(c, st, (const double*)lamN, c->adj_w.as<double>(), c->adj_ub.as<double>(),
                                        c->adj_gam.as<double>(), (double*)lamO, has_alpha);
            else
                launch_adj_step<float>(c, st, (const float*)lamN, c->adj_w.as<float>(), c->adj_ub.as<float>(),
                                       c->adj_gam.as<float>(), (float*)lamO, has_alpha);
            if (has_src && dLdL && c->n_inj_entries > 0) {
                int64_t SG = c->n_src * G;   // one warp each
                if (c->fp64)
                    k_adj_inject<double><<<nblk_(SG * 32, 128), 128, 0, st>>>(
                        c->src_off.as<int64_t>(), c->src_entry_gas.as<int32_t>(), c->src_entry_xi.as<double>(),
                        c->V_d.as<double>(), (const double*)lamO, c->n_src, G, c->dt_dev.as<double>(), dLdL);
                else
                    k_adj_inject<float><<<nblk_(SG * 32, 128), 128, 0, st>>>(
                        c->src_off.as<int64_t>(), c->src_entry_gas.as<int32_t>(), c->src_entry_xi.as<double>(),
                        c->V_d.as<double>(), (const float*)lamO, c->n_src, G, c->dt_dev.as<double>(), dLdL);
                ++c->launches;
            }
            RT_CUDA(c, cudaGetLastError());
            std::swap(lamN, lamO);     // lamN: dL/dU at the start of this step
        }
    }
    if (lamN != lam0) RT_CUDA(c, cudaMemcpyAsync(lam0, lamN, S, cudaMemcpyDeviceToDevice, st));
    return RT_OK;
}

}  // namespace rt
