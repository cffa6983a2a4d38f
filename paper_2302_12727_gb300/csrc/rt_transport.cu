// Transport kernels of the FVPM photon-transport step (Ivkovic 2023, Part III,
// "One RT Time Step"): injection, least-squares gradients, the pair flux loop with
// minmod-limited face states, M1 closure and GLF flux, the explicit update, the grey sink
// and the energy diagnostic.
//
// Layout (cell-sorted order): per particle a state record of 4G values (E, Fx, Fy, Fz per
// group), a gradient record of 12G values (d/dx, d/dy, d/dz per component), a position
// record (fixed-point uint4 for the float path, 4 doubles for the double path) and a
// geometry record of 8 values {1/H, h, Bp (6)} with Bp = V^2 sigma / H^3 B so that
// V_i psitilde_j(x_i) = Bp_i d w(q).  A neighbour's data is then a few 16-byte loads.
//
// The gradient kernels run one thread per particle (or per particle and group) over its
// symmetric neighbour list; the double path keeps the geometry of pairs and rows.  The flux of each unordered pair (k < l) is evaluated once, by
// one thread with k as the left state, and stored in the pair's slot (three launch variants:
// direct loads, cp.async staging, or TMA row gathers of packed flux rows that the gradient
// pass writes); a gather kernel lets every particle add the fluxes of its upper pairs and
// subtract those of its lower pairs in a fixed order.  Both particles thus apply the very
// same Phi_kl with opposite signs: the exchange is exactly antisymmetric, and so exactly
// conservative, deterministic, and free of atomics.  With individual time bins the same
// kernels run on the active sets of each min-step (BINS instantiations, k_gather_bins) and the fluxes are
// weighted by min(dt_k, dt_l) and accumulated until each particle's step ends.
#include <cuda.h>
#include <cudaTypedefs.h>

#include "rt_pair.cuh"

namespace rt {

static inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// Default block sizes of the shuffle gradient and the per-group gather (rt_tuning's
// gradient_block and gather_block choose others at run time).  Rows of different lengths
// make the warps of a block finish at different times, and a block's registers are freed
// only with its last warp: 64-thread gradient blocks run 3% faster than 256-thread ones
// (0.139 against 0.144 ms per launch on the 262,144-particle set); the gather, whose warps
// finish more evenly, keeps 256 (128 is 2% slower there).  The kernels are compiled for the
// largest block of their range, with the register cap the default block had.
constexpr int kGradBlock = 64, kGatherBlock = 256, kGradBlockMax = 256, kGatherBlockMax = 512;

static int grad_block(const rt_ctx* c) {
    if (c->tune.gradient_block > 0) return c->tune.gradient_block;
    return c->tune.gradient_variant == 2 ? kGradBlock : 256;
}
static int gather_block(const rt_ctx* c) { return c->tune.gather_block > 0 ? c->tune.gather_block : kGatherBlock; }
// fewer (particle, group)s than eight warps per SM: the gradient and the gather then take the
// kernels with more loads in flight per thread, with the default gradient (variant 2) only, so that
// the other variants time what they name.  50 sub-cycles of one to four groups just below the line:
// 2.48 -> 2.15, 2.05 -> 1.66, 1.95 -> 1.59 and 1.97 -> 1.58 ms; at a sixteenth of it 1.60 -> 1.00,
// 1.54 -> 1.02, 1.28 -> 0.94 and 1.45 -> 0.96 ms (up to 4% of that from other kernels)
static bool few_threads(const rt_ctx* c, int gc) {
    return c->tune.gradient_variant == 2 && c->n * gc < (int64_t)c->sm_count * 256;
}
static int pair_warps(const rt_ctx* c) { return c->tune.pair_warps > 0 ? c->tune.pair_warps : 1; }

// ------------------------------------------------------------------------------------
// caller order <-> cell-sorted records
// One thread per particle (caller order) and four components: the caller's planes are read and
// written side by side, the records in pieces of four values.  Records filled in sorted order
// instead, each value a 4-byte read at a random place, took 0.385 ms for 2,097,152 particles of
// four groups.
template <class T>
__global__ void __launch_bounds__(256) k_state_in(const T* __restrict__ src, const int32_t* __restrict__ inv_perm,
                                                  int64_t n, int RS, T* __restrict__ rec) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = 4 * blockIdx.y;
    T v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = src[(c + q) * n + i];
    vstore<4>(rec + (int64_t)inv_perm[i] * RS + c, v);
}

template <class T>
__global__ void __launch_bounds__(256) k_state_out(const T* __restrict__ rec, const int32_t* __restrict__ inv_perm,
                                                   int64_t n, int RS, T* __restrict__ dst) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = 4 * blockIdx.y;
    T v[4];
    vload<4>(rec + (int64_t)inv_perm[i] * RS + c, v);
#pragma unroll
    for (int q = 0; q < 4; ++q) dst[(c + q) * n + i] = v[q];
}

// plain SoA gathers (double per-particle fields)
template <class T>
__global__ void k_from_sorted(const T* __restrict__ src, const int32_t* __restrict__ inv_perm, int64_t n, int comps,
                              T* dst) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t p = inv_perm[i];
    for (int c = 0; c < comps; ++c) dst[c * n + i] = src[c * n + p];
}

template <class T>
__global__ void k_alpha_sorted(const double* __restrict__ alpha, const int32_t* __restrict__ perm, int64_t n, T* out) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    out[p] = (T)alpha[perm[p]];
}

// per-group absorption [G][N] (caller order) -> [N][G] sorted, working precision
template <class T>
__global__ void k_alpha_g_sorted(const double* __restrict__ ag, const int32_t* __restrict__ perm, int64_t n, int G,
                                 T* out) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int64_t i = perm[p];
    for (int g = 0; g < G; ++g) out[p * G + g] = (T)ag[(int64_t)g * n + i];
}

__global__ void k_set_scalar(double* dst, double dt, int64_t n_targets) {
    dst[0] = dt;
    reinterpret_cast<int64_t*>(dst)[1] = n_targets;
}

// ------------------------------------------------------------------------------------
// a5: injection, one thread per target particle: E_g += dt * sum_e coef_e L[src_e][g]
// (coef = xi / V_target), accumulated in double.
// the number of targets stands behind dt (set_step_inputs): a captured graph outlives a rebuild
// that changes it
__device__ __forceinline__ int64_t n_targets_of(const double* dt_dev) { return reinterpret_cast<const int64_t*>(dt_dev)[1]; }

template <class T>
__global__ void k_inject(const int32_t* __restrict__ targets, const int32_t* __restrict__ off,
                         const int32_t* __restrict__ src, const double* __restrict__ coef,
                         const double* __restrict__ L, int G, const double* __restrict__ dt_dev, int RS, T* rec,
                         const int8_t* __restrict__ bins, int s) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n_targets_of(dt_dev)) return;
    double dt = *dt_dev;
    int64_t p = targets[t];
    if (bins) {   // time bins: only particles starting a step, for their own step
        const int b = bins[p];
        if (s & ((1 << b) - 1)) return;
        dt = ldexp(dt, b);
    }
    for (int g = 0; g < G; ++g) {
        double acc = 0.0;
        for (int e = off[t]; e < off[t + 1]; ++e) acc += coef[e] * L[(int64_t)src[e] * G + g];
        T* E = rec + p * RS + 4 * g;
        *E = (T)__dadd_rn((double)*E, __dmul_rn(dt, acc));
    }
}

// The same increments dt sum coef L per (particle, group) into inj [N][G] (zeroed before),
// for a gather epilogue to add: E = (T)((double)E + inj) rounds as k_inject does.
__global__ void k_inject_dense(const int32_t* __restrict__ targets, const int32_t* __restrict__ off,
                               const int32_t* __restrict__ src, const double* __restrict__ coef,
                               const double* __restrict__ L, int G, const double* __restrict__ dt_dev,
                               int64_t n_targets, double* __restrict__ inj) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n_targets) return;
    const double dt = *dt_dev;
    const int64_t p = targets[t];
    for (int g = 0; g < G; ++g) {
        double acc = 0.0;
        for (int e = off[t]; e < off[t + 1]; ++e) acc += coef[e] * L[(int64_t)src[e] * G + g];
        inj[p * G + g] = __dmul_rn(dt, acc);
    }
}

// the logical words of particle i's packed flux row (after its prefix)
template <class T>
__device__ __forceinline__ T* packed_row(const PairArgs<T>& a, int64_t i) {
    return a.frec + i * (int64_t)(a.RW + kRowRot) + kRowRot;
}

// logical words [w, w + K) of a packed row (w a multiple of 4); those among the last kRowRot
// are written into the prefix too
template <int K, class T>
__device__ __forceinline__ void row_store(const PairArgs<T>& a, T* row, int w, const T* v) {
    vstore<K>(row + w, v);
#pragma unroll
    for (int k = 0; k < K; k += 4)
        if (w + k >= a.RW - kRowRot) vstore<4>(row + (w + k) - a.RW, v + k);
}

// position and geometry words of particle i's packed flux row (never among the last kRowRot)
template <class T>
__device__ __forceinline__ void packed_static(const PairArgs<T>& a, int64_t i, T* row) {
    if constexpr (std::is_same<T, float>::value) {
        *reinterpret_cast<uint4*>(row) = reinterpret_cast<const uint4*>(a.pos)[i];
        float g8[8];
        vload<8>(a.geo + 8 * i, g8);
        vstore<8>(row + 4, g8);
    }
}

// ------------------------------------------------------------------------------------
// a6: least-squares gradient (Eq. gradient) of the groups [g0, g0 + GC):
// grad Q_i = omega_i Bp_i sum_j (Q_j - Q_i) w(r_ij / H_i) d_ij,  d_ij = x_j - x_i
template <class T, int GC, bool BINS = false>
__global__ void __launch_bounds__(128) k_gradient(PairArgs<T> a, const T* __restrict__ rec, T* __restrict__ grad,
                                                  int g0) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if constexpr (BINS) {   // time bins: the particles starting a step (an ordered prefix)
        if (i >= a.count) return;
        i = a.order[i];
    } else {
        if (i >= a.n) return;
    }
    constexpr int NC = 4 * GC;
    const T* tag = nullptr;
    Pos<T> pi = load_pos(tag, a.pos, i);
    const T iH = a.geo[8 * i];
    const int RS = 4 * a.G;
    T ui[NC];
    vload<NC>(rec + i * RS + 4 * g0, ui);
    T acc[NC][3];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c][0] = acc[c][1] = acc[c][2] = T(0);
    const int64_t e0 = a.row_off[i], e1 = a.row_off[i + 1];
    // two neighbours per iteration: both neighbours' loads are in flight together
    for (int64_t e = e0; e < e1; e += 2) {
        const bool two = e + 1 < e1;
        const int j0 = a.cols[e];
        const int j1 = two ? a.cols[e + 1] : j0;
        Pos<T> p0 = load_pos(tag, a.pos, j0);
        Pos<T> p1 = load_pos(tag, a.pos, j1);
        T u0[NC], u1[NC];
        vload<NC>(rec + (int64_t)j0 * RS + 4 * g0, u0);
        vload<NC>(rec + (int64_t)j1 * RS + 4 * g0, u1);
        T dx0, dy0, dz0, dx1, dy1, dz1;
        sep(a.sp, pi, p0, dx0, dy0, dz0);
        sep(a.sp, pi, p1, dx1, dy1, dz1);
        T w0 = spline_w_(sqrt_(norm2_(dx0, dy0, dz0)), iH);
        T w1 = two ? spline_w_(sqrt_(norm2_(dx1, dy1, dz1)), iH) : T(0);
        T wx0 = w0 * dx0, wy0 = w0 * dy0, wz0 = w0 * dz0;
        T wx1 = w1 * dx1, wy1 = w1 * dy1, wz1 = w1 * dz1;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            T dq0 = u0[c] - ui[c];
            T dq1 = u1[c] - ui[c];
            acc[c][0] = fma_rn(dq1, wx1, fma_rn(dq0, wx0, acc[c][0]));
            acc[c][1] = fma_rn(dq1, wy1, fma_rn(dq0, wy0, acc[c][1]));
            acc[c][2] = fma_rn(dq1, wz1, fma_rn(dq0, wz0, acc[c][2]));
        }
    }
    T M[6];
    const T om = a.omega[i];
#pragma unroll
    for (int k = 0; k < 6; ++k) M[k] = om * a.geo[8 * i + 2 + k];
    T out[3 * NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) sym_mv(M, acc[c][0], acc[c][1], acc[c][2], out[3 * c], out[3 * c + 1], out[3 * c + 2]);
    if (a.frec) {
        T* row = packed_row(a, i);
        row_store<3 * NC>(a, row, 12 + NC, out);
        row_store<NC>(a, row, 12, ui);
        packed_static(a, i, row);
    } else {
        vstore<3 * NC>(grad + i * 12 * a.G + 12 * g0, out);
    }
}

// The double path's kept pair geometry (load_pair_geo, k_gradient_wd): one thread per pair slot
// writes the flux geometry and the two spline weights, one warp per row the entries' w d.
// The double pipe bounds this path, and every sub-cycle and reverse step of a build shares
// the geometry, which is a third of the flux kernel's double instructions and three quarters of
// the gradient's; reading it back costs 64 bytes a pair and 24 an entry.
__global__ void __launch_bounds__(128) k_pair_geometry(PairArgs<double> a, double c, PairGeo<double>* pg,
                                                       double* wkl) {
    const int64_t slot = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (slot >= a.pairs()) return;
    const int2 kl = a.ends[slot];
    PairGeo<double> p;
    double sk, sl;
    load_pair_geo(a, slot, kl.x, kl.y, c, p, sk, sl);
    vstore<8>(reinterpret_cast<double*>(pg + slot), reinterpret_cast<const double*>(&p));
    *reinterpret_cast<double2*>(wkl + 2 * slot) = make_double2(sk, sl);
}

__global__ void __launch_bounds__(256) k_row_weights(PairArgs<double> a, double* __restrict__ wd) {
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= a.n) return;
    const double* tag = nullptr;
    const Pos<double> pi = load_pos(tag, a.pos, i);
    const double iH = a.geo[8 * i];
    for (int64_t e = a.row_off[i] + lane; e < a.row_off[i + 1]; e += 32) {
        const Pos<double> pj = load_pos(tag, a.pos, a.cols[e]);
        double dx, dy, dz;
        sep(a.sp, pi, pj, dx, dy, dz);
        const double r2 = norm2_(dx, dy, dz);
        const double w = r2 > 0.0 ? spline_w_(sqrt_fast(r2), iH) : 0.0;
        wd[3 * e] = w * dx;
        wd[3 * e + 1] = w * dy;
        wd[3 * e + 2] = w * dz;
    }
}

rt_status prepare_pair_geometry(rt_ctx* c) {
    if (!c->fp64 || c->pair_geo_ready || !c->pair_geo.p) return RT_OK;
    const PairArgs<double> a = pair_args<double>(c);   // pair_geo_ready is false: computes
    k_pair_geometry<<<nblk(std::max<int64_t>(a.n_pairs, 1), 128), 128, 0, c->stream>>>(
        a, c->cfg.c_red, static_cast<PairGeo<double>*>(c->pair_geo.p), c->pair_w.as<double>());
    k_row_weights<<<nblk(c->n * 32, 256), 256, 0, c->stream>>>(a, c->row_wd.as<double>());
    c->launches += 2;
    RT_CUDA(c, cudaGetLastError());
    c->pair_geo_ready = true;
    return RT_OK;
}

// Double gradient from the kept row weights: 16 double instructions per entry and group are
// left.  LN lanes share the row of one (particle, group), every LN-th entry each, so that small
// sets still fill the double pipes of all SMs; at LN = 4 the sums are reduced so that each
// lane ends with one component and applies B_i to it alone.
template <int GC, int LN, bool BINS>
__global__ void __launch_bounds__(128) k_gradient_wd(PairArgs<double> a, const double* __restrict__ rec,
                                                     double* __restrict__ grad, int g0) {
    static_assert(LN == 1 || LN == 4, "lanes per (particle, group)");
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int sub = (int)(t % LN);
    const int64_t q = t / LN;
    int64_t i = q / GC;
    const int g = (int)(q - i * GC);
    const bool act = i < (BINS ? a.count : a.n);
    i = act ? (BINS ? (int64_t)a.order[i] : i) : 0;
    const int RS = 4 * a.G, off = 4 * (g0 + g);
    double ui[4], acc[4][3];
    vload<4>(rec + i * RS + off, ui);
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c][0] = acc[c][1] = acc[c][2] = 0.0;
    const int64_t e1 = act ? a.row_off[i + 1] : 0;
#pragma unroll 2
    for (int64_t e = act ? a.row_off[i] + sub : 0; e < e1; e += LN) {
        double u[4];
        vload<4>(rec + (int64_t)a.cols[e] * RS + off, u);
        const double wx = a.wd[3 * e], wy = a.wd[3 * e + 1], wz = a.wd[3 * e + 2];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const double dq = u[c] - ui[c];
            acc[c][0] += dq * wx;
            acc[c][1] += dq * wy;
            acc[c][2] += dq * wz;
        }
    }
    if constexpr (LN == 4) {
        const bool hi = sub & 2, odd = sub & 1;
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int d = 0; d < 3; ++d) {   // lanes 0, 1 keep components 0, 1; lanes 2, 3 the others
                const double give = hi ? acc[c][d] : acc[c + 2][d], keep = hi ? acc[c + 2][d] : acc[c][d];
                acc[c][d] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
            }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double give = odd ? acc[0][d] : acc[1][d], keep = odd ? acc[1][d] : acc[0][d];
            acc[0][d] = keep + __shfl_xor_sync(0xffffffffu, give, 1);
        }
    }
    if (!act) return;
    double M[6];
    const double om = a.omega[i];
#pragma unroll
    for (int k = 0; k < 6; ++k) M[k] = om * a.geo[8 * i + 2 + k];
    double* out = grad + i * 12 * a.G + 12 * (g0 + g) + 3 * sub;
#pragma unroll
    for (int c = 0; c < (LN == 4 ? 1 : 4); ++c)
        sym_mv(M, acc[c][0], acc[c][1], acc[c][2], out[3 * c], out[3 * c + 1], out[3 * c + 2]);
}

// lanes per (particle, group) of the double gradient: four up to the size where one lane each
// gives every SM's four double pipes eight warps
template <int GC, bool BINS>
static void launch_gradient_wd(rt_ctx* c, cudaStream_t s, const PairArgs<double>& a, const double* rec, double* grad,
                               int g0) {
    const int64_t m = (BINS ? a.count : a.n) * GC;
    if (c->n * GC < (int64_t)c->sm_count * 1024)
        k_gradient_wd<GC, 4, BINS><<<nblk(4 * m, 128), 128, 0, s>>>(a, rec, grad, g0);
    else
        k_gradient_wd<GC, 1, BINS><<<nblk(m, 128), 128, 0, s>>>(a, rec, grad, g0);
}

// Float gradient with one thread per (particle, group): the GC lanes of a particle read the
// same neighbour position and neighbouring 16-byte pieces of the same state record, so a
// warp request touches about 32 / GC records instead of 32.  Same neighbour pairing and
// order of accumulation as k_gradient.
template <int GC, bool BINS = false>
__global__ void __launch_bounds__(256) k_gradient_g(PairArgs<float> a, const float* __restrict__ rec,
                                                    float* __restrict__ grad, int g0) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t i = t / GC;
    const int g = (int)(t - i * GC);
    if (i >= (BINS ? a.count : a.n)) return;
    if constexpr (BINS) i = a.order[i];      // the particles starting a step (an ordered prefix)
    const float* tag = nullptr;
    const Pos<float> pi = load_pos(tag, a.pos, i);
    const float iH = a.geo[8 * i];
    const int RS = 4 * a.G;
    const int off = 4 * (g0 + g);
    float ui[4];
    vload<4>(rec + i * RS + off, ui);
    float acc[4][3];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c][0] = acc[c][1] = acc[c][2] = 0.f;
    const int64_t e0 = a.row_off[i], e1 = a.row_off[i + 1];
    for (int64_t e = e0; e < e1; e += 2) {
        const bool two = e + 1 < e1;
        const int j0 = a.cols[e];
        const int j1 = two ? a.cols[e + 1] : j0;
        Pos<float> p0 = load_pos(tag, a.pos, j0);
        Pos<float> p1 = load_pos(tag, a.pos, j1);
        float u0[4], u1[4];
        vload<4>(rec + (int64_t)j0 * RS + off, u0);
        vload<4>(rec + (int64_t)j1 * RS + off, u1);
        float dx0, dy0, dz0, dx1, dy1, dz1;
        sep(a.sp, pi, p0, dx0, dy0, dz0);
        sep(a.sp, pi, p1, dx1, dy1, dz1);
        float w0 = spline_w_(sqrt_(norm2_(dx0, dy0, dz0)), iH);
        float w1 = two ? spline_w_(sqrt_(norm2_(dx1, dy1, dz1)), iH) : 0.f;
        float wx0 = mul_rn(w0, dx0), wy0 = mul_rn(w0, dy0), wz0 = mul_rn(w0, dz0);
        float wx1 = w1 * dx1, wy1 = w1 * dy1, wz1 = w1 * dz1;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float dq0 = u0[c] - ui[c];
            float dq1 = u1[c] - ui[c];
            acc[c][0] = fma_rn(dq1, wx1, fma_rn(dq0, wx0, acc[c][0]));
            acc[c][1] = fma_rn(dq1, wy1, fma_rn(dq0, wy0, acc[c][1]));
            acc[c][2] = fma_rn(dq1, wz1, fma_rn(dq0, wz0, acc[c][2]));
        }
    }
    float M[6];
    const float om = a.omega[i];
#pragma unroll
    for (int k = 0; k < 6; ++k) M[k] = om * a.geo[8 * i + 2 + k];
    float out[12];
#pragma unroll
    for (int c = 0; c < 4; ++c) sym_mv(M, acc[c][0], acc[c][1], acc[c][2], out[3 * c], out[3 * c + 1], out[3 * c + 2]);
    if (a.frec) {
        float* row = packed_row(a, i);
        row_store<12>(a, row, 12 + 4 * GC + 12 * g, out);
        row_store<4>(a, row, 12 + 4 * g, ui);
        if (g == 0) packed_static(a, i, row);
    } else {
        vstore<12>(grad + i * 12 * a.G + 12 * (g0 + g), out);
    }
}

// k_gradient_g for sets too small to fill the GPU, where the gradient is the latency of one
// thread's chain of loads: eight neighbours' indices, then their positions and states in
// flight together instead of two.  Same order and sums.  4,096 particles, one group: 24.1 us a
// launch with two in flight.
constexpr int kWide = 8;
template <int GC>
__global__ void __launch_bounds__(64) k_gradient_w(PairArgs<float> a, const float* __restrict__ rec,
                                                   float* __restrict__ grad, int g0) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = t / GC;
    if (i >= a.n) return;
    const int g = (int)(t - i * GC);
    const float* tag = nullptr;
    const Pos<float> pi = load_pos(tag, a.pos, i);
    const int RS = 4 * a.G;
    const int off = 4 * (g0 + g);
    const int64_t e0 = a.row_off[i];
    const int m = (int)(a.row_off[i + 1] - e0);
    const int32_t* row = a.cols + e0;
    float ui[4], geo[8];
    vload<4>(rec + i * RS + off, ui);
    vload<8>(a.geo + 8 * i, geo);
    const float om = a.omega[i], iH = geo[0];
    float acc[4][3];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c][0] = acc[c][1] = acc[c][2] = 0.f;
    int j[kWide];
#pragma unroll
    for (int k = 0; k < kWide; ++k) j[k] = m > 0 ? row[min(k, m - 1)] : (int)i;   // past the end: weight zero
    for (int b = 0; b < m; b += kWide) {
        Pos<float> p[kWide];
        float u[kWide][4];
#pragma unroll
        for (int k = 0; k < kWide; ++k) {
            p[k] = load_pos(tag, a.pos, j[k]);
            vload<4>(rec + (int64_t)j[k] * RS + off, u[k]);
        }
#pragma unroll
        for (int k = 0; k < kWide; ++k) j[k] = row[min(b + kWide + k, m - 1)];
#pragma unroll
        for (int k = 0; k < kWide; ++k) {
            float dx, dy, dz;
            sep(a.sp, pi, p[k], dx, dy, dz);
            const float w = b + k < m ? spline_w_(sqrt_(norm2_(dx, dy, dz)), iH) : 0.f;
            const float wx = w * dx, wy = w * dy, wz = w * dz;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float dq = u[k][c] - ui[c];
                acc[c][0] = fma_rn(dq, wx, acc[c][0]);
                acc[c][1] = fma_rn(dq, wy, acc[c][1]);
                acc[c][2] = fma_rn(dq, wz, acc[c][2]);
            }
        }
    }
    float M[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) M[k] = om * geo[2 + k];
    float out[12];
#pragma unroll
    for (int c = 0; c < 4; ++c) sym_mv(M, acc[c][0], acc[c][1], acc[c][2], out[3 * c], out[3 * c + 1], out[3 * c + 2]);
    if (a.frec) {
        float* to = packed_row(a, i);
        row_store<12>(a, to, 12 + 4 * GC + 12 * g, out);
        row_store<4>(a, to, 12 + 4 * g, ui);
        if (g == 0) packed_static(a, i, to);
    } else {
        vstore<12>(grad + i * 12 * a.G + 12 * (g0 + g), out);
    }
}

// Float gradient with the GC lanes of a particle sharing the neighbour geometry: a warp
// holds 32 / GC particles; per block of 2 GC neighbours each lane computes the separation,
// spline weight and w d of two consecutive neighbours and passes them to the particle's
// other lanes with warp shuffles, so the geometry is computed once instead of GC times.
// Neighbours stay paired (e, e + 1) from the row start and the accumulation is the same
// expression in the same order as k_gradient_g, so the result bits are the same.  With four
// groups (eight particles per warp, every lane busy) five blocks per SM (48 registers, a few
// spilled) beat four at 64 registers by 7%; with three groups they lose 2%.
template <int GC, bool BINS = false>
__global__ void __launch_bounds__(kGradBlockMax, GC == 4 ? 1280 / kGradBlockMax : 0) k_gradient_s(PairArgs<float> a, const float* __restrict__ rec,
                                                    float* __restrict__ grad, int g0) {
    constexpr int P = 32 / GC;                     // particles per warp
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int q = lane / GC, g = lane - (lane / GC) * GC;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    // BINS: the particles starting a step (an ordered prefix)
    const int64_t at = warp * P + q;
    const bool act = q < P && at < (BINS ? a.count : a.n);   // lanes past P GC and past the last particle idle
    const int64_t i = act ? (BINS ? (int64_t)a.order[at] : at) : 0;
    const int64_t ii = i;
    const float* tag = nullptr;
    const Pos<float> pi = load_pos(tag, a.pos, ii);
    const float iH = a.geo[8 * ii];
    const int RS = 4 * a.G;
    const int off = 4 * (g0 + g);
    float ui[4];
    vload<4>(rec + ii * RS + off, ui);
    float acc[4][3];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c][0] = acc[c][1] = acc[c][2] = 0.f;
    const int64_t e0 = a.row_off[ii], e1 = act ? a.row_off[ii + 1] : e0;
    int nit = (int)((e1 - e0 + 2 * GC - 1) / (2 * GC));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nit = max(nit, __shfl_xor_sync(FULL, nit, o));
    const int base = q * GC;                       // first lane of this particle
    // this lane's pair of neighbours; below four groups their indices load one iteration
    // ahead (at four, the register cap of five blocks per SM leaves no room for them)
    constexpr bool PF = GC < 4;
    int64_t ea = e0 + 2 * g;
    int j0 = 0, j1 = 0;
    if constexpr (PF) {
        j0 = ea < e1 ? a.cols[ea] : 0;
        j1 = ea + 1 < e1 ? a.cols[ea + 1] : j0;
    }
    for (int it = 0; it < nit; ++it) {
        const bool has = ea < e1, two = ea + 1 < e1;
        if constexpr (!PF) {
            j0 = has ? a.cols[ea] : 0;
            j1 = two ? a.cols[ea + 1] : j0;
        }
        const int64_t en = ea + 2 * GC;
        int j0n = 0, j1n = 0;
        if constexpr (PF) {
            j0n = en < e1 ? a.cols[en] : 0;
            j1n = en + 1 < e1 ? a.cols[en + 1] : j0n;
        }
        const Pos<float> p0 = load_pos(tag, a.pos, j0);
        const Pos<float> p1 = load_pos(tag, a.pos, j1);
        float dx0, dy0, dz0, dx1, dy1, dz1;
        sep(a.sp, pi, p0, dx0, dy0, dz0);
        sep(a.sp, pi, p1, dx1, dy1, dz1);
        float w0 = spline_w_(sqrt_(norm2_(dx0, dy0, dz0)), iH);
        float w1 = two ? spline_w_(sqrt_(norm2_(dx1, dy1, dz1)), iH) : 0.f;
        float wx0 = mul_rn(w0, dx0), wy0 = mul_rn(w0, dy0), wz0 = mul_rn(w0, dz0);
        float wx1 = w1 * dx1, wy1 = w1 * dy1, wz1 = w1 * dz1;
        const int hj0 = has ? j0 : -1;
#pragma unroll
        for (int u = 0; u < GC; ++u) {
            const int src = base + u;
            const int J0 = __shfl_sync(FULL, hj0, src), J1 = __shfl_sync(FULL, j1, src);
            const float X0 = __shfl_sync(FULL, wx0, src), Y0 = __shfl_sync(FULL, wy0, src),
                        Z0 = __shfl_sync(FULL, wz0, src);
            const float X1 = __shfl_sync(FULL, wx1, src), Y1 = __shfl_sync(FULL, wy1, src),
                        Z1 = __shfl_sync(FULL, wz1, src);
            if (J0 < 0) continue;
            float u0[4], u1[4];
            vload<4>(rec + (int64_t)J0 * RS + off, u0);
            vload<4>(rec + (int64_t)J1 * RS + off, u1);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float dq0 = u0[c] - ui[c];
                float dq1 = u1[c] - ui[c];
                acc[c][0] = fma_rn(dq1, X1, fma_rn(dq0, X0, acc[c][0]));
                acc[c][1] = fma_rn(dq1, Y1, fma_rn(dq0, Y0, acc[c][1]));
                acc[c][2] = fma_rn(dq1, Z1, fma_rn(dq0, Z0, acc[c][2]));
            }
        }
        ea = en;
        if constexpr (PF) {
            j0 = j0n;
            j1 = j1n;
        }
    }
    if (!act) return;
    float M[6];
    const float om = a.omega[i];
#pragma unroll
    for (int k = 0; k < 6; ++k) M[k] = om * a.geo[8 * i + 2 + k];
    float out[12];
#pragma unroll
    for (int c = 0; c < 4; ++c) sym_mv(M, acc[c][0], acc[c][1], acc[c][2], out[3 * c], out[3 * c + 1], out[3 * c + 2]);
    if (a.frec) {
        float* row = packed_row(a, i);
        row_store<12>(a, row, 12 + 4 * GC + 12 * g, out);
        row_store<4>(a, row, 12 + 4 * g, ui);
        if (g == 0) packed_static(a, i, row);
    } else {
        vstore<12>(grad + i * 12 * a.G + 12 * (g0 + g), out);
    }
}

// ------------------------------------------------------------------------------------
// a7 + a8: pair fluxes, explicit update, grey sink, optional fix-up, groups [g0, g0 + GC).

// The fluxes of a pair with a state beyond the closure's range (M1Top) again, over its slot: the groups'
// states lie at uk, ul, their gradients at gk, gl, side by side
template <bool HLL, int GC, class T>
__device__ __forceinline__ void store_wide(const T* uk, const T* ul, const T* gk, const T* gl, const PairGeo<T>& pr, T c,
                                           const T* wave, T wgt, T* to) {
    M1Top<T> top;
#pragma unroll 1
    for (int g = 0; g < GC; ++g) {
        T ui[4], uj[4], gri[12], grj[12], phi[4];
        vload<4>(uk + 4 * g, ui);
        vload<4>(ul + 4 * g, uj);
        vload<12>(gk + 12 * g, gri);
        vload<12>(gl + 12 * g, grj);
        pair_flux<HLL, true>(ui, uj, gri, grj, pr, c, wave, phi, top);
#pragma unroll
        for (int q = 0; q < 4; ++q) phi[q] *= wgt;
        vstore<4>(to + 4 * g, phi);
    }
}

// Pass 1 of the flux: one thread per unordered pair (k, l), k < l, evaluates Phi_kl once with
// k as the left state and stores it in the pair's slot.
template <class T, int GC, bool HLL, bool BINS = false>
__global__ void __launch_bounds__(128) k_flux(PairArgs<T> a, FluxExtra<T> x, const T* __restrict__ rec,
                                              T* __restrict__ pairbuf, int g0) {
    int64_t slot = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if constexpr (BINS) {   // time bins: the pairs with a starting member (an ordered prefix)
        if (slot >= a.count) return;
        slot = a.order[slot];
    } else {
        if (slot >= a.pairs()) return;
    }
    constexpr int NC = 4 * GC;
    const int G = a.G, RS = 4 * G;
    const int2 kl = a.ends[slot];
    const int64_t i = kl.x, j = kl.y;
    T wgt = T(1);
    if constexpr (BINS) wgt = T(1 << min(a.bins[i], a.bins[j]));   // min(dt_k, dt_l) / dt_min
    PairGeo<T> pr;
    T sk, sl;
    load_pair_geo(a, slot, i, j, x.c, pr, sk, sl);
    const T* ri = rec + i * RS;
    const T* rj = rec + j * RS;
    const T* qi = a.grad + i * 12 * G;
    const T* qj = a.grad + j * 12 * G;
    T out[NC];
    M1Top<T> top;
#pragma unroll
    for (int g = 0; g < GC; ++g) {
        const int gg = g0 + g;
        T ui[4], uj[4], gri[12], grj[12];
        vload<4>(ri + 4 * gg, ui);
        vload<4>(rj + 4 * gg, uj);
        vload<12>(qi + 12 * gg, gri);
        vload<12>(qj + 12 * gg, grj);
        pair_flux<HLL, false>(ui, uj, gri, grj, pr, x.c, x.wave, &out[4 * g], top);
    }
    if constexpr (BINS) {
#pragma unroll
        for (int c = 0; c < NC; ++c) out[c] *= wgt;
    }
    vstore<NC>(pairbuf + slot * NC, out);
    if (top.any)
        store_wide<HLL, GC>(ri + 4 * g0, rj + 4 * g0, qi + 12 * g0, qj + 12 * g0, pr, x.c, x.wave, wgt,
                            pairbuf + slot * NC);
}

// ------------------------------------------------------------------------------------
// Per-particle sum of one group's pair fluxes (E, Fx, Fy, Fz), in a fixed order.  The double
// path adds in double.  The float path keeps the energy row as a compensated float sum:
// Knuth's TwoSum gives the exact rounding error of every addition and a second float
// collects those errors (the cascaded summation of Ogita, Rump and Oishi, "Accurate sum and
// dot product", 2005), so for the ~50 terms of a particle the sum's error stays near
// (50 u)^2 of the sum of magnitudes (u = 2^-24) instead of 50 u; the update then forms the
// energy from the pair in double.  The flux rows add in float.  (A double energy sum costs
// the same gather 2.4 times its time on GB300, whose FP64 rate is 1/64 of FP32; compensated
// flux rows 1.3 times.)  With individual time bins the accumulators stay in memory between
// min-steps: 32 bytes per (particle, group) in both precisions.
template <class T>
struct FluxAcc;

template <>
struct FluxAcc<double> {
    double v[4];
    __device__ __forceinline__ void zero() { v[0] = v[1] = v[2] = v[3] = 0.0; }
    __device__ __forceinline__ void add(const double p[4]) {
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] += p[c];
    }
    __device__ __forceinline__ void sub(const double p[4]) {
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] -= p[c];
    }
    __device__ __forceinline__ double energy() const { return v[0]; }
    __device__ __forceinline__ double flux(int c) const { return v[1 + c]; }
    __device__ __forceinline__ void load(const double* m) { vload<4>(m, v); }
    __device__ __forceinline__ void store(double* m) const { vstore<4>(m, v); }
};

// s + x = t + e exactly (TwoSum, branch-free); e is added to the error sum k
__device__ __forceinline__ void two_sum_into(float& s, float& k, float x) {
    const float t = __fadd_rn(s, x);
    const float z = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z));
    k = __fadd_rn(k, e);
    s = t;
}

template <>
struct FluxAcc<float> {
    float es, ek;    // energy row: sum and error sum
    float f[3];      // flux rows
    __device__ __forceinline__ void zero() { es = ek = f[0] = f[1] = f[2] = 0.f; }
    __device__ __forceinline__ void add(const float p[4]) {
        two_sum_into(es, ek, p[0]);
#pragma unroll
        for (int c = 0; c < 3; ++c) f[c] += p[1 + c];
    }
    __device__ __forceinline__ void sub(const float p[4]) {
        two_sum_into(es, ek, -p[0]);
#pragma unroll
        for (int c = 0; c < 3; ++c) f[c] -= p[1 + c];
    }
    __device__ __forceinline__ double energy() const { return (double)es + (double)ek; }
    __device__ __forceinline__ float flux(int c) const { return f[c]; }
    // record: {es, ek, f0, f1 | f2, unused x 3}
    __device__ __forceinline__ void load(const float* m) {
        const float4 a = *reinterpret_cast<const float4*>(m);
        es = a.x; ek = a.y; f[0] = a.z; f[1] = a.w;
        f[2] = m[4];
    }
    __device__ __forceinline__ void store(float* m) const {
        *reinterpret_cast<float4*>(m) = make_float4(es, ek, f[0], f[1]);
        m[4] = f[2];
    }
};

// words of T per (particle, group) accumulator record in memory (32 bytes)
template <class T>
struct AccRec {
    static constexpr int words = 32 / (int)sizeof(T);
};

// U_g(t + dt) = (U_g - f acc_g) sink for one group (Eq. transport-update-explicit with
// f = dt / V_i, then the forward-Euler sink), the fix-up E >= 0 when on (returns 1 if it
// fired), then the next sub-cycle's injection inj (double, 0 when none).  The float path
// forms the energy from its compensated sum in double and rounds once, before the fix-up
// and the injection, exactly where a plain step stores it.
template <class T>
__device__ __forceinline__ int update_group(T u[4], const FluxAcc<T>& acc, T f, T sink, int clamp, const double* inj) {
    T v0;
    if constexpr (std::is_same<T, float>::value)
        v0 = (float)(((double)u[0] - (double)f * acc.energy()) * (double)sink);
    else
        v0 = (u[0] - f * acc.energy()) * sink;
    int fired = 0;
    if (clamp && v0 < T(0)) {
        v0 = T(0);
        fired = 1;
    }
    if (inj) v0 = (T)__dadd_rn((double)v0, *inj);
    u[0] = v0;
#pragma unroll
    for (int c = 0; c < 3; ++c) u[1 + c] = (u[1 + c] - f * acc.flux(c)) * sink;
    return fired;
}

// Pass 2 with individual time bins: particle i adds to its accumulators the slots of the
// pairs that interacted at min-step s (all of them if i starts a step, else those whose
// partner starts one), in the same order as the uniform gather; at the end of its own step
// ((s + 1) mod 2^b_i = 0) it applies U_i - dt_min / V_i acc_i, the sink over its step
// dt_min 2^b_i and the fix-up, and clears the accumulators.  The states are updated in place
// (this pass runs after the pair pass, and each particle writes only its own record).  One
// thread per (particle, group), the partners' bins and the slots of up to eight pairs in flight:
// one thread per particle and a pair at a time took 0.161 ms a min-step on 262,144 particles of
// four groups.
template <class T, int GC>
__global__ void __launch_bounds__(256) k_gather_bins(PairArgs<T> a, FluxExtra<T> x, const T* __restrict__ pairbuf,
                                                     T* __restrict__ rec, int g0) {
    constexpr int NC = 4 * GC, AW = AccRec<T>::words, B = std::is_same<T, float>::value ? 8 : 4;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t q = t / GC;
    if (q >= a.count) return;
    const int g = (int)(t - q * GC), gg = g0 + g;
    const int64_t i = a.order[q];
    const int bi = a.bins[i];
    const int mask = (1 << bi) - 1;
    const bool start_i = !(a.s & mask);
    T* accp = x.acc + (i * a.G + gg) * AW;
    FluxAcc<T> acc;
    acc.load(accp);
    const int64_t r0 = a.row_off[i], s0 = a.up_off[i];
    const int nu = (int)(a.up_off[i + 1] - s0), nl = a.n_low[i];
    const T* pb = pairbuf + 4 * g;
    // the pairs [e, e + B) of one half of the row: their partners start a step, or i does
    auto batch = [&](const int32_t* cols, int e, int m, auto&& slot, auto&& put) {
        bool on[B];
#pragma unroll
        for (int u = 0; u < B; ++u)
            on[u] = e + u < m && (start_i || !(a.s & ((1 << a.bins[cols[e + u]]) - 1)));
        T p[B][4];
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (on[u]) vload<4>(pb + slot(e + u) * NC, p[u]);
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (on[u]) put(p[u]);
    };
    const int32_t* up = a.cols + r0 + nl;
    for (int e = 0; e < nu; e += B)
        batch(up, e, nu, [&](int u) { return s0 + u; }, [&](const T* p) { acc.add(p); });
    const int32_t* ls = a.low_slot + (r0 - s0);
    for (int e = 0; e < nl; e += B)
        batch(a.cols + r0, e, nl, [&](int u) { return (int64_t)ls[u]; }, [&](const T* p) { acc.sub(p); });
    if ((a.s + 1) & mask) {   // the step of i goes on (the state is updated in place)
        acc.store(accp);
        return;
    }
    T* u = rec + i * 4 * a.G + 4 * gg;
    T ui[4];
    vload<4>(u, ui);
    const T dt = (T)(*x.dt_dev), dti = (T)ldexp(*x.dt_dev, bi);
    T sink = T(1);
    if (x.alpha) sink = fmax_(T(1) - x.c * x.alpha[i] * dti, T(0));
    if (x.alpha_g) sink = fmax_(T(1) - x.c * x.alpha_g[i * a.G + gg] * dti, T(0));
    const int nclamp = update_group<T>(ui, acc, dt * a.omega[i], sink, x.clamp, nullptr);
    acc.zero();
    acc.store(accp);
    vstore<4>(u, ui);
    if (nclamp) atomicAdd(x.clamp_count, (unsigned long long)nclamp);
}

// particles whose step ends at min-step s without any interaction at s (no starting partner,
// nmin > tz): apply the accumulators, the sink over the step and the fix-up, in place
template <class T, int GC>
__global__ void k_finalize_bins(PairArgs<T> a, FluxExtra<T> x, T* __restrict__ rec, int g0) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= a.count) return;
    const int64_t i = a.order[t];
    if (a.nmin[i] <= a.tz) return;       // finalised by the gather of this min-step
    constexpr int NC = 4 * GC, AW = AccRec<T>::words;
    const int RS = 4 * a.G;
    T* accp = x.acc + (i * a.G + g0) * AW;
    T ui[NC];
    vload<NC>(rec + i * RS + 4 * g0, ui);
    const int bi = a.bins[i];
    const T dt = (T)(*x.dt_dev);
    const T dti = (T)ldexp(*x.dt_dev, bi);
    const T f = dt * a.omega[i];
    T sink = T(1);
    if (x.alpha) sink = fmax_(T(1) - x.c * x.alpha[i] * dti, T(0));
    int nclamp = 0;
#pragma unroll
    for (int g = 0; g < GC; ++g) {
        FluxAcc<T> acc;
        acc.load(accp + g * AW);
        const T sk = x.alpha_g ? fmax_(T(1) - x.c * x.alpha_g[i * a.G + g0 + g] * dti, T(0)) : sink;
        nclamp += update_group<T>(ui + 4 * g, acc, f, sk, x.clamp, nullptr);
        acc.zero();
        acc.store(accp + g * AW);
    }
    vstore<NC>(rec + i * RS + 4 * g0, ui);
    if (nclamp) atomicAdd(x.clamp_count, (unsigned long long)nclamp);
}

// Pass 2: particle i adds the fluxes of its own upper pairs (contiguous slots) and subtracts
// those of its lower pairs (k < i, read from k's slots), in a fixed order; then
// U_i(t + dt) = U_i - dt / V_i sum_l F_il . A_il, the sink and the fix-up.
template <class T, int GC>
__global__ void __launch_bounds__(128) k_flux_gather(PairArgs<T> a, FluxExtra<T> x, const T* __restrict__ rec,
                                                     const T* __restrict__ pairbuf, T* __restrict__ out, int g0) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    constexpr int NC = 4 * GC;
    const int RS = 4 * a.G;
    FluxAcc<T> acc[GC];
#pragma unroll
    for (int g = 0; g < GC; ++g) acc[g].zero();
    const int64_t r0 = a.row_off[i], s0 = a.up_off[i], s1 = a.up_off[i + 1];
    for (int64_t sl = s0; sl < s1; ++sl) {
        T phi[NC];
        vload<NC>(pairbuf + sl * NC, phi);
#pragma unroll
        for (int g = 0; g < GC; ++g) acc[g].add(phi + 4 * g);
    }
    const int nl = a.n_low[i];
    const int32_t* ls = a.low_slot + (r0 - s0);
    int e = 0;
    for (; e + 4 <= nl; e += 4) {     // four loads in flight, subtracted in order
        T p[4][NC];
#pragma unroll
        for (int u = 0; u < 4; ++u) vload<NC>(pairbuf + (int64_t)ls[e + u] * NC, p[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int g = 0; g < GC; ++g) acc[g].sub(p[u] + 4 * g);
    }
    for (; e < nl; ++e) {
        T phi[NC];
        vload<NC>(pairbuf + (int64_t)ls[e] * NC, phi);
#pragma unroll
        for (int g = 0; g < GC; ++g) acc[g].sub(phi + 4 * g);
    }
    const T dt = (T)(*x.dt_dev);
    const T f = dt * a.omega[i];
    T sink = T(1);
    if (x.alpha) sink = fmax_(T(1) - x.c * x.alpha[i] * dt, T(0));
    T ui[NC];
    vload<NC>(rec + i * RS + 4 * g0, ui);
    int nclamp = 0;
#pragma unroll
    for (int g = 0; g < GC; ++g) {
        const T sk = x.alpha_g ? fmax_(T(1) - x.c * x.alpha_g[i * a.G + g0 + g] * dt, T(0)) : sink;
        nclamp += update_group<T>(ui + 4 * g, acc[g], f, sk, x.clamp, x.inj ? x.inj + i * a.G + g0 + g : nullptr);
    }
    vstore<NC>(out + i * RS + 4 * g0, ui);
    if (nclamp) atomicAdd(x.clamp_count, (unsigned long long)nclamp);
}

// Float pass 1 with the neighbour records staged through shared memory.  One thread per
// pair slot as in k_flux, but the 32 l-records a warp needs (position, geometry, state and
// gradient of the launched groups) are first copied by the whole warp, one array at a time,
// so that each 16-byte request of the warp covers a few consecutive records instead of 32
// scattered ones; the per-pair loads of the direct kernel saturate the L1 data pipe.  The
// k side needs no staging: consecutive slots mostly share k, so its loads are broadcasts.
// The arithmetic is the same as k_flux's.
template <int GC>
struct Staged {
    static constexpr int RW = 12 + 16 * GC;   // words per staged record: pos 4, geo 8, state 4GC, grad 12GC
    static constexpr int WARPS = 4;
    static constexpr size_t bytes = (size_t)WARPS * 32 * RW * sizeof(float);
};

template <int GC, bool HLL>
__global__ void __launch_bounds__(128) k_flux_staged(PairArgs<float> a, FluxExtra<float> x,
                                                     const float* __restrict__ rec, float* __restrict__ pairbuf,
                                                     int g0) {
    constexpr int NC = 4 * GC, RW = Staged<GC>::RW;
    // RW / 4 is odd for every GC, so the lanes' 16-byte reads of their own records are free
    // of bank conflicts
    __shared__ __align__(16) float st[Staged<GC>::WARPS * 32 * RW];
    const int lane = threadIdx.x & 31;
    float* ws = st + (threadIdx.x >> 5) * 32 * RW;
    const int64_t slot = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool act = slot < a.pairs();
    // lanes past the last slot stage particle 0 (always present) and store nothing
    const int2 kl = act ? a.ends[slot] : make_int2(0, 0);
    const int G = a.G, RS = 4 * G;
    const unsigned FULL = 0xffffffffu;
    cp_async16(ws + lane * RW, reinterpret_cast<const uint4*>(a.pos) + kl.y);
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        const int t = m * 32 + lane, r = t >> 1, q = t & 1;
        const int64_t l = __shfl_sync(FULL, kl.y, r);
        cp_async16(ws + r * RW + 4 + 4 * q, a.geo + 8 * l + 4 * q);
    }
#pragma unroll
    for (int m = 0; m < GC; ++m) {
        const int t = m * 32 + lane, r = t / GC, q = t - r * GC;
        const int64_t l = __shfl_sync(FULL, kl.y, r);
        cp_async16(ws + r * RW + 12 + 4 * q, rec + l * RS + 4 * g0 + 4 * q);
    }
#pragma unroll
    for (int m = 0; m < 3 * GC; ++m) {
        const int t = m * 32 + lane, r = t / (3 * GC), q = t - r * (3 * GC);
        const int64_t l = __shfl_sync(FULL, kl.y, r);
        cp_async16(ws + r * RW + 12 + 4 * GC + 4 * q, a.grad + l * 12 * G + 12 * g0 + 4 * q);
    }
    const float* tag = nullptr;
    const int64_t i = kl.x;
    const Pos<float> pi = load_pos(tag, a.pos, i);
    float gi8[8], gj8[8];
    vload<8>(a.geo + 8 * i, gi8);
    cp_async_wait_all();
    __syncwarp();
    const float* mine = ws + lane * RW;
    const uint4 pv = *reinterpret_cast<const uint4*>(mine);
    const Pos<float> pj = {pv.x, pv.y, pv.z};
    vload<8>(mine + 4, gj8);
    float dx, dy, dz;
    sep(a.sp, pi, pj, dx, dy, dz);
    PairGeo<float> pr;
    float sk, sl;
    pair_geo(dx, dy, dz, gi8, gj8, x.c, pr, sk, sl);
    const float* ri = rec + i * RS;
    const float* qi = a.grad + i * 12 * G;
    float out[NC];
    M1Top<float> top;
#pragma unroll
    for (int g = 0; g < GC; ++g) {
        const int gg = g0 + g;
        float ui[4], uj[4], gri[12], grj[12];
        vload<4>(ri + 4 * gg, ui);
        vload<4>(mine + 12 + 4 * g, uj);
        vload<12>(qi + 12 * gg, gri);
        vload<12>(mine + 12 + 4 * GC + 12 * g, grj);
        pair_flux<HLL, false>(ui, uj, gri, grj, pr, x.c, x.wave, &out[4 * g], top);
    }
    if (act) vstore<NC>(pairbuf + slot * NC, out);
    if (act && top.any)
        store_wide<HLL, GC>(ri + 4 * g0, rec + kl.y * (int64_t)RS + 4 * g0, qi + 12 * g0,
                            a.grad + kl.y * (int64_t)(12 * G) + 12 * g0, pr, x.c, x.wave, 1.f, pairbuf + slot * NC);
}

// Float pass 1 with the neighbour rows fetched by the tensor memory accelerator.  The
// gradient pass has packed each particle's flux inputs (position, geometry, state and
// gradient) into one row; each warp gathers the rows of its 32 l-particles into shared
// memory with eight tile::gather4 copies (four rows each).  The copies bypass the
// load/store pipeline whose wavefronts bound the direct kernel; the k side is loaded
// directly (mostly broadcasts).  Same arithmetic as k_flux.  A copy that does not complete
// within the wait budget sets err_flag, and the warp returns without storing.
template <int G>
struct PackedRows {
    static constexpr int RW = 12 + 16 * G;              // words per row
    static constexpr int SLOT = (4 * RW + 31) / 32 * 32; // four rows, padded to 128 bytes
    static constexpr int WF = 8 * SLOT;                 // floats per warp
    static constexpr uint32_t bytes = 32u * RW * 4u;    // bytes gathered per warp
};

// BINS: the pairs of the ordered prefix a.order[0, a.count) (time bins: those with a
// starting member), their fluxes scaled by 2^min(b_k, b_l) as in k_flux.
// One warp per block: each warp's shared rows are freed as soon as it finishes, instead of
// with the last warp of a four-warp block, and the register cap of 27 (24 for four groups)
// resident blocks per SM lets shared memory, not registers, bound the occupancy.  Measured
// against four-warp blocks at 80 registers: 0.169 against 0.180 ms per launch on the
// 262,144-particle set (G = 3), 1.78 against 1.93 ms on the 2,097,152-particle set (G = 4).
// Up to kTmaWarpsMax warps per block (rt_tuning's pair_warps, default 1); the register cap is
// that of 27 (24 at G = 4) one-warp blocks per SM whatever the block size
constexpr int kTmaWarpsMax = 4;
template <int G>
struct TmaMinBlocks {
    static constexpr int value = G >= 4 ? 6 : 7;   // blocks of kTmaWarpsMax warps
};
template <int G, bool HLL, bool BINS = false>
__global__ void __launch_bounds__(kTmaWarpsMax * 32, TmaMinBlocks<G>::value) k_flux_tma(PairArgs<float> a, FluxExtra<float> x,
                                                  float* __restrict__ pairbuf,
                                                  const __grid_constant__ CUtensorMap rows, int* err_flag,
                                                  unsigned long long budget) {
    using R = PackedRows<G>;
    constexpr int NC = 4 * G, RW = R::RW;
    // dynamic: R::WF floats per warp of the block plus 128 bytes, from which the rows start at
    // the first 128-byte boundary (the slots of the row gathers are 128-byte aligned)
    extern __shared__ __align__(128) float sm_dyn[];
    __shared__ __align__(8) uint64_t bar[kTmaWarpsMax];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t sm0 = smem_u32(sm_dyn);
    float* sm = sm_dyn + (((sm0 + 127u) & ~127u) - sm0) / 4u;
    float* ws = sm + wid * R::WF;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t np = BINS ? a.count : a.pairs();
    const bool act = t < np;
    if (t - lane >= np) return;       // a captured grid covers more slots than a build may have
    const int64_t slot = BINS ? (act ? (int64_t)a.order[t] : 0) : t;
    // lanes past the last slot gather particle 0 (always present) and store nothing
    const int2 kl = act ? a.ends[slot] : make_int2(0, 0);
    const uint32_t mb = smem_u32(&bar[wid]);
    if (lane == 0) {
        mbar_init(mb, 1);
        mbar_expect_tx(mb, R::bytes);
    }
    __syncwarp();
    const unsigned FULL = 0xffffffffu;
    const int q = lane & 7;
    const int r0 = __shfl_sync(FULL, kl.y, 4 * q), r1 = __shfl_sync(FULL, kl.y, 4 * q + 1);
    const int r2 = __shfl_sync(FULL, kl.y, 4 * q + 2), r3 = __shfl_sync(FULL, kl.y, 4 * q + 3);
    // even slots get the rows as they are (copy from word kRowRot), odd slots rotated by four
    // chunks (copy from word 0 of the prefixed row)
    if (lane < 8) tma_gather4(smem_u32(ws + q * R::SLOT), &rows, (q & 1) ? 0 : kRowRot, r0, r1, r2, r3, mb);
    const int64_t i = kl.x;
    const float* rk = packed_row(a, i);
    const uint4 pkv = *reinterpret_cast<const uint4*>(rk);
    const Pos<float> pi = {pkv.x, pkv.y, pkv.z};
    float gi8[8], gj8[8];
    vload<8>(rk + 4, gi8);
    if (!mbar_wait(mb, 0, budget)) {
        atomicExch(err_flag, 1);
        // let the copies still in flight land before the block exits, however short the
        // caller's budget (a copy lands in microseconds; this wait too is bounded)
        mbar_wait(mb, 0, budget > 2000000000ull ? budget : 2000000000ull);
        return;
    }
    // this lane's row: slot lane / 4, row lane % 4 within it.  A quarter-warp reads the rows
    // of one even and one odd slot; the slots start on the same bank, and the rows of a slot
    // cover four of the eight 16-byte bank groups at any one chunk, so the odd slot's rotation
    // by four chunks sends its lanes to the other four (all but the last four chunks).
    // Logical chunk c is at chunk c (even slot), c + 4 or, for the last four, c + 4 - RW / 4.
    const float* rl = ws + (lane >> 2) * R::SLOT + (lane & 3) * RW;
    const bool odd = (lane >> 2) & 1;
    const float* rlA = rl + (odd ? kRowRot : 0);
    const float* rlB = rl + (odd ? kRowRot - RW : 0);
    constexpr int NCH = RW / 4;
    auto lrow = [&](int c) -> const float* { return (c < NCH - kRowRot / 4 ? rlA : rlB) + 4 * c; };
    const uint4 pv = *reinterpret_cast<const uint4*>(lrow(0));
    const Pos<float> pj = {pv.x, pv.y, pv.z};
    vload<8>(lrow(1), gj8);
    float dx, dy, dz;
    sep(a.sp, pi, pj, dx, dy, dz);
    PairGeo<float> pr;
    float sk, sl;
    pair_geo(dx, dy, dz, gi8, gj8, x.c, pr, sk, sl);
    float out[NC];
    M1Top<float> top;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        float ui[4], uj[4], gri[12], grj[12];
        vload<4>(rk + 12 + 4 * g, ui);
        vload<4>(lrow(3 + g), uj);
        vload<12>(rk + 12 + 4 * G + 12 * g, gri);
        vload<4>(lrow(3 + G + 3 * g), grj);
        vload<4>(lrow(4 + G + 3 * g), grj + 4);
        vload<4>(lrow(5 + G + 3 * g), grj + 8);
        pair_flux<HLL, false>(ui, uj, gri, grj, pr, x.c, x.wave, &out[4 * g], top);
    }
    float wgt = 1.f;
    if constexpr (BINS) {
        wgt = (float)(1 << min(a.bins[kl.x], a.bins[kl.y]));   // min(dt_k, dt_l) / dt_min
#pragma unroll
        for (int c = 0; c < NC; ++c) out[c] *= wgt;
    }
    if (act) vstore<NC>(pairbuf + slot * NC, out);
    if (act && top.any) {
        const float* rg = packed_row(a, (int64_t)kl.y);
        store_wide<HLL, G>(rk + 12, rg + 12, rk + 12 + 4 * G, rg + 12 + 4 * G, pr, x.c, x.wave, wgt, pairbuf + slot * NC);
    }
}

// The same pair pass for the HLL solver, with the wave-speed table (81,608 bytes) in shared memory: one
// block per SM, as many warps as rows fit beside the table, each walking batches of 32 slots.
// A batch's 32 lanes read 32 scattered nodes of the table in each of its 8 lookups a group:
// from L1 that is a wavefront a line and the kernel's bound (0.251 ms on 131,071 particles and
// three groups), from shared memory a few bank conflicts.
template <int G>
struct HllShape {
    static constexpr int table = RT_WAVE_NF * RT_WAVE_NTH * 8;
    static constexpr int warps = (226 * 1024 - 512 - table) / (PackedRows<G>::WF * 4) < 20
                                     ? (226 * 1024 - 512 - table) / (PackedRows<G>::WF * 4)
                                     : 20;
    static constexpr int smem = 128 + warps * PackedRows<G>::WF * 4 + table;
};
template <int G>
__global__ void __launch_bounds__(HllShape<G>::warps * 32, 1)
k_flux_hll(PairArgs<float> a, FluxExtra<float> x, float* __restrict__ pairbuf,
           const __grid_constant__ CUtensorMap rows, int* err_flag, unsigned long long budget) {
    using R = PackedRows<G>;
    constexpr int NC = 4 * G, RW = R::RW;
    extern __shared__ __align__(128) float sm_dyn[];
    __shared__ __align__(8) uint64_t bar[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t sm0 = smem_u32(sm_dyn);
    float* sm = sm_dyn + (((sm0 + 127u) & ~127u) - sm0) / 4u;
    float* ws = sm + wid * R::WF;
    const float2* tab = reinterpret_cast<const float2*>(sm + (blockDim.x >> 5) * R::WF);
    for (int k = threadIdx.x; k < RT_WAVE_NF * RT_WAVE_NTH; k += blockDim.x)
        const_cast<float2*>(tab)[k] = reinterpret_cast<const float2*>(x.wave)[k];
    const unsigned FULL = 0xffffffffu;
    const uint32_t mb = smem_u32(&bar[wid]);
    if (lane == 0) mbar_init(mb, 1);
    __syncthreads();
    const int64_t np = a.pairs(), stride = gridDim.x * (int64_t)blockDim.x;
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    // lanes past the last slot gather particle 0 (always present) and store nothing
    int2 kl = t < np ? a.ends[t] : make_int2(0, 0);
    for (uint32_t parity = 0; t - lane < np; parity ^= 1) {
        if (lane == 0) mbar_expect_tx(mb, R::bytes);
        __syncwarp();
        const int q = lane & 7;
        const int r0 = __shfl_sync(FULL, kl.y, 4 * q), r1 = __shfl_sync(FULL, kl.y, 4 * q + 1);
        const int r2 = __shfl_sync(FULL, kl.y, 4 * q + 2), r3 = __shfl_sync(FULL, kl.y, 4 * q + 3);
        // even slots get the rows as they are (copy from word kRowRot), odd slots rotated by four
        // chunks (copy from word 0 of the prefixed row)
        if (lane < 8) tma_gather4(smem_u32(ws + q * R::SLOT), &rows, (q & 1) ? 0 : kRowRot, r0, r1, r2, r3, mb);
        // the next batch's ends, under this batch's copies and arithmetic
        const int64_t slot = t;
        t += stride;
        const int2 kl_next = t < np ? a.ends[t] : make_int2(0, 0);
        const float* rk = packed_row(a, (int64_t)kl.x);
        const uint4 pkv = *reinterpret_cast<const uint4*>(rk);
        const Pos<float> pi = {pkv.x, pkv.y, pkv.z};
        float gi8[8], gj8[8];
        vload<8>(rk + 4, gi8);
        if (!mbar_wait(mb, parity, budget)) {
            atomicExch(err_flag, 1);
            // let the copies still in flight land before the block exits, however short the
            // caller's budget (a copy lands in microseconds; this wait too is bounded)
            mbar_wait(mb, parity, budget > 2000000000ull ? budget : 2000000000ull);
            return;
        }
        // this lane's row: slot lane / 4, row lane % 4 within it.  A quarter-warp reads the rows
        // of one even and one odd slot; the slots start on the same bank, and the rows of a slot
        // cover four of the eight 16-byte bank groups at any one chunk, so the odd slot's rotation
        // by four chunks sends its lanes to the other four (all but the last four chunks).
        // Logical chunk c is at chunk c (even slot), c + 4 or, for the last four, c + 4 - RW / 4.
        const float* rl = ws + (lane >> 2) * R::SLOT + (lane & 3) * RW;
        const bool odd = (lane >> 2) & 1;
        const float* rlA = rl + (odd ? kRowRot : 0);
        const float* rlB = rl + (odd ? kRowRot - RW : 0);
        constexpr int NCH = RW / 4;
        auto lrow = [&](int c) -> const float* { return (c < NCH - kRowRot / 4 ? rlA : rlB) + 4 * c; };
        const uint4 pv = *reinterpret_cast<const uint4*>(lrow(0));
        const Pos<float> pj = {pv.x, pv.y, pv.z};
        vload<8>(lrow(1), gj8);
        float dx, dy, dz;
        sep(a.sp, pi, pj, dx, dy, dz);
        PairGeo<float> pr;
        float sk, sl;
        pair_geo(dx, dy, dz, gi8, gj8, x.c, pr, sk, sl);
        float out[NC];
        M1Top<float> top;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            float ui[4], uj[4], gri[12], grj[12];
            vload<4>(rk + 12 + 4 * g, ui);
            vload<4>(lrow(3 + g), uj);
            vload<12>(rk + 12 + 4 * G + 12 * g, gri);
            vload<4>(lrow(3 + G + 3 * g), grj);
            vload<4>(lrow(4 + G + 3 * g), grj + 4);
            vload<4>(lrow(5 + G + 3 * g), grj + 8);
            pair_flux<true, false>(ui, uj, gri, grj, pr, x.c, reinterpret_cast<const float*>(tab), &out[4 * g], top);
        }
        if (slot < np) vstore<NC>(pairbuf + slot * NC, out);
        if (slot < np && top.any) {
            const float* rg = packed_row(a, (int64_t)kl.y);
            store_wide<true, G>(rk + 12, rg + 12, rk + 12 + 4 * G, rg + 12 + 4 * G, pr, x.c, x.wave, 1.f,
                                pairbuf + slot * NC);
        }
        kl = kl_next;
        __syncwarp();      // every lane has read its row before the next copies overwrite it
    }
}

// Float pass 2 with one thread per (particle, group): the lanes of one particle read the
// 16-byte pieces of a slot that lie side by side, so a warp request touches about 32 / GC
// slots instead of 32.  Same order of additions and subtractions as k_flux_gather.
// B loads in flight a thread: eight, or (WIDE) 24, a whole half row, with the lower slots' indices
// loaded beside the upper slots: for sets too small to fill the GPU, where the launch is the
// latency of one thread's chain of loads (4,096 particles, one group: 14.4 us with eight).
template <class T, int GC, bool WIDE = false>
__global__ void __launch_bounds__(WIDE ? 64 : kGatherBlockMax) k_flux_gather_g(PairArgs<T> a, FluxExtra<T> x,
                                                       const T* __restrict__ rec,
                                                       const T* __restrict__ pairbuf, T* __restrict__ out,
                                                       int g0) {
    constexpr int B = (WIDE ? 24 : 8) * 4 / (int)sizeof(T);
    // blocks run from the last particles to the first: the pair pass wrote the slots in
    // ascending order, so the most recent (still L2-resident) slots are read first
    const int64_t t = (gridDim.x - 1 - blockIdx.x) * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = t / GC;
    if (i >= a.n) return;
    const int g = (int)(t - i * GC);
    constexpr int NC = 4 * GC;
    const int RS = 4 * a.G;
    const T* pb = pairbuf + 4 * g;
    FluxAcc<T> acc;
    acc.zero();
    const int64_t r0 = a.row_off[i], s0 = a.up_off[i], s1 = a.up_off[i + 1];
    const int nl = a.n_low[i];
    const int32_t* ls = a.low_slot + (r0 - s0);
    int32_t q[B];
    if constexpr (WIDE) {
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (u < nl) q[u] = ls[u];
    }
    // batches of up to B loads in flight (the last one predicated), added in order
    for (int64_t sl = s0; sl < s1; sl += B) {
        const int m = s1 - sl < B ? (int)(s1 - sl) : B;
        T p[B][4];
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (u < m) vload<4>(pb + (sl + u) * NC, p[u]);
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (u < m) acc.add(p[u]);
    }
    for (int e = 0; e < nl; e += B) {   // up to B slot indices, then their loads in flight
        const int m = nl - e < B ? nl - e : B;
        if (!WIDE || e > 0) {
#pragma unroll
            for (int u = 0; u < B; ++u)
                if (u < m) q[u] = ls[e + u];
        }
        T p[B][4];
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (u < m) vload<4>(pb + (int64_t)q[u] * NC, p[u]);
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (u < m) acc.sub(p[u]);
    }
    const T dt = (T)(*x.dt_dev);
    const T f = dt * a.omega[i];
    T sink = T(1);
    if (x.alpha) sink = fmax_(T(1) - x.c * x.alpha[i] * dt, T(0));
    if (x.alpha_g) sink = fmax_(T(1) - x.c * x.alpha_g[i * a.G + g0 + g] * dt, T(0));
    T ui[4];
    const int64_t o = i * RS + 4 * (g0 + g);
    vload<4>(rec + o, ui);
    const int nclamp = update_group<T>(ui, acc, f, sink, x.clamp, x.inj ? x.inj + i * a.G + g0 + g : nullptr);
    vstore<4>(out + o, ui);
    if (nclamp) atomicAdd(x.clamp_count, (unsigned long long)nclamp);
}

// ------------------------------------------------------------------------------------
// Drift correction (Sec. "Dealing With Particle Drifts"): U_i += grad U_i . (v_i dt_drift)
// for every component, on the sorted records; v in caller order (SoA doubles).
template <class T>
__global__ void k_drift(T* __restrict__ rec, const T* __restrict__ grad, const double* __restrict__ v,
                        const int32_t* __restrict__ perm, int64_t n, int G, double dt) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int64_t i = perm[p];
    const T dx = (T)(v[i] * dt), dy = (T)(v[n + i] * dt), dz = (T)(v[2 * n + i] * dt);
    T* u = rec + p * 4 * G;
    const T* g = grad + p * 12 * G;
    for (int c = 0; c < 4 * G; ++c) u[c] += g[3 * c] * dx + g[3 * c + 1] * dy + g[3 * c + 2] * dz;
}

rt_status launch_drift(rt_ctx* c, cudaStream_t s, void* rec, const double* v, double dt) {
    unsigned nb = nblk(c->n, 256);
    if (c->fp64)
        k_drift<double><<<nb, 256, 0, s>>>((double*)rec, c->grad_t.as<double>(), v, c->perm.as<int32_t>(), c->n,
                                           c->cfg.n_groups, dt);
    else
        k_drift<float><<<nb, 256, 0, s>>>((float*)rec, c->grad_t.as<float>(), v, c->perm.as<int32_t>(), c->n,
                                          c->cfg.n_groups, dt);
    ++c->launches;
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

// ------------------------------------------------------------------------------------
// a10: energy per group, sum_i V_i E_i,g in double; fixed grid and tree order.
constexpr int kEnergyBlocks = 512;

// Reads the caller's state, particles [0, owned) (the ghost copies of a domain decomposition come
// after them); V is in sorted order.
template <class T>
__global__ void __launch_bounds__(256)
k_energy_part(const T* __restrict__ U, const double* __restrict__ V, int64_t n, int G,
              const int32_t* __restrict__ inv_perm, int64_t owned, double* __restrict__ part) {
    __shared__ double sm[256];
    for (int g0 = 0; g0 < G; g0 += kMaxGC) {
        double s[kMaxGC] = {0.0, 0.0, 0.0, 0.0};
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < owned;
             i += (int64_t)gridDim.x * blockDim.x) {
            const double v = V[inv_perm[i]];
#pragma unroll
            for (int g = 0; g < kMaxGC; ++g)
                if (g0 + g < G) s[g] += v * (double)U[(int64_t)4 * (g0 + g) * n + i];
        }
        for (int g = 0; g < kMaxGC && g0 + g < G; ++g) {
            sm[threadIdx.x] = s[g];
            __syncthreads();
            for (int w = blockDim.x / 2; w > 0; w >>= 1) {
                if (threadIdx.x < w) sm[threadIdx.x] += sm[threadIdx.x + w];
                __syncthreads();
            }
            if (threadIdx.x == 0) part[(g0 + g) * gridDim.x + blockIdx.x] = sm[0];
            __syncthreads();
        }
    }
}

// one block of kEnergyBlocks threads per group adds the partial sums in a fixed tree: 4 us where
// one thread adding the 512 in turn took 34
__global__ void __launch_bounds__(kEnergyBlocks) k_energy_final(const double* __restrict__ part, double* out) {
    __shared__ double sm[kEnergyBlocks];
    const int g = blockIdx.x, t = threadIdx.x;
    sm[t] = part[g * kEnergyBlocks + t];
    __syncthreads();
    for (int w = kEnergyBlocks / 2; w > 0; w >>= 1) {
        if (t < w) sm[t] += sm[t + w];
        __syncthreads();
    }
    if (t == 0) out[g] = sm[0];
}

// ------------------------------------------------------------------------------------
// the pair kernels use no shared memory: give the whole unified L1 to the cache
template <class T>
static void set_carveouts() {
    static bool done = false;
    if (done) return;
    done = true;
    const void* fs[] = {(const void*)k_gradient<T, 1>, (const void*)k_gradient<T, 2>, (const void*)k_gradient<T, 3>,
                        (const void*)k_gradient<T, 4>, (const void*)k_flux<T, 1, false>,
                        (const void*)k_flux<T, 2, false>, (const void*)k_flux<T, 3, false>,
                        (const void*)k_flux<T, 4, false>, (const void*)k_flux<T, 1, true>,
                        (const void*)k_flux<T, 2, true>, (const void*)k_flux<T, 3, true>,
                        (const void*)k_flux<T, 4, true>};
    for (const void* f : fs) cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
    if constexpr (std::is_same<T, float>::value) {
        const void* gs[] = {(const void*)k_flux_gather<T, 1>, (const void*)k_flux_gather<T, 2>,
                            (const void*)k_flux_gather<T, 3>, (const void*)k_flux_gather<T, 4>};
        for (const void* f : gs) cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
    }
    (void)cudaGetLastError();
}

template <class T>
static void launch_gradient_t(rt_ctx* c, cudaStream_t s, T* rec, bool packed = false, int only = -1) {
    set_carveouts<T>();
    PairArgs<T> a = pair_args<T>(c);
    const int G = c->cfg.n_groups;
    unsigned nb = nblk(c->n, 128);
    for (int g0 = 0; g0 < G; g0 += chunk_groups(G)) {
        if (only >= 0 && g0 != only) continue;
        int gc = G - g0 < chunk_groups(G) ? G - g0 : chunk_groups(G);
        if (packed) {
            a.frec = c->frec.as<T>();
            a.RW = 12 + 16 * gc;
        }
        int pr = prof_begin(c, s, RT_KERNEL_GRADIENT);
        if constexpr (std::is_same<T, float>::value) {
            if (few_threads(c, gc)) {
                float* gr = c->grad_t.as<float>();
                const unsigned nbw = nblk(c->n * gc, 64);
                switch (gc) {
                    case 1: k_gradient_w<1><<<nbw, 64, 0, s>>>(a, rec, gr, g0); break;
                    case 2: k_gradient_w<2><<<nbw, 64, 0, s>>>(a, rec, gr, g0); break;
                    case 3: k_gradient_w<3><<<nbw, 64, 0, s>>>(a, rec, gr, g0); break;
                    default: k_gradient_w<4><<<nbw, 64, 0, s>>>(a, rec, gr, g0); break;
                }
                prof_end(c, s, pr);
                ++c->launches;
                continue;
            }
            if (c->tune.gradient_variant == 2 && gc > 1) {
                // warps of 32 / gc particles: ceil(n / (32 / gc)) warps of 32 lanes
                const int64_t warps = (c->n + 32 / gc - 1) / (32 / gc);
                const int gb = grad_block(c);
                unsigned nbs = nblk(warps * 32, gb);
                float* gr = c->grad_t.as<float>();
                switch (gc) {
                    case 2: k_gradient_s<2><<<nbs, gb, 0, s>>>(a, rec, gr, g0); break;
                    case 3: k_gradient_s<3><<<nbs, gb, 0, s>>>(a, rec, gr, g0); break;
                    default: k_gradient_s<4><<<nbs, gb, 0, s>>>(a, rec, gr, g0); break;
                }
                prof_end(c, s, pr);
                ++c->launches;
                continue;
            }
            if (c->tune.gradient_variant >= 1) {
                const int gb = c->tune.gradient_block > 0 ? c->tune.gradient_block : 256;
                unsigned nbg = nblk(c->n * gc, gb);
                float* gr = c->grad_t.as<float>();
                switch (gc) {
                    case 1: k_gradient_g<1><<<nbg, gb, 0, s>>>(a, rec, gr, g0); break;
                    case 2: k_gradient_g<2><<<nbg, gb, 0, s>>>(a, rec, gr, g0); break;
                    case 3: k_gradient_g<3><<<nbg, gb, 0, s>>>(a, rec, gr, g0); break;
                    default: k_gradient_g<4><<<nbg, gb, 0, s>>>(a, rec, gr, g0); break;
                }
                prof_end(c, s, pr);
                ++c->launches;
                continue;
            }
        }
        if constexpr (std::is_same<T, double>::value) {
            if (a.wd) {
                switch (gc) {
                    case 1: launch_gradient_wd<1, false>(c, s, a, rec, c->grad_t.as<T>(), g0); break;
                    case 2: launch_gradient_wd<2, false>(c, s, a, rec, c->grad_t.as<T>(), g0); break;
                    case 3: launch_gradient_wd<3, false>(c, s, a, rec, c->grad_t.as<T>(), g0); break;
                    default: launch_gradient_wd<4, false>(c, s, a, rec, c->grad_t.as<T>(), g0); break;
                }
                prof_end(c, s, pr);
                ++c->launches;
                continue;
            }
        }
        switch (gc) {
            case 1: k_gradient<T, 1><<<nb, 128, 0, s>>>(a, rec, c->grad_t.as<T>(), g0); break;
            case 2: k_gradient<T, 2><<<nb, 128, 0, s>>>(a, rec, c->grad_t.as<T>(), g0); break;
            case 3: k_gradient<T, 3><<<nb, 128, 0, s>>>(a, rec, c->grad_t.as<T>(), g0); break;
            default: k_gradient<T, 4><<<nb, 128, 0, s>>>(a, rec, c->grad_t.as<T>(), g0); break;
        }
        prof_end(c, s, pr);
        ++c->launches;
    }
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link-time libcuda)
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        (void)cudaGetLastError();
    }
    return fn;
}

// tensor map of the packed rows [n][kRowRot + 12 + 16 gc] floats of a chunk of gc groups, box of
// the 12 + 16 gc logical words of a row (for tile::gather4); encoded again whenever the buffer or
// its shape changes
static bool packed_rows_map(rt_ctx* c, int gc) {
    const int RW = 12 + 16 * gc;
    if (c->rows_map_for[gc] == c->frec.p && c->rows_map_n[gc] == c->n) return true;
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc || !c->frec.p) return false;
    // rows of kRowRot + RW words (the prefix first); the box is the RW logical words
    cuuint64_t dims[2] = {(cuuint64_t)(RW + kRowRot), (cuuint64_t)c->n};
    cuuint64_t strides[1] = {(cuuint64_t)(RW + kRowRot) * 4};
    cuuint32_t box[2] = {(cuuint32_t)RW, 1};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(&c->rows_map[gc], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, c->frec.p, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return false;
    c->rows_map_for[gc] = c->frec.p;
    c->rows_map_n[gc] = c->n;
    return true;
}

// whether the float pair pass fetches packed rows: its variant, and tensor maps for the chunks
static bool packed_rows(rt_ctx* c) {
    const int G = c->cfg.n_groups, cs = chunk_groups(G);
    if (c->fp64 || c->tune.flux_variant != 2) return false;
    for (int g0 = 0; g0 < G; g0 += cs)
        if (!packed_rows_map(c, G - g0 < cs ? G - g0 : cs)) return false;
    return true;
}

// whether k_flux_hll<GC>, which needs more shared memory than a launch gets unasked, may run on the
// context's device.  The permission belongs to the function on one device: each context asks
// for its own, once, and a refusal leaves k_flux_tma
template <int GC>
static bool hll_table_in_smem(rt_ctx* c) {
    if (c->hll_smem[GC] == 0) {
        const cudaError_t e = cudaFuncSetAttribute((const void*)k_flux_hll<GC>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, HllShape<GC>::smem);
        if (e != cudaSuccess) (void)cudaGetLastError();
        c->hll_smem[GC] = e == cudaSuccess ? 1 : -1;
    }
    return c->hll_smem[GC] > 0;
}

// float pass 1 and 2 in the variants chosen by the context's tuning
template <int GC, bool HLL>
static void flux_float(rt_ctx* c, cudaStream_t s, const PairArgs<float>& a, const FluxExtra<float>& x,
                       const float* rec, float* pb, float* out, int g0) {
    static bool attr = false;
    if (!attr) {
        attr = true;
        cudaFuncSetAttribute((const void*)k_flux_staged<GC, HLL>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
        cudaFuncSetAttribute((const void*)k_flux_gather_g<float, GC>, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
        cudaFuncSetAttribute((const void*)k_flux_tma<GC, HLL>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
        (void)cudaGetLastError();
    }
    unsigned npb = nblk(std::max<int64_t>(a.n_pairs, 1), 128);
    int variant = c->tune.flux_variant;
    if (variant == 2 && !a.frec) variant = 0;
    int pr = prof_begin(c, s, RT_KERNEL_FLUX);
    if (variant == 2) {
        unsigned long long budget = c->cfg.device_wait_budget_cycles ? c->cfg.device_wait_budget_cycles
                                                                     : 4000000000ull;
        const int pw = pair_warps(c);
        int* ef = c->flags.as<int>() + F_TIMEOUT;
        // HLL: with two batches a warp or more, the table in shared memory is worth loading
        if (HLL && a.n_pairs >= (int64_t)c->sm_count * HllShape<GC>::warps * 64 && hll_table_in_smem<GC>(c))
            k_flux_hll<GC><<<c->sm_count, HllShape<GC>::warps * 32, HllShape<GC>::smem, s>>>(
                a, x, pb, c->rows_map[GC], ef, budget);
        else
            k_flux_tma<GC, HLL><<<nblk(std::max<int64_t>(a.n_pairs, 1), pw * 32), pw * 32,
                                  (size_t)pw * PackedRows<GC>::WF * sizeof(float) + 128, s>>>(
                a, x, pb, c->rows_map[GC], ef, budget);
    } else if (variant == 1) {
        k_flux_staged<GC, HLL><<<npb, 128, 0, s>>>(a, x, rec, pb, g0);
    } else {
        k_flux<float, GC, HLL><<<npb, 128, 0, s>>>(a, x, rec, pb, g0);
    }
    prof_end(c, s, pr);
    pr = prof_begin(c, s, RT_KERNEL_FLUX_GATHER);
    if (c->tune.gather_variant == 1 && few_threads(c, GC))
        k_flux_gather_g<float, GC, true><<<nblk(c->n * GC, 64), 64, 0, s>>>(a, x, rec, pb, out, g0);
    else if (c->tune.gather_variant == 1)
        k_flux_gather_g<float, GC><<<nblk(c->n * GC, gather_block(c)), gather_block(c), 0, s>>>(a, x, rec, pb, out, g0);
    else
        k_flux_gather<float, GC><<<nblk(c->n, 128), 128, 0, s>>>(a, x, rec, pb, out, g0);
    prof_end(c, s, pr);
    c->launches += 2;
}

template <class T>
static void launch_flux_t(rt_ctx* c, cudaStream_t s, const T* rec, T* out, bool has_alpha, bool packed = false,
                          bool inject_after = false, int only = -1) {
    PairArgs<T> a = pair_args<T>(c);
    FluxExtra<T> x;
    const bool hll = c->cfg.riemann_solver == RT_RIEMANN_HLL;
    x.wave = hll ? c->wave_t.as<T>() : nullptr;
    x.alpha = has_alpha ? c->alpha_s.as<T>() : nullptr;
    x.alpha_g = c->step_alpha_g ? c->alpha_g_s.as<T>() : nullptr;
    x.acc = nullptr;
    x.inj = inject_after ? c->inj_dense.as<double>() : nullptr;
    x.dt_dev = c->dt_dev.as<double>();
    x.c = (T)c->cfg.c_red;
    x.clamp = c->cfg.clamp_negative;
    x.clamp_count = reinterpret_cast<unsigned long long*>(c->flags.as<int>() + F_CLAMP);
    const int G = c->cfg.n_groups;
    unsigned nb = nblk(c->n, 128);
    T* pb = c->pairbuf.as<T>();
    unsigned npb = nblk(std::max<int64_t>(a.n_pairs, 1), 128);
    for (int g0 = 0; g0 < G; g0 += chunk_groups(G)) {
        if (only >= 0 && g0 != only) continue;
        int gc = G - g0 < chunk_groups(G) ? G - g0 : chunk_groups(G);
        if (packed) {
            a.frec = c->frec.as<T>();
            a.RW = 12 + 16 * gc;
        }
        if constexpr (std::is_same<T, float>::value) {
            if (hll) {
                switch (gc) {
                    case 1: flux_float<1, true>(c, s, a, x, rec, pb, out, g0); break;
                    case 2: flux_float<2, true>(c, s, a, x, rec, pb, out, g0); break;
                    case 3: flux_float<3, true>(c, s, a, x, rec, pb, out, g0); break;
                    default: flux_float<4, true>(c, s, a, x, rec, pb, out, g0); break;
                }
            } else {
                switch (gc) {
                    case 1: flux_float<1, false>(c, s, a, x, rec, pb, out, g0); break;
                    case 2: flux_float<2, false>(c, s, a, x, rec, pb, out, g0); break;
                    case 3: flux_float<3, false>(c, s, a, x, rec, pb, out, g0); break;
                    default: flux_float<4, false>(c, s, a, x, rec, pb, out, g0); break;
                }
            }
            continue;
        }
        int pr = prof_begin(c, s, RT_KERNEL_FLUX);
        if (hll) {
            switch (gc) {
                case 1: k_flux<T, 1, true><<<npb, 128, 0, s>>>(a, x, rec, pb, g0); break;
                case 2: k_flux<T, 2, true><<<npb, 128, 0, s>>>(a, x, rec, pb, g0); break;
                case 3: k_flux<T, 3, true><<<npb, 128, 0, s>>>(a, x, rec, pb, g0); break;
                default: k_flux<T, 4, true><<<npb, 128, 0, s>>>(a, x, rec, pb, g0); break;
            }
        } else {
            switch (gc) {
                case 1: k_flux<T, 1, false><<<npb, 128, 0, s>>>(a, x, rec, pb, g0); break;
                case 2: k_flux<T, 2, false><<<npb, 128, 0, s>>>(a, x, rec, pb, g0); break;
                case 3: k_flux<T, 3, false><<<npb, 128, 0, s>>>(a, x, rec, pb, g0); break;
                default: k_flux<T, 4, false><<<npb, 128, 0, s>>>(a, x, rec, pb, g0); break;
            }
        }
        prof_end(c, s, pr);
        pr = prof_begin(c, s, RT_KERNEL_FLUX_GATHER);
        const unsigned nbg = nblk(c->n * gc, 128);
        switch (gc) {
            case 1: k_flux_gather_g<T, 1><<<nbg, 128, 0, s>>>(a, x, rec, pb, out, g0); break;
            case 2: k_flux_gather_g<T, 2><<<nbg, 128, 0, s>>>(a, x, rec, pb, out, g0); break;
            case 3: k_flux_gather_g<T, 3><<<nbg, 128, 0, s>>>(a, x, rec, pb, out, g0); break;
            default: k_flux_gather_g<T, 4><<<nbg, 128, 0, s>>>(a, x, rec, pb, out, g0); break;
        }
        prof_end(c, s, pr);
        c->launches += 2;
    }
}

template <class T>
static void launch_inject_t(rt_ctx* c, cudaStream_t s, T* rec, const int8_t* bins = nullptr, int step = 0) {
    if (c->n_inj_targets <= 0) return;
    int pr = prof_begin(c, s, RT_KERNEL_INJECT);
    k_inject<T><<<nblk(c->capturing ? c->target_cap : c->n_inj_targets, 128), 128, 0, s>>>(
        c->inj_targets.as<int32_t>(), c->inj_off.as<int32_t>(), c->inj_src.as<int32_t>(), c->inj_coef.as<double>(),
        c->L_dev.as<double>(), c->cfg.n_groups, c->dt_dev.as<double>(), 4 * c->cfg.n_groups, rec, bins, step);
    prof_end(c, s, pr);
    ++c->launches;
}

rt_status launch_inject(rt_ctx* c, cudaStream_t s, void* rec) {
    if (c->fp64) launch_inject_t<double>(c, s, (double*)rec);
    else launch_inject_t<float>(c, s, (float*)rec);
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

rt_status launch_gradient(rt_ctx* c, cudaStream_t s, void* rec) {
    if (c->fp64) launch_gradient_t<double>(c, s, (double*)rec);
    else launch_gradient_t<float>(c, s, (float*)rec);
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

// packed flux rows of the groups [g0, g0 + gc) from sorted states and gradients given in grad_t
// (one thread per particle and group): what the gradient kernels write beside their gradients
__global__ void k_pack_rows(PairArgs<float> a, const float* __restrict__ rec, const float* __restrict__ grad, int g0,
                            int gc) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = t / gc;
    if (i >= a.n) return;
    const int g = (int)(t - i * gc);
    float* row = packed_row(a, i);
    float gq[12], u[4];
    vload<12>(grad + i * 12 * a.G + 12 * (g0 + g), gq);
    vload<4>(rec + i * 4 * a.G + 4 * (g0 + g), u);
    row_store<12>(a, row, 12 + 4 * gc + 12 * g, gq);
    row_store<4>(a, row, 12 + 4 * g, u);
    if (g == 0) packed_static(a, i, row);
}

rt_status launch_flux_given(rt_ctx* c, cudaStream_t s, void* Uin, void* Uout, bool has_alpha) {
    if (c->fp64) {
        launch_flux_t<double>(c, s, (const double*)Uin, (double*)Uout, has_alpha);
    } else {
        const int G = c->cfg.n_groups, cs = chunk_groups(G);
        if (!packed_rows(c)) {
            launch_flux_t<float>(c, s, (const float*)Uin, (float*)Uout, has_alpha);
        } else {
            for (int g0 = 0; g0 < G; g0 += cs) {
                const int gc = G - g0 < cs ? G - g0 : cs;
                PairArgs<float> a = pair_args<float>(c);
                a.frec = c->frec.as<float>();
                a.RW = 12 + 16 * gc;
                k_pack_rows<<<nblk(c->n * gc, 256), 256, 0, s>>>(a, (const float*)Uin, c->grad_t.as<float>(), g0, gc);
                ++c->launches;
                launch_flux_t<float>(c, s, (const float*)Uin, (float*)Uout, has_alpha, true, false, g0);
            }
        }
    }
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

// omega, V = 1 / omega and B of caller particles [first, first + count) from the caller
// (omega [count], B [count][3][3], double), with the pair kernels' records derived from them
// as k_geometry derives its own
template <class T>
__global__ void k_set_fields(const double* __restrict__ omega, const double* __restrict__ B9,
                             const int32_t* __restrict__ inv_perm, int64_t first, int64_t count, int64_t n,
                             const double* __restrict__ h, double* omega_d, double* V_d, double* B_d, T* geo_t,
                             T* om_t) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= count) return;
    const int64_t p = inv_perm[first + k];
    const double om = omega[k];
    const double* b = B9 + 9 * k;
    const double B[6] = {b[0], b[4], b[8], b[1], b[2], b[5]};   // xx yy zz xy xz yz
    const double hi = h[p], H = kKappa * hi, iH = 1.0 / H;
    const double V = 1.0 / om;
    const double bp = V * V * kSigma * iH * iH * iH;
    omega_d[p] = om;
    V_d[p] = V;
    geo_t[8 * p] = (T)iH;
    geo_t[8 * p + 1] = (T)hi;
    for (int e = 0; e < 6; ++e) {
        B_d[e * n + p] = B[e];
        geo_t[8 * p + 2 + e] = (T)(bp * B[e]);
    }
    om_t[p] = (T)om;
}

rt_status set_fields(rt_ctx* c, int64_t first, int64_t count, const double* omega, const double* B) {
    if (count <= 0) return RT_OK;
    const unsigned nb = nblk(count, 128);
    if (c->fp64)
        k_set_fields<double><<<nb, 128, 0, c->stream>>>(omega, B, c->inv_perm.as<int32_t>(), first, count, c->n,
                                                        c->h_d.as<double>(), c->omega_d.as<double>(),
                                                        c->V_d.as<double>(), c->B_d.as<double>(),
                                                        c->geo_t.as<double>(), c->omega_t.as<double>());
    else
        k_set_fields<float><<<nb, 128, 0, c->stream>>>(omega, B, c->inv_perm.as<int32_t>(), first, count, c->n,
                                                       c->h_d.as<double>(), c->omega_d.as<double>(),
                                                       c->V_d.as<double>(), c->B_d.as<double>(),
                                                       c->geo_t.as<float>(), c->omega_t.as<float>());
    ++c->launches;
    RT_CUDA(c, cudaGetLastError());
    c->pair_geo_ready = false;   // B changed: the kept surfaces are computed again
    return RT_OK;
}

// one min-step of a hydro step with individual time bins, on the active sets only: the
// injection and gradients of the starting particles, the pair fluxes of the pairs with a
// starting member, the gather of the particles they touch (finalising those whose step ends
// now), and the finalisation of the other particles whose step ends now.  In place.
// the time-bin pair pass by row gathers (float, one group chunk); other T: never called
template <int GC, class T>
static void bins_flux_tma(rt_ctx* c, cudaStream_t s, const PairArgs<T>& af, const FluxExtra<T>& x, T* pb, bool hll) {
    if constexpr (std::is_same<T, float>::value) {
        static bool attr = false;
        if (!attr) {
            attr = true;
            cudaFuncSetAttribute((const void*)k_flux_tma<GC, false, true>,
                                 cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
            cudaFuncSetAttribute((const void*)k_flux_tma<GC, true, true>,
                                 cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
            (void)cudaGetLastError();
        }
        const unsigned long long budget = c->cfg.device_wait_budget_cycles ? c->cfg.device_wait_budget_cycles
                                                                           : 4000000000ull;
        int* ef = c->flags.as<int>() + F_TIMEOUT;
        const int pw = pair_warps(c);
        const size_t smem = (size_t)pw * PackedRows<GC>::WF * sizeof(float) + 128;
        const unsigned nbt = nblk(std::max<int64_t>(af.count, 1), pw * 32);
        if (hll) k_flux_tma<GC, true, true><<<nbt, pw * 32, smem, s>>>(af, x, pb, c->rows_map[GC], ef, budget);
        else k_flux_tma<GC, false, true><<<nbt, pw * 32, smem, s>>>(af, x, pb, c->rows_map[GC], ef, budget);
    }
}

template <class T>
static void launch_step_bins_t(rt_ctx* c, cudaStream_t s, int step, T* rec, bool has_src, bool has_alpha) {
    set_carveouts<T>();
    const int8_t* bins = c->bins_s.as<int8_t>();
    if (has_src) launch_inject_t<T>(c, s, rec, bins, step);
    const int B = c->bins_max;
    const int tz = step == 0 ? B : __builtin_ctz((unsigned)step);
    const int tz1 = __builtin_ctz((unsigned)(step + 1)) < B ? __builtin_ctz((unsigned)(step + 1)) : B;
    PairArgs<T> a = pair_args<T>(c);
    a.bins = bins;
    a.s = step;
    a.nmin = c->bins_nmin.as<int8_t>();
    a.tz = tz;
    FluxExtra<T> x;
    const bool hll = c->cfg.riemann_solver == RT_RIEMANN_HLL;
    x.wave = hll ? c->wave_t.as<T>() : nullptr;
    x.alpha = has_alpha ? c->alpha_s.as<T>() : nullptr;
    x.alpha_g = c->step_alpha_g ? c->alpha_g_s.as<T>() : nullptr;
    x.acc = c->acc_t.as<T>();
    x.inj = nullptr;
    x.dt_dev = c->dt_dev.as<double>();
    x.c = (T)c->cfg.c_red;
    x.clamp = c->cfg.clamp_negative;
    x.clamp_count = reinterpret_cast<unsigned long long*>(c->flags.as<int>() + F_CLAMP);
    const int G = c->cfg.n_groups;
    T* pb = c->pairbuf.as<T>();
    T* gr = c->grad_t.as<T>();
    const int64_t n_start = c->cum_b[tz], n_touch = c->cum_m[tz], n_pairs = c->cum_q[tz], n_end = c->cum_b[tz1];
    PairArgs<T> ag = a, af = a, ah = a, ae = a;
    ag.order = c->order_b.as<int32_t>();
    ag.count = n_start;
    af.order = c->order_q.as<int32_t>();
    af.count = n_pairs;
    ah.order = c->order_m.as<int32_t>();
    ah.count = n_touch;
    ae.order = c->order_b.as<int32_t>();
    ae.count = n_end;
    const unsigned nbg = nblk(std::max<int64_t>(n_start, 1), 128), nbf = nblk(std::max<int64_t>(n_pairs, 1), 128);
    const unsigned nbe = nblk(std::max<int64_t>(n_end, 1), 128);
    // the float pair pass by row gathers of the packed rows: the gradient kernel writes the
    // rows of the particles starting a step (their state after injection and their new
    // gradient); every other particle's row still holds the state and gradient of its own
    // step start, which is what its pairs use until its step ends
    bool packed = false;
    if constexpr (std::is_same<T, float>::value)
        packed = G <= kMaxGC && packed_rows(c);
    if (packed) {
        ag.frec = c->frec.as<T>();
        af.frec = c->frec.as<T>();
    }
    for (int g0 = 0; g0 < G; g0 += chunk_groups(G)) {
        const int gc = G - g0 < chunk_groups(G) ? G - g0 : chunk_groups(G);
        if (n_start == 0) break;
        if constexpr (std::is_same<T, double>::value) {
            if (ag.wd) {
                switch (gc) {
                    case 1: launch_gradient_wd<1, true>(c, s, ag, rec, gr, g0); break;
                    case 2: launch_gradient_wd<2, true>(c, s, ag, rec, gr, g0); break;
                    case 3: launch_gradient_wd<3, true>(c, s, ag, rec, gr, g0); break;
                    default: launch_gradient_wd<4, true>(c, s, ag, rec, gr, g0); break;
                }
                ++c->launches;
                continue;
            }
        }
        if constexpr (std::is_same<T, float>::value) {
            const int64_t w = (n_start + 32 / gc - 1) / (32 / gc);       // warps of the shuffle gradient
            const unsigned nbs = nblk(w * 32, kGradBlock);
            switch (gc) {
                case 1: k_gradient_g<1, true><<<nblk(n_start, 256), 256, 0, s>>>(ag, rec, gr, g0); break;
                case 2: k_gradient_s<2, true><<<nbs, kGradBlock, 0, s>>>(ag, rec, gr, g0); break;
                case 3: k_gradient_s<3, true><<<nbs, kGradBlock, 0, s>>>(ag, rec, gr, g0); break;
                default: k_gradient_s<4, true><<<nbs, kGradBlock, 0, s>>>(ag, rec, gr, g0); break;
            }
        } else {
            switch (gc) {
                case 1: k_gradient<T, 1, true><<<nbg, 128, 0, s>>>(ag, rec, gr, g0); break;
                case 2: k_gradient<T, 2, true><<<nbg, 128, 0, s>>>(ag, rec, gr, g0); break;
                case 3: k_gradient<T, 3, true><<<nbg, 128, 0, s>>>(ag, rec, gr, g0); break;
                default: k_gradient<T, 4, true><<<nbg, 128, 0, s>>>(ag, rec, gr, g0); break;
            }
        }
        ++c->launches;
    }
    for (int g0 = 0; g0 < G; g0 += chunk_groups(G)) {
        const int gc = G - g0 < chunk_groups(G) ? G - g0 : chunk_groups(G);
#define RT_BINS_FLUX(GC_)                                                                    \
    if (n_pairs > 0) {                                                                       \
        if (packed)                                                                          \
            bins_flux_tma<GC_>(c, s, af, x, pb, hll);                                        \
        else if (hll)                                                                        \
            k_flux<T, GC_, true, true><<<nbf, 128, 0, s>>>(af, x, rec, pb, g0);              \
        else                                                                                 \
            k_flux<T, GC_, false, true><<<nbf, 128, 0, s>>>(af, x, rec, pb, g0);             \
        ++c->launches;                                                                       \
    }                                                                                        \
    if (n_touch > 0) {                                                                       \
        k_gather_bins<T, GC_><<<nblk(n_touch * GC_, 256), 256, 0, s>>>(ah, x, pb, rec, g0);   \
        ++c->launches;                                                                       \
    }                                                                                        \
    if (n_end > 0) {                                                                         \
        k_finalize_bins<T, GC_><<<nbe, 128, 0, s>>>(ae, x, rec, g0);                         \
        ++c->launches;                                                                       \
    }
        switch (gc) {
            case 1: RT_BINS_FLUX(1) break;
            case 2: RT_BINS_FLUX(2) break;
            case 3: RT_BINS_FLUX(3) break;
            default: RT_BINS_FLUX(4) break;
        }
#undef RT_BINS_FLUX
    }
}

rt_status launch_step_bins(rt_ctx* c, cudaStream_t s, int step, void* U, bool has_src, bool has_alpha) {
    if (c->fp64)
        launch_step_bins_t<double>(c, s, step, (double*)U, has_src, has_alpha);
    else
        launch_step_bins_t<float>(c, s, step, (float*)U, has_src, has_alpha);
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

rt_status launch_step(rt_ctx* c, cudaStream_t s, void* Uin, void* Uout, bool has_src, bool has_alpha,
                      bool inject_first, bool inject_after) {
    inject_first = inject_first && has_src;
    inject_after = inject_after && has_src && c->inj_dense_ready;
    if (c->fp64) {
        if (inject_first) launch_inject_t<double>(c, s, (double*)Uin);
        launch_gradient_t<double>(c, s, (double*)Uin);
        launch_flux_t<double>(c, s, (const double*)Uin, (double*)Uout, has_alpha, false, inject_after);
    } else {
        if (inject_first) launch_inject_t<float>(c, s, (float*)Uin);
        // packed rows for the tensor-memory-accelerator pair pass, which hold one chunk of groups:
        // each chunk's gradient, fluxes and update in turn (a chunk reads and writes its own
        // groups only).  99,991 particles and five groups: 0.166 ms of pair passes a sub-cycle
        // with direct loads
        if (packed_rows(c)) {
            const int G = c->cfg.n_groups;
            for (int g0 = 0; g0 < G; g0 += chunk_groups(G)) {
                launch_gradient_t<float>(c, s, (float*)Uin, true, g0);
                launch_flux_t<float>(c, s, (const float*)Uin, (float*)Uout, has_alpha, true, inject_after, g0);
            }
        } else {
            launch_gradient_t<float>(c, s, (float*)Uin);
            launch_flux_t<float>(c, s, (const float*)Uin, (float*)Uout, has_alpha, false, inject_after);
        }
    }
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

rt_status state_in(rt_ctx* c, const void* U_user, void* rec, int comps) {
    const dim3 nb(nblk(c->n, 256), comps / 4);
    if (c->fp64)
        k_state_in<double><<<nb, 256, 0, c->stream>>>((const double*)U_user, c->inv_perm.as<int32_t>(), c->n, comps,
                                                      (double*)rec);
    else
        k_state_in<float><<<nb, 256, 0, c->stream>>>((const float*)U_user, c->inv_perm.as<int32_t>(), c->n, comps,
                                                     (float*)rec);
    ++c->launches;
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

rt_status state_out(rt_ctx* c, const void* rec, void* U_user, int comps) {
    const dim3 nb(nblk(c->n, 256), comps / 4);
    if (c->fp64)
        k_state_out<double><<<nb, 256, 0, c->stream>>>((const double*)rec, c->inv_perm.as<int32_t>(), c->n, comps,
                                                       (double*)U_user);
    else
        k_state_out<float><<<nb, 256, 0, c->stream>>>((const float*)rec, c->inv_perm.as<int32_t>(), c->n, comps,
                                                      (float*)U_user);
    ++c->launches;
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

rt_status field_out(rt_ctx* c, const double* src_sorted, double* dst_user, int comps) {
    k_from_sorted<double><<<nblk(c->n, 256), 256, 0, c->stream>>>(src_sorted, c->inv_perm.as<int32_t>(), c->n, comps,
                                                                  dst_user);
    ++c->launches;
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

rt_status set_step_inputs(rt_ctx* c, double dt, const double* Lsrc, const double* alpha) {
    cudaStream_t s = c->stream;
    k_set_scalar<<<1, 1, 0, s>>>(c->dt_dev.as<double>(), dt, c->n_inj_targets);
    ++c->launches;
    if (Lsrc && c->n_src > 0)
        RT_CUDA(c, cudaMemcpyAsync(c->L_dev.p, Lsrc, (size_t)c->n_src * c->cfg.n_groups * sizeof(double),
                                   cudaMemcpyDeviceToDevice, s));
    if (alpha) {
        unsigned nb = nblk(c->n, 256);
        if (c->fp64) k_alpha_sorted<double><<<nb, 256, 0, s>>>(alpha, c->perm.as<int32_t>(), c->n, c->alpha_s.as<double>());
        else k_alpha_sorted<float><<<nb, 256, 0, s>>>(alpha, c->perm.as<int32_t>(), c->n, c->alpha_s.as<float>());
        ++c->launches;
    }
    // the photo-ionisation sink per group applies when no grey alpha is given
    c->step_alpha_g = !alpha && c->has_alpha_g;
    if (c->step_alpha_g) {
        unsigned nb = nblk(c->n, 256);
        const int G = c->cfg.n_groups;
        if (c->fp64)
            k_alpha_g_sorted<double><<<nb, 256, 0, s>>>(c->alpha_g_c.as<double>(), c->perm.as<int32_t>(), c->n, G,
                                                        c->alpha_g_s.as<double>());
        else
            k_alpha_g_sorted<float><<<nb, 256, 0, s>>>(c->alpha_g_c.as<double>(), c->perm.as<int32_t>(), c->n, G,
                                                       c->alpha_g_s.as<float>());
        ++c->launches;
    }
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

// one warp waits on a barrier that nothing completes (rt_wait_selftest)
__global__ void k_wait_selftest(unsigned long long budget, int* ran_out) {
    __shared__ __align__(8) uint64_t bar;
    const uint32_t b = smem_u32(&bar);
    if (threadIdx.x == 0) mbar_init(b, 1);
    __syncwarp();
    const bool done = mbar_wait(b, 0, budget);
    if (!__any_sync(0xffffffffu, done) && threadIdx.x == 0) *ran_out = 1;
}

rt_status wait_selftest(rt_ctx* c, unsigned long long budget, bool* ran_out) {
    int* f = c->flags.as<int>() + F_SELFTEST;
    RT_CUDA(c, cudaMemsetAsync(f, 0, sizeof(int), c->stream));
    k_wait_selftest<<<1, 32, 0, c->stream>>>(budget, f);
    ++c->launches;
    RT_CUDA(c, cudaGetLastError());
    int h = 0;
    RT_CUDA(c, cudaMemcpyAsync(&h, f, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    RT_CUDA(c, cudaStreamSynchronize(c->stream));
    *ran_out = h != 0;
    return RT_OK;
}

rt_status set_dense_injection(rt_ctx* c, bool on) {
    c->inj_dense_ready = false;
    if (!on || c->n_inj_targets <= 0 || !c->inj_dense.p) return RT_OK;
    cudaStream_t s = c->stream;
    const int G = c->cfg.n_groups;
    RT_CUDA(c, cudaMemsetAsync(c->inj_dense.p, 0, (size_t)G * c->n * 8, s));
    k_inject_dense<<<nblk(c->n_inj_targets, 128), 128, 0, s>>>(
        c->inj_targets.as<int32_t>(), c->inj_off.as<int32_t>(), c->inj_src.as<int32_t>(), c->inj_coef.as<double>(),
        c->L_dev.as<double>(), G, c->dt_dev.as<double>(), c->n_inj_targets, c->inj_dense.as<double>());
    ++c->launches;
    RT_CUDA(c, cudaGetLastError());
    c->inj_dense_ready = true;
    return RT_OK;
}

rt_status launch_energy(rt_ctx* c, cudaStream_t s, const void* U, double* out_dev) {
    double* part = c->energy_part.as<double>();
    const int32_t* inv = c->inv_perm.as<int32_t>();
    if (c->fp64)
        k_energy_part<double><<<kEnergyBlocks, 256, 0, s>>>((const double*)U, c->V_d.as<double>(), c->n,
                                                            c->cfg.n_groups, inv, c->n_owned, part);
    else
        k_energy_part<float><<<kEnergyBlocks, 256, 0, s>>>((const float*)U, c->V_d.as<double>(), c->n,
                                                           c->cfg.n_groups, inv, c->n_owned, part);
    k_energy_final<<<c->cfg.n_groups, kEnergyBlocks, 0, s>>>(part, out_dev);
    c->launches += 2;
    RT_CUDA(c, cudaGetLastError());
    return RT_OK;
}

}  // namespace rt
