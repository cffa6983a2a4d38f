// Neighbour search and particle geometry of the FVPM photon-transport step:
// cell list, smoothing lengths, symmetric pair lists, E_i / B_i, source injection weights.
//
// Part II of Ivkovic (2023), "The Neighbor Search: Determining the Smoothing Length"
// (Eq. number-of-neighbors), Eqs. omega / particle-volume, matrix_E / matrix_B; Part III,
// "Weights For Distribution Of Energy Density of a Star onto Particles"
// (Eq. isotropy-correction-with-zero).  The thesis runs these as SWIFT cell tasks on CPUs;
// here each is a data-parallel kernel over cell-sorted particles.
#include <cub/cub.cuh>

#include <cmath>
#include <type_traits>
#include <vector>

#include "rt_pair.cuh"

namespace rt {


struct Box {
    double box[3];
    int periodic;
};

struct Grid {
    int nc[3];
    double cell[3];
    double inv_cell[3];
    float cellf[3], inv_cellf[3];
    double box[3];
    int periodic;
    const int32_t* cell_start;   // [ncells + 1], lower bound of each cell in sorted order
};

// atomic min / max of positive doubles through their bit patterns (ordered like integers)
__device__ __forceinline__ void atomic_min_pos(unsigned long long* a, double v) {
    atomicMin(a, (unsigned long long)__double_as_longlong(v));
}
__device__ __forceinline__ void atomic_max_pos(unsigned long long* a, double v) {
    atomicMax(a, (unsigned long long)__double_as_longlong(v));
}
__device__ __forceinline__ void warp_minmax(double& mn, double& mx) {
    for (int o = 16; o > 0; o >>= 1) {
        mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
}

__device__ __forceinline__ int wrap_cell(int c, int nc) {
    c %= nc;
    return c < 0 ? c + nc : c;
}

// Visit every particle (sorted index) whose cell can hold points within R of p.  Rows of
// cells along x are contiguous in sorted order; rows whose (y, z) extent is farther than R
// are skipped and each row is clipped to the chord of the sphere, so the visited volume
// is close to the sphere plus one cell layer.  An axis whose span covers the whole grid is
// walked once without clipping.  With ASC the ranges come in ascending cell index (a
// periodic axis is walked from the cell that wraps to the lowest index), so that the
// candidates, being sorted by cell, come in ascending particle index.  Where fr returns a bool,
// false ends the walk.
__device__ __forceinline__ int first_wrapped(int lo, int hi, int nc) {
    return lo < 0 ? 0 : (hi >= nc ? nc : lo);
}

template <bool ASC = false, class F>
__device__ __forceinline__ void for_each_candidate_range(const Grid& g, float px, float py, float pz, float R,
                                                         F&& fr) {
    // float arithmetic with a relative margin of 1e-4 on R: cells are never missed
    const float Rc = R * 1.0001f + 1e-6f * (g.cellf[0] + g.cellf[1] + g.cellf[2]);
    const float R2 = Rc * Rc;
    const float p[3] = {px, py, pz};
    int lo[3], hi[3];
    bool all[3];
    for (int a = 0; a < 3; ++a) {
        lo[a] = (int)floorf((p[a] - Rc) * g.inv_cellf[a]);
        hi[a] = (int)floorf((p[a] + Rc) * g.inv_cellf[a]);
        all[a] = (hi[a] - lo[a] + 1 >= g.nc[a]);
        if (all[a]) {
            lo[a] = 0;
            hi[a] = g.nc[a] - 1;
        } else if (!g.periodic) {
            lo[a] = max(lo[a], 0);
            hi[a] = min(hi[a], g.nc[a] - 1);
        }
    }
    const int nzs = hi[2] - lo[2] + 1, nys = hi[1] - lo[1] + 1;
    const int z0 = ASC ? first_wrapped(lo[2], hi[2], g.nc[2]) : lo[2];
    const int y0 = ASC ? first_wrapped(lo[1], hi[1], g.nc[1]) : lo[1];
    for (int kz = 0; kz < nzs; ++kz) {
        int z = z0 + kz;
        if (z > hi[2]) z -= nzs;
        float dz = 0.f;
        if (!all[2]) dz = fmaxf(0.f, fmaxf(z * g.cellf[2] - pz, pz - (z + 1) * g.cellf[2]));
        if (dz * dz >= R2) continue;
        int zz = wrap_cell(z, g.nc[2]);
        for (int ky = 0; ky < nys; ++ky) {
            int y = y0 + ky;
            if (y > hi[1]) y -= nys;
            float dy = 0.f;
            if (!all[1]) dy = fmaxf(0.f, fmaxf(y * g.cellf[1] - py, py - (y + 1) * g.cellf[1]));
            float rem = R2 - dy * dy - dz * dz;
            if (rem <= 0.f) continue;
            int yy = wrap_cell(y, g.nc[1]);
            int64_t base = ((int64_t)zz * g.nc[1] + yy) * g.nc[0];
            int xa, xb;
            if (all[0]) {
                xa = 0;
                xb = g.nc[0] - 1;
            } else {
                float w = sqrtf(rem);
                xa = (int)floorf((px - w) * g.inv_cellf[0]);
                xb = (int)floorf((px + w) * g.inv_cellf[0]);
                if (!g.periodic) {
                    xa = max(xa, 0);
                    xb = min(xb, g.nc[0] - 1);
                }
            }
            int sl[2], sh[2], ns = 0;
            if (xa < 0) {
                if (ASC) { sl[ns] = 0; sh[ns++] = xb; sl[ns] = xa + g.nc[0]; sh[ns++] = g.nc[0] - 1; }
                else { sl[ns] = xa + g.nc[0]; sh[ns++] = g.nc[0] - 1; sl[ns] = 0; sh[ns++] = xb; }
            } else if (xb >= g.nc[0]) {
                if (ASC) { sl[ns] = 0; sh[ns++] = xb - g.nc[0]; sl[ns] = xa; sh[ns++] = g.nc[0] - 1; }
                else { sl[ns] = xa; sh[ns++] = g.nc[0] - 1; sl[ns] = 0; sh[ns++] = xb - g.nc[0]; }
            } else { sl[ns] = xa; sh[ns++] = xb; }
            for (int sI = 0; sI < ns; ++sI) {
                int b = g.cell_start[base + sl[sI]];
                int e = g.cell_start[base + sh[sI] + 1];
                if constexpr (std::is_same<decltype(fr(b, e)), bool>::value) {
                    if (!fr(b, e)) return;
                } else {
                    fr(b, e);
                }
            }
        }
    }
}

// every candidate of for_each_candidate_range, one at a time
template <bool ASC = false, class F>
__device__ __forceinline__ void for_each_candidate(const Grid& g, float px, float py, float pz, float R, F&& f) {
    for_each_candidate_range<ASC>(g, px, py, pz, R, [&](int b, int e) {
        for (int j = b; j < e; ++j) f(j);
    });
}

// number of particles in the 3 x 3 x 3 cells around (cx, cy, cz): a local density for the
// first guess of h
__device__ __forceinline__ int count_27(const Grid& g, int cx, int cy, int cz) {
    int cnt = 0;
    for (int dz = -1; dz <= 1; ++dz) {
        int z = cz + dz;
        if (!g.periodic && (z < 0 || z >= g.nc[2])) continue;
        int zz = wrap_cell(z, g.nc[2]);
        for (int dy = -1; dy <= 1; ++dy) {
            int y = cy + dy;
            if (!g.periodic && (y < 0 || y >= g.nc[1])) continue;
            int yy = wrap_cell(y, g.nc[1]);
            int64_t base = ((int64_t)zz * g.nc[1] + yy) * g.nc[0];
            for (int dx = -1; dx <= 1; ++dx) {
                int x = cx + dx;
                if (!g.periodic && (x < 0 || x >= g.nc[0])) continue;
                int xx = wrap_cell(x, g.nc[0]);
                cnt += g.cell_start[base + xx + 1] - g.cell_start[base + xx];
            }
        }
    }
    return cnt;
}

__device__ __forceinline__ int cell_coord(double x, double inv_cell, int nc) {
    int c = (int)floor(x * inv_cell);
    return min(max(c, 0), nc - 1);
}

// exact (no contraction) minimal-image separation, identical to a plain double evaluation
__device__ __forceinline__ double sep_exact(double xj, double xi, double box, int periodic) {
    double v = __dsub_rn(xj, xi);
    if (periodic) v = __dsub_rn(v, __dmul_rn(box, rint(__ddiv_rn(v, box))));
    return v;
}

__device__ __forceinline__ double norm2_exact(double a, double b, double c) {
    return __dadd_rn(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)), __dmul_rn(c, c));
}

// fast minimal image (same value except at exactly half a box, which never neighbours)
__device__ __forceinline__ double sep_fast(double xj, double xi, double box, double half, int periodic) {
    double v = xj - xi;
    if (periodic) {
        if (v > half) v -= box;
        else if (v < -half) v += box;
    }
    return v;
}

// ------------------------------------------------------------------------------------
// a1: cell keys, validation
// A coordinate that is not finite or not in the box is refused, but the host learns of it only after
// the search has been queued.  Until then a value spread over the box by the particle's index
// stands in for it, in the keys and in the sorted copies, so that every walk stays in the cell
// table and meets no more candidates than an even set has.
__device__ __forceinline__ double position_in_box(double v, double box, int64_t i, int axis, bool& bad) {
    if (v >= 0.0 && v < box) return v;
    bad = true;
    uint32_t u = (uint32_t)i * 0x9e3779b9u + (uint32_t)axis * 0x85ebca6bu;   // a multiplicative hash
    u = (u ^ (u >> 16)) * 0x7feb352du;
    u = (u ^ (u >> 15)) * 0x846ca68bu;
    return box * ((double)(u ^ (u >> 16)) * 0x1p-32);
}

__global__ void k_keys(const double* __restrict__ x, int64_t n, Grid g, uint32_t* keys, int32_t* idx, int* flags) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int c[3];
    bool bad = false;
    for (int a = 0; a < 3; ++a) {
        c[a] = cell_coord(position_in_box(x[a * n + i], g.box[a], i, a, bad), g.inv_cell[a], g.nc[a]);
    }
    if (bad) atomicExch(&flags[F_BADPOS], 1);
    keys[i] = (uint32_t)(((int64_t)c[2] * g.nc[1] + c[1]) * g.nc[0] + c[0]);
    idx[i] = (int32_t)i;
}

__global__ void k_cell_start(const uint32_t* __restrict__ keys, int64_t n, int64_t ncells, int32_t* cell_start) {
    int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c > ncells) return;
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (keys[mid] < (uint32_t)c) lo = mid + 1; else hi = mid;
    }
    cell_start[c] = (int32_t)lo;
}

__global__ void k_gather_positions(const double* __restrict__ x, const double* __restrict__ m,
                                   const int32_t* __restrict__ perm, int64_t n, Box b, double q0, double q1, double q2,
                                   double* xs, uint4* xq, double* ms, int32_t* inv_perm) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    int64_t i = perm[p];
    double qs[3] = {q0, q1, q2};
    uint32_t qv[3];
    for (int a = 0; a < 3; ++a) {
        bool bad = false;
        const double v = position_in_box(x[a * n + i], b.box[a], i, a, bad);
        xs[a * n + p] = v;
        double f = floor(v * qs[a]);
        f = fmin(fmax(f, 0.0), 4294967295.0);
        qv[a] = (uint32_t)f;
    }
    xq[p] = make_uint4(qv[0], qv[1], qv[2], 0u);   // one 16-byte record a particle for the walks
    ms[p] = m ? m[i] : 0.0;
    inv_perm[i] = (int32_t)p;
}

// ------------------------------------------------------------------------------------
// Walk of one warp for one particle: the rows of cells of for_each_candidate_range<true>, one
// row per lane, so that the range arithmetic and the cell-table loads of up to 32 rows run side
// by side; their candidates, numbered by a prefix sum over the lanes, are then dealt 32 at a time
// to the lanes.  f(j, valid) sees them in ascending index, called by the whole warp, and ends the
// walk by returning false (the same in every lane).  A thread that walks its own sphere runs
// row by row on the latency of the table and record loads, half of a warp's lanes idle (14.8
// active of 32) behind the longest row; a warp per particle that takes the rows in turn repeats the row
// arithmetic in every lane.  Periodic cells wrap once, so (px, py, pz) has to lie in the box, its
// upper edge included (position_in_box, k_src_positions).
__device__ __forceinline__ int wrap_once(int c, int nc) { return c < 0 ? c + nc : (c >= nc ? c - nc : c); }

// ASC false: the order of for_each_candidate_range<false>, which differs where a sphere wraps.
template <bool ASC = true, class F>
__device__ __forceinline__ void warp_walk(const Grid& g, float px, float py, float pz, float R, int lane, F&& f) {
    const unsigned FULL = 0xffffffffu;
    const float Rc = R * 1.0001f + 1e-6f * (g.cellf[0] + g.cellf[1] + g.cellf[2]);
    const float R2 = Rc * Rc;
    const float p[3] = {px, py, pz};
    int lo[3], hi[3];
    bool all[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = (int)floorf((p[a] - Rc) * g.inv_cellf[a]);
        hi[a] = (int)floorf((p[a] + Rc) * g.inv_cellf[a]);
        all[a] = (hi[a] - lo[a] + 1 >= g.nc[a]);
        if (all[a]) {
            lo[a] = 0;
            hi[a] = g.nc[a] - 1;
        } else if (!g.periodic) {
            lo[a] = max(lo[a], 0);
            hi[a] = min(hi[a], g.nc[a] - 1);
        }
    }
    const int nzs = hi[2] - lo[2] + 1, nys = hi[1] - lo[1] + 1;
    const int z0 = ASC ? first_wrapped(lo[2], hi[2], g.nc[2]) : lo[2];
    const int y0 = ASC ? first_wrapped(lo[1], hi[1], g.nc[1]) : lo[1];
    const int rows = nzs > 0 && nys > 0 ? nzs * nys : 0;
    for (int r0 = 0; r0 < rows; r0 += 32) {
        const int r = r0 + lane;
        int b1 = 0, n1 = 0, b2 = 0, n2 = 0;
        if (r < rows) {
            const int kz = r / nys, ky = r - kz * nys;
            int z = z0 + kz, y = y0 + ky;
            if (z > hi[2]) z -= nzs;
            if (y > hi[1]) y -= nys;
            const float dz = all[2] ? 0.f : fmaxf(0.f, fmaxf(z * g.cellf[2] - pz, pz - (z + 1) * g.cellf[2]));
            const float dy = all[1] ? 0.f : fmaxf(0.f, fmaxf(y * g.cellf[1] - py, py - (y + 1) * g.cellf[1]));
            const float rem = R2 - dy * dy - dz * dz;
            if (rem > 0.f) {
                const int base = (wrap_once(z, g.nc[2]) * g.nc[1] + wrap_once(y, g.nc[1])) * g.nc[0];
                int xa = 0, xb = g.nc[0] - 1;
                if (!all[0]) {
                    const float w = sqrtf(rem);
                    xa = (int)floorf((px - w) * g.inv_cellf[0]);
                    xb = (int)floorf((px + w) * g.inv_cellf[0]);
                    if (!g.periodic) {
                        xa = max(xa, 0);
                        xb = min(xb, g.nc[0] - 1);
                    }
                }
                // up to two ranges of cells, the wrapped part first
                int s1 = xa, e1 = xb, s2 = 0, e2 = -1;
                if (xa < 0) {
                    s1 = 0; e1 = xb; s2 = xa + g.nc[0]; e2 = g.nc[0] - 1;
                } else if (xb >= g.nc[0]) {
                    s1 = 0; e1 = xb - g.nc[0]; s2 = xa; e2 = g.nc[0] - 1;
                }
                if (!ASC && s2 <= e2) {
                    const int s = s1, e = e1;
                    s1 = s2; e1 = e2; s2 = s; e2 = e;
                }
                if (s1 <= e1) {
                    b1 = g.cell_start[base + s1];
                    n1 = g.cell_start[base + e1 + 1] - b1;
                }
                if (s2 <= e2) {
                    b2 = g.cell_start[base + s2];
                    n2 = g.cell_start[base + e2 + 1] - b2;
                }
            }
        }
        int end = n1 + n2;      // inclusive prefix sum of the rows' candidates
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, end, o);
            if (lane >= o) end += v;
        }
        const int off = end - n1 - n2, total = __shfl_sync(FULL, end, 31);
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + lane;
            int L = 0;          // the last row whose first candidate is not past t
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(FULL, off, L + o) <= t) L += o;
            const int c = t - __shfl_sync(FULL, off, L), m = __shfl_sync(FULL, n1, L);
            const int u1 = __shfl_sync(FULL, b1, L), u2 = __shfl_sync(FULL, b2, L);
            if (!f(c < m ? u1 + c : u2 + (c - m), t < total)) return;
        }
    }
}

// whether the two orders of that walk may differ
__device__ __forceinline__ bool walk_wraps(const Grid& g, float px, float py, float pz, float R) {
    const float Rc = R * 1.0001f + 1e-6f * (g.cellf[0] + g.cellf[1] + g.cellf[2]);
    const float p[3] = {px, py, pz};
    bool w = false;
#pragma unroll
    for (int a = 0; a < 3; ++a)
        w |= p[a] - Rc < g.cellf[a] || p[a] + Rc > (g.nc[a] - 1) * g.cellf[a];
    return g.periodic && w;
}

// ------------------------------------------------------------------------------------
// a2: smoothing lengths, h = eta omega(h)^(-1/3) with omega(h) = sum_j W(r_ij, h) and the self
// term.  With S(h) = sum_j w(r_ij / H) the equation is S(h) = S* = (kappa eta)^3 / sigma, the
// same number for every particle.
//
// Float phase (k_h_lists): safeguarded Newton on f(h) = h - eta omega(h)^(-1/3), nearly linear
// in h, from the h of the previous call or a local particle count.  The candidates are walked
// once, out to a little more than the first guess's support: their indices go to the
// particle's list in memory, from which the double phase and the pair search take them, their
// distances to shared memory, over which the iterations sum.  Where they overflow the list (a particle
// that has moved into a dense clump with the h of a void) each iteration walks.
//
// The iterates are those of one thread that adds w in double and dw/dh in float, candidate by
// candidate in the order of for_each_candidate_range<false>: the sum of w is kept to 1e-14 (Sum2), and the
// sum of dw/dh, whose float rounding decides the last bits of an iterate, is added in that order.  h,
// omega, V and B are therefore the same, to 1e-14, however the candidates are dealt out.
//
// Double phase (k_h_refine): Newton on S(h) - S* in double on the exact separations.  On the
// FP64 path it runs for every particle.  On the float path it runs only for the
// particles that have a candidate within the near band of their own support radius at the float
// root: that is within a few 1e-6 of the exact one, so for every other particle no neighbour
// can change side of H_i, and the pair lists, which are decided by H_i and H_j, are those of the
// exact roots.
struct HParams {
    double eta, h0, h_cap;
    double s_star, eta3;   // S* = (kappa eta)^3 / sigma, and eta^3
    float scale[3];
    int max_iter;
    float tol32;
    int refine64;   // 1: the double phase follows for every particle, 0: for the flagged ones
};

// |r^2 - H^2| < kNearBand H^2 at the float root flags the particle for the double phase; kNear, a
// little more than its half, is the margin in r that lists keep around H
constexpr float kNearBand = 2e-4f, kNear = 1.1e-4f;

__device__ __forceinline__ float fsep(uint32_t a, uint32_t b, float scale) { return (float)(int32_t)(a - b) * scale; }

// compensated float sum
struct Kahan {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v) {
        float y = v - c;
        float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// float sum with the exact rounding error of every addition (TwoSum) in a second float: as good as a
// double sum to 1e-14 over a row
struct Sum2 {
    float s = 0.f, e = 0.f;
    __device__ __forceinline__ void add(float v, float ev = 0.f) {
        const float t = __fadd_rn(s, v), z = __fsub_rn(t, s);
        const float r = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(v, z));
        e = __fadd_rn(__fadd_rn(e, ev), r);
        s = t;
    }
};

// One Newton step of the float phase from the sums at h: whether h is the root to the tolerance,
// else the next iterate
__device__ __forceinline__ bool h_newton(const HParams& hp, float h, float sw, float sdw, int it, float& lo,
                                         float& hi, float& next) {
    const float kapf = (float)kKappa, sigf = (float)kSigma, eta = (float)hp.eta;
    const float H = kapf * h;
    const float iH = 1.f / H;
    float om = sigf * iH * iH * iH * sw;
    float dom = -kapf * sigf * iH * iH * iH * iH * sdw;      // d omega / d h
    float cb = cbrtf(om);
    float f = h - eta / cb;
    float fp = 1.f + (eta / 3.f) / (cb * om) * dom;
    if (f < 0.f) lo = h; else hi = h;
    float step = f / fp;
    // converged: residual at the rounding floor, a tiny Newton step, or a collapsed
    // bracket (where f' is small, rounding alone keeps the step above tolerance)
    if (fabsf(f) <= 1e-6f * h || (fp > 0.f && fabsf(step) <= hp.tol32 * h) || (hi - lo) <= hp.tol32 * h) return true;
    float hn = h - step;
    // safeguarded Newton; plain bisection of the bracket after 24 Newton steps
    if (it >= 24 || !(hn > lo && hn < hi) || !(fp > 0.f)) hn = isinf(hi) ? 2.f * h : 0.5f * (lo + hi);
    if (hn > (float)hp.h_cap) hn = (float)hp.h_cap;
    next = hn;
    return false;
}

// w and t = 3 w + q w' of one candidate at distance r.  Rounded as written: h must not depend on which
// of the two sums below, or which order of the lanes, a particle takes.
__device__ __forceinline__ float h_term(float r, float iH, float& t) {
    const float q = __fmul_rn(r, iH);
    t = 0.f;
    if (q >= 1.f) return 0.f;
    const float u = __fsub_rn(1.f, q);
    float w = __fmul_rn(__fmul_rn(u, u), u), d = __fmul_rn(__fmul_rn(-3.f, u), u);
    if (q <= 0.5f) {
        const float v = __fsub_rn(0.5f, q);
        w = __fmaf_rn(-__fmul_rn(__fmul_rn(4.f, v), v), v, w);
        d = __fmaf_rn(__fmul_rn(12.f, v), v, d);
    }
    t = __fmaf_rn(3.f, w, __fmul_rn(q, d));
    return w;
}
__device__ __forceinline__ float r2_rn(float dx, float dy, float dz) {
    return __fmaf_rn(dz, dz, __fmaf_rn(dx, dx, __fmul_rn(dy, dy)));
}

// lanes a particle of the sums, warps and particles a block
constexpr int kSumLanes = 8, kListWarps = 8, kListParticles = kListWarps * 32 / kSumLanes;

// entries a particle's candidate list holds: twice what 1.1 support radii hold of an even set (128
// at the usual eta), at most what the blocks' 48 KB of shared distances allow
static int list_capacity(double eta) {
    const double even = 4.18879 * std::pow(kKappa * eta * 1.1, 3.0);
    return (int)std::min(352.0, std::max(32.0, std::floor((2.0 * even + 31.0) / 32.0) * 32.0));
}

// SOLVE: h by Newton, and the list of the candidates within at least H (1 + 2 kNear) of it.
// Otherwise h_out holds the smoothing lengths, and only the lists are made.  list_cnt is the
// list's length, or -1 where it overflowed.  Each warp walks for its four particles in turn; the
// sums of the four then run side by side on eight lanes each.
// 262,144 particles that moved by a tenth of their spacing took 0.88 ms with a thread per
// particle and a walk of the cells every iteration.  A whole search of 1,000,000 strongly clustered
// particles takes 5.8 ms (17 ms), and up to 24 ms (172 ms) where some had the h of a place far less
// dense: those walk the clump, its derivative terms one after the other (loading the next records
// ahead of the sums spills and takes 26 ms).
template <bool SOLVE>
__global__ void __launch_bounds__(kListWarps * 32)
k_h_lists(Grid g, const double* __restrict__ xs, const uint4* __restrict__ xq, int64_t n, HParams hp,
          const double* __restrict__ h_prev, const int32_t* __restrict__ perm, const double* __restrict__ h_given,
          float* __restrict__ h_sum, int* flags, int32_t* refine_list, int* refine_count,
          int32_t* __restrict__ list, int32_t* __restrict__ list_cnt, int cap) {
    constexpr int PW = 32 / kSumLanes;            // particles a warp
    const unsigned FULL = 0xffffffffu;
    extern __shared__ float st_all[];             // distances of the stored candidates, cap a particle
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int a = lane / kSumLanes, sub = lane % kSumLanes;
    const int64_t p0 = (blockIdx.x * (int64_t)kListWarps + wid) * PW, p = p0 + a;
    const bool active = p < n;
    float* st = st_all + wid * PW * cap;
    const float kapf = (float)kKappa;
    float h = 0.f;
    if (active) {
        if (!SOLVE) {
            h = (float)h_given[p];
        } else if (h_prev) {
            // first guess: the particle's h of the previous call (particles move little between
            // calls), else the particle count of the surrounding 27 cells
            h = (float)h_prev[perm[p]];
        } else {
            int cnt = count_27(g, cell_coord(xs[p], g.inv_cell[0], g.nc[0]),
                               cell_coord(xs[n + p], g.inv_cell[1], g.nc[1]),
                               cell_coord(xs[2 * n + p], g.inv_cell[2], g.nc[2]));
            double vol27 = 27.0 * g.cell[0] * g.cell[1] * g.cell[2];
            h = cnt > 1 ? (float)(hp.eta * cbrt(vol27 / (double)cnt)) : (float)hp.h0;
        }
        if (SOLVE && (!(h > 0.f) || !(h < (float)hp.h_cap))) h = (float)hp.h0;
    }
    float lo = 0.f, hi = INFINITY, Rs = 0.f, h_over = 0.f;
    // wants: the list is in use (until it overflows); Rs and cnt describe it
    bool done = !active, ok = false, near = false, wants = true;
    int cnt = 0, it = 0;
    Sum2 S_last;
    while (__any_sync(FULL, !done)) {
        const float H = kapf * h, iH = 1.f / H;
        const bool fill = !done && wants && H * (1.f + 2.f * kNear) > Rs;
        unsigned todo = __ballot_sync(FULL, fill && sub == 0);
        while (todo) {          // walks that store, one particle at a time
            const int src = __ffs(todo) - 1, b = src / kSumLanes;
            todo &= todo - 1;
            const int64_t q = p0 + b;
            const uint4 qp = xq[q];
            const float R = __shfl_sync(FULL, H, src) * (SOLVE ? 1.10f : 1.f + 4.f * kNear), R2 = R * R;
            const float bx = (float)qp.x * hp.scale[0], by = (float)qp.y * hp.scale[1], bz = (float)qp.z * hp.scale[2];
            int c = 0;
            auto store = [&](int j, bool valid, bool to_list, bool to_sum) {
                float r2 = INFINITY;
                if (valid) {
                    const uint4 qj = xq[j];
                    const float dx = fsep(qj.x, qp.x, hp.scale[0]);
                    const float dy = fsep(qj.y, qp.y, hp.scale[1]);
                    const float dz = fsep(qj.z, qp.z, hp.scale[2]);
                    r2 = r2_rn(dx, dy, dz);
                }
                const bool in = r2 < R2;
                const unsigned m = __ballot_sync(FULL, in);
                const int pos = c + __popc(m & ((1u << lane) - 1u));
                if (in && pos < cap) {
                    if (to_list) list[q * cap + pos] = j;
                    if (to_sum) st[b * cap + pos] = sqrtf(r2);
                }
                c += __popc(m);
                return c <= cap;
            };
            const bool wraps = SOLVE && walk_wraps(g, bx, by, bz, R);
            if (wraps) {
                warp_walk<false>(g, bx, by, bz, R, lane, [&](int j, bool v) { return store(j, v, false, true); });
                c = 0;
            }
            warp_walk(g, bx, by, bz, R, lane, [&](int j, bool v) { return store(j, v, true, SOLVE && !wraps); });
            if (a == b) {
                cnt = c;
                Rs = R;
                if (c > cap) {
                    wants = false;
                    Rs = 0.f;
                    h_over = h;
                    if (!SOLVE) done = true;
                }
            }
        }
        __syncwarp();
        if (!SOLVE) break;
        bool band = false;
        // S compensated, its derivative a plain float sum in the order of the walk: the eight terms of a
        // round are added one after the other in every lane, so that the iterates and the root
        // do not depend on how the candidates are dealt
        Sum2 sw;
        float sdw = 0.f, gap = INFINITY;
        const int mine = !done && wants ? cnt : 0;
        const int most = __reduce_max_sync(FULL, mine);
        for (int k0 = 0; k0 < most; k0 += kSumLanes) {
            const int k = k0 + sub;
            float t = 0.f;
            if (k < mine) {
                const float r = st[a * cap + k], q = r * iH;
                gap = fminf(gap, fabsf(fabsf(q * q - 1.f) - kNearBand));
                band |= fabsf(q * q - 1.f) < kNearBand;
                if (r < H) sw.add(h_term(r, iH, t));
            }
#pragma unroll
            for (int u = 0; u < kSumLanes; ++u) sdw += __shfl_sync(FULL, t, u, kSumLanes);
        }
#pragma unroll
        for (int o = kSumLanes / 2; o > 0; o >>= 1) {
            sw.add(__shfl_xor_sync(FULL, sw.s, o), __shfl_xor_sync(FULL, sw.e, o));
            gap = fminf(gap, __shfl_xor_sync(FULL, gap, o));
        }
        // walks that sum, for the particles whose candidates overflow the list
        todo = __ballot_sync(FULL, !done && !wants && sub == 0);
        while (todo) {
            const int src = __ffs(todo) - 1, b = src / kSumLanes;
            todo &= todo - 1;
            const uint4 qp = xq[p0 + b];
            const float Hb = __shfl_sync(FULL, H, src), iHb = 1.f / Hb, H2b = __fmul_rn(Hb, Hb);
            Sum2 swb;
            float sdb = 0.f;
            bool nb = false;
            warp_walk<false>(g, (float)qp.x * hp.scale[0], (float)qp.y * hp.scale[1], (float)qp.z * hp.scale[2],
                             Hb * (1.f + 2.f * kNear), lane, [&](int j, bool valid) {
                                 float t = 0.f;
                                 if (valid) {
                                     const uint4 qj = xq[j];
                                     const float dx = fsep(qj.x, qp.x, hp.scale[0]);
                                     const float dy = fsep(qj.y, qp.y, hp.scale[1]);
                                     const float dz = fsep(qj.z, qp.z, hp.scale[2]);
                                     const float r2 = r2_rn(dx, dy, dz);
                                     nb |= fabsf(__fsub_rn(r2, H2b)) < kNearBand * H2b;
                                     if (r2 < H2b) swb.add(h_term(sqrtf(r2), iHb, t));
                                 }
                                 if (__any_sync(FULL, t != 0.f)) {
#pragma unroll
                                     for (int u = 0; u < 32; ++u) sdb += __shfl_sync(FULL, t, u);
                                 }
                                 return true;
                             });
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) swb.add(__shfl_xor_sync(FULL, swb.s, o), __shfl_xor_sync(FULL, swb.e, o));
            nb = __any_sync(FULL, nb);
            if (a == b) {
                sw = swb;
                sdw = sdb;
                gap = INFINITY;
                band = nb;
            }
        }
        bool edge = false;
        if (!done) {
            S_last = sw;
            float hn = h;
            if (h_newton(hp, h, __fadd_rn(sw.s, sw.e), sdw, it, lo, hi, hn)) {
                ok = done = true;
                near = band;
                edge = gap < 2e-6f;
            } else if (hn == h || it + 1 >= hp.max_iter) {
                done = true;      // no progress possible: reported as not converged
            } else {
                h = hn;
                wants = wants || h < 0.85f * h_over;
            }
            ++it;
        }
        // a candidate within rounding of the band's edge: the band on the separations themselves
        if (__any_sync(FULL, edge)) {
            if (edge) {
                const uint4 qp = xq[p];
                const float H2 = __fmul_rn(H, H);
                near = false;
                for (int k = sub; k < cnt; k += kSumLanes) {
                    const uint4 qj = xq[list[p * cap + k]];
                    const float dx = fsep(qj.x, qp.x, hp.scale[0]);
                    const float dy = fsep(qj.y, qp.y, hp.scale[1]);
                    const float dz = fsep(qj.z, qp.z, hp.scale[2]);
                    const float r2 = r2_rn(dx, dy, dz);
                    near |= fabsf(__fsub_rn(r2, H2)) < kNearBand * H2;
                }
            }
        }
    }
    near = __any_sync(((1u << kSumLanes) - 1u) << (a * kSumLanes), near);
    if (active && sub == 0) {
        list_cnt[p] = wants ? cnt : -1;
        if (SOLVE) {
            if (!ok) atomicExch(&flags[F_NOCONV], 1);
            if (ok && near && !hp.refine64) refine_list[atomicAdd(refine_count, 1)] = (int32_t)p;
            h_sum[p] = h;
            h_sum[n + p] = S_last.s;
            h_sum[2 * n + p] = S_last.e;
        }
    }
}

// What the float phase leaves to one thread per particle (its few double instructions would cost
// k_h_lists, with eight lanes a particle, eight times as much): h, omega = sigma / H^3 S and the
// float H^2, also in the free word of the position record, so that the pair search reads a
// candidate's position and support radius with one 16-byte load; the smallest and largest h
// and the sum of H^3 (which only steers the reported pair_build).  With h_sum NULL (given h) only the
// record is filled.
__global__ void __launch_bounds__(256)
k_h_finish(const float* __restrict__ h_sum, int64_t n, int reduce, double* __restrict__ h_out,
           double* __restrict__ omega_out, float* __restrict__ H2f, uint4* __restrict__ xq,
           unsigned long long* hminmax) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    double mn = INFINITY, mx = 0.0, h3 = 0.0;
    if (p < n) {
        float H2;
        if (h_sum) {
            const double hd = (double)h_sum[p], H = kKappa * hd;
            H2 = (float)(H * H);
            h3 = H * H * H;
            mn = mx = hd;
            h_out[p] = hd;
            omega_out[p] = kSigma / h3 * ((double)h_sum[n + p] + (double)h_sum[2 * n + p]);
            H2f[p] = H2;
        } else {
            H2 = H2f[p];
        }
        reinterpret_cast<unsigned*>(xq + p)[3] = __float_as_uint(H2);
    }
    if (!h_sum || !reduce) return;
    warp_minmax(mn, mx);
    for (int o = 16; o > 0; o >>= 1) h3 += __shfl_xor_sync(0xffffffffu, h3, o);
    if ((threadIdx.x & 31) == 0 && mx > 0.0) {
        atomic_min_pos(&hminmax[0], mn);
        atomic_max_pos(&hminmax[1], mx);
        atomicAdd(reinterpret_cast<double*>(&hminmax[4]), h3);
    }
}

// Newton on S(h) = S* in double from the float root hd, by the lanes of a group: sums(H, iH, S, D)
// adds this lane's share of S and D = sum q w'(q) = -h dS/dh.  The step after one of less than
// 1e-8 h is exact to rounding, and at the root omega is (eta/h)^3, so two evaluations do, with no
// cube root and two reciprocals: these scalar parts, which a group's lanes all repeat, were
// three quarters of the double instructions in the omega^(-1/3) form.
template <int LN, class F>
__device__ __forceinline__ bool newton_double(const HParams& hp, unsigned group, double& hd, double& om_d, F&& sums) {
    double lod = 0.0, hid = INFINITY;
    for (int it = 0; it < 60; ++it) {
        const double H = kKappa * hd, iH = rcp_fast(H);
        double S = 0.0, D = 0.0;
        sums(H, iH, S, D);
#pragma unroll
        for (int o = LN / 2; o > 0; o >>= 1) {
            S += __shfl_xor_sync(group, S, o);
            D += __shfl_xor_sync(group, D, o);
        }
        const double f = S - hp.s_star;
        if (f < 0.0) lod = hd; else hid = hd;
        const double step = D < 0.0 ? -f * hd * rcp_fast(D) : INFINITY;
        if (fabs(step) <= 1e-8 * hd) {
            hd -= step;
            om_d = hp.eta3 * rcp_fast(hd * hd * hd);
            return true;
        }
        if (hid - lod <= 1e-14 * hd) {
            om_d = kSigma * iH * iH * iH * S;
            return true;
        }
        double hn = hd - step;
        if (it >= 12 || !(hn > lod && hn < hid)) hn = isinf(hid) ? 1.01 * hd : 0.5 * (lod + hid);
        hd = hn;
    }
    return false;
}

// one distance's share of S and D
__device__ __forceinline__ void newton_term(double rr, double iH, double& S, double& D) {
    const double q = rr * iH;
    if (q < 1.0) {
        const double a = 1.0 - q, a2 = a * a;
        double w = a2 * a, d = -3.0 * a2;
        if (q < 0.5) {
            const double b = 0.5 - q, b2 = b * b;
            w -= 4.0 * (b2 * b);
            d += 12.0 * b2;
        }
        S += w;
        D += q * d;
    }
}

// exact distance of candidate j from particle p; beyond the float bound R2f: infinite
struct ExactDist {
    const double* xs;
    const uint4* xq;
    int64_t n;
    double px, py, pz, b0, b1, b2;
    uint4 q;
    float s0, s1, s2;
    int periodic;
    __device__ __forceinline__ ExactDist(const Grid& g, const double* xs_, const uint4* xq_, int64_t n_, const float* sc,
                                         int64_t p)
        : xs(xs_), xq(xq_), n(n_), px(xs_[p]), py(xs_[n_ + p]), pz(xs_[2 * n_ + p]), b0(g.box[0]), b1(g.box[1]),
          b2(g.box[2]), q(xq_[p]), s0(sc[0]), s1(sc[1]), s2(sc[2]), periodic(g.periodic) {}
    __device__ __forceinline__ double operator()(int j, float R2f) const {
        const uint4 qj = xq[j];
        const float ax = fsep(qj.x, q.x, s0), ay = fsep(qj.y, q.y, s1), az = fsep(qj.z, q.z, s2);
        if (ax * ax + ay * ay + az * az >= R2f) return INFINITY;
        const double dx = sep_fast(xs[j], px, b0, 0.5 * b0, periodic);
        const double dy = sep_fast(xs[n + j], py, b1, 0.5 * b1, periodic);
        const double dz = sep_fast(xs[2 * n + j], pz, b2, 0.5 * b2, periodic);
        const double r2 = dx * dx + dy * dy + dz * dz;
        return r2 > 0.0 ? sqrt_fast(r2) : 0.0;
    }
};

// what the double phase leaves behind for particle p
__device__ __forceinline__ void store_refined(int64_t p, bool ok, double hd, double om_d, double* h_out,
                                              double* omega_out, float* H2f_out, uint4* xq_out, int* flags) {
    if (!ok) atomicExch(&flags[F_NOCONV], 1);
    h_out[p] = hd;
    omega_out[p] = om_d;
    const double Hd = kKappa * hd;
    H2f_out[p] = (float)(Hd * Hd);
    reinterpret_cast<unsigned*>(xq_out + p)[3] = __float_as_uint((float)(Hd * Hd));
}
__device__ __forceinline__ void reduce_refined(double mn, double mx, double h3, bool sum, unsigned long long* hminmax) {
    warp_minmax(mn, mx);
    for (int o = 16; o > 0; o >>= 1) h3 += __shfl_xor_sync(0xffffffffu, h3, o);
    if ((threadIdx.x & 31) == 0 && mx > 0.0) {
        atomic_min_pos(&hminmax[0], mn);
        atomic_max_pos(&hminmax[1], mx);
        if (sum) atomicAdd(reinterpret_cast<double*>(&hminmax[4]), h3);
    }
}

// The double phase, LN lanes per particle, from the particle's list: it holds every candidate
// within kNear of the float support, which contains every neighbour of every iterate.  It runs
// for the particles k_h_lists flagged (todo, of arbitrary order; each particle's result depends
// on its own position and neighbours only) or for all of them (FP64, todo NULL), eight lanes
// each, whose repeated scalar parts the double pipe bears; on small sets, where the flagged ones
// are a handful and each a chain of latencies, 32.  The
// distances are dealt to the lanes and kept in registers, SLOTS a lane.  A particle without a
// list, with more neighbours than slots (eta above about 1.55: nearly all; a search of 110,592
// particles at 1.6 in double takes 6.4 ms, 15.6 with a thread each) or with an iterate beyond the
// list goes to `rest`.  The smallest and largest h are widened to the refined values.
template <int LN, int SLOTS>
__global__ void __launch_bounds__(128)
k_h_refine(Grid g, const double* __restrict__ xs, const uint4* __restrict__ xq, int64_t n, HParams hp,
           const int32_t* __restrict__ todo, const int* __restrict__ count, const int32_t* __restrict__ list,
           const int32_t* __restrict__ list_cnt, int cap, double* h_out, double* omega_out, float* H2f_out,
           uint4* xq_out, unsigned long long* hminmax, int* flags, int32_t* rest, int* rest_n) {
    const int lane = threadIdx.x & (LN - 1);
    const unsigned group = LN == 32 ? 0xffffffffu : ((1u << (LN & 31)) - 1u) << (threadIdx.x & 31 & ~(LN - 1));
    const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / LN;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) / LN;
    const int64_t cnt = todo ? (int64_t)*count : n;
    double mn = INFINITY, mx = 0.0, h3 = 0.0;
    for (int64_t t = w0; t < cnt; t += nw) {
        const int64_t p = todo ? (int64_t)todo[t] : t;
        const int have = list_cnt[p];
        double hd = h_out[p], om_d = omega_out[p];
        const double Rc = kKappa * hd * (1.0 + kNear);
        const float Rf = (float)Rc * 1.0001f;
        const ExactDist dist(g, xs, xq, n, hp.scale, p);
        double r[SLOTS];
        int c = 0;
        for (int k = lane; k < have; k += LN) {
            const double rr = dist(list[p * cap + k], Rf * Rf);
            if (rr < Rc) {
#pragma unroll
                for (int u = 0; u < SLOTS; ++u)   // static indices keep r in registers
                    if (u == c) r[u] = rr;
                ++c;
            }
        }
        bool kept = have >= 0 && !__any_sync(group, c > SLOTS);
        bool ok = false;
        if (kept)
            ok = newton_double<LN>(hp, group, hd, om_d, [&](double H, double iH, double& S, double& D) {
                if (H > Rc) kept = false;
#pragma unroll
                for (int k = 0; k < SLOTS; ++k)
                    if (k < c) newton_term(r[k], iH, S, D);
            });
        if (lane != 0) continue;
        if (!kept || kKappa * hd > Rc) {
            rest[atomicAdd(rest_n, 1)] = (int32_t)p;
            continue;
        }
        store_refined(p, ok, hd, om_d, h_out, omega_out, H2f_out, xq_out, flags);
        const double Hd = kKappa * hd;
        mn = fmin(mn, hd);
        mx = fmax(mx, hd);
        h3 += Hd * Hd * Hd;
    }
    reduce_refined(mn, mx, h3, !todo, hminmax);
}

// The double phase of the rest, a warp each: one walk a little beyond the float support, its
// distances in shared memory (kRestDist of them; each evaluation walks where they overflow).
// Such a particle may move far enough that its list, if any, no longer covers it: none is left.
constexpr int kRestDist = 1024, kRestWarps = 4;
__global__ void __launch_bounds__(kRestWarps * 32)
k_h_refine_walk(Grid g, const double* __restrict__ xs, const uint4* __restrict__ xq, int64_t n, HParams hp,
                const int32_t* __restrict__ rest, const int* __restrict__ rest_n, int32_t* list_cnt, double* h_out,
                double* omega_out, float* H2f_out, uint4* xq_out, unsigned long long* hminmax, int sum, int* flags) {
    __shared__ double dists[kRestWarps][kRestDist];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned FULL = 0xffffffffu;
    double* st = dists[wid];
    double mn = INFINITY, mx = 0.0, h3 = 0.0;
    const int cnt = *rest_n, nw = gridDim.x * kRestWarps;
    for (int t = blockIdx.x * kRestWarps + wid; t < cnt; t += nw) {
        const int64_t p = rest[t];
        double hd = h_out[p], om_d = omega_out[p], Rs = 0.0;
        const ExactDist dist(g, xs, xq, n, hp.scale, p);
        const float pxf = (float)dist.px, pyf = (float)dist.py, pzf = (float)dist.pz;
        int c = 0;
        const bool ok = newton_double<32>(hp, FULL, hd, om_d, [&](double H, double iH, double& S, double& D) {
            if (H > Rs) {
                Rs = H * 1.001;
                const float Rf = (float)Rs * 1.0001f;
                c = 0;
                __syncwarp();
                warp_walk(g, pxf, pyf, pzf, Rf, lane, [&](int j, bool valid) {
                    const double rr = valid ? dist(j, Rf * Rf) : INFINITY;
                    const bool in = rr < Rs;
                    const unsigned m = __ballot_sync(FULL, in);
                    const int pos = c + __popc(m & ((1u << lane) - 1u));
                    if (in && pos < kRestDist) st[pos] = rr;
                    c += __popc(m);
                    return c <= kRestDist;
                });
                __syncwarp();
            }
            if (c <= kRestDist) {
                for (int k = lane; k < c; k += 32) newton_term(st[k], iH, S, D);
            } else {
                const float Rf = (float)H * 1.0001f;
                warp_walk(g, pxf, pyf, pzf, Rf, lane, [&](int j, bool valid) {
                    if (valid) newton_term(dist(j, Rf * Rf), iH, S, D);
                    return true;
                });
            }
        });
        if (lane == 0) {
            store_refined(p, ok, hd, om_d, h_out, omega_out, H2f_out, xq_out, flags);
            list_cnt[p] = -1;
            const double Hd = kKappa * hd;
            mn = fmin(mn, hd);
            mx = fmax(mx, hd);
            h3 += Hd * Hd * Hd;
        }
    }
    reduce_refined(mn, mx, h3, sum != 0, hminmax);
}

// Smoothing lengths given by the caller (rt_neighbours_given_h): h_i from h_in (caller order)
// and omega_i = sum_j W(r_ij, h_i) at it, evaluated like the last iteration of the solve (the
// float path: float weights summed in double; the FP64 path: double).  Non-positive or
// non-finite h sets the F_BADH flag.
__global__ void k_h_given(Grid g, const double* __restrict__ xs, const uint4* __restrict__ xq, int64_t n,
                          HParams hp, const double* __restrict__ h_in, const int32_t* __restrict__ perm,
                          double* h_out, double* omega_out, float* H2f_out, unsigned long long* hminmax, int* flags) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool active = p < n;
    double hd = 0.0;
    if (active) {
        hd = h_in[perm[p]];
        if (!(hd > 0.0) || !(hd < (double)hp.h_cap) || !isfinite(hd)) {
            atomicExch(&flags[F_BADH], 1);
            hd = hp.h0;
        }
        const uint4 q4p = xq[p];
        const uint32_t qx = q4p.x, qy = q4p.y, qz = q4p.z;
        const double px = xs[p], py = xs[n + p], pz = xs[2 * n + p];
        const float pxf = (float)px, pyf = (float)py, pzf = (float)pz;
        const double H = kKappa * hd, iH = 1.0 / H, H2 = H * H;
        double sw = 0.0;
        if (hp.refine64) {
            const double half[3] = {0.5 * g.box[0], 0.5 * g.box[1], 0.5 * g.box[2]};
            const float Hf = (float)H * 1.001f, H2f = Hf * Hf;
            for_each_candidate(g, pxf, pyf, pzf, Hf, [&](int j) {
                float dxf = fsep(xq[j].x, qx, hp.scale[0]);
                float dyf = fsep(xq[j].y, qy, hp.scale[1]);
                float dzf = fsep(xq[j].z, qz, hp.scale[2]);
                if (dxf * dxf + dyf * dyf + dzf * dzf >= H2f) return;
                double dx = sep_fast(xs[j], px, g.box[0], half[0], g.periodic);
                double dy = sep_fast(xs[n + j], py, g.box[1], half[1], g.periodic);
                double dz = sep_fast(xs[2 * n + j], pz, g.box[2], half[2], g.periodic);
                double r2 = dx * dx + dy * dy + dz * dz;
                if (r2 < H2) sw += spline_w(sqrt(r2) * iH);
            });
        } else {
            const float Hf = (float)H, iHf = 1.f / Hf, H2f = Hf * Hf;
            for_each_candidate(g, pxf, pyf, pzf, Hf, [&](int j) {
                float dx = fsep(xq[j].x, qx, hp.scale[0]);
                float dy = fsep(xq[j].y, qy, hp.scale[1]);
                float dz = fsep(xq[j].z, qz, hp.scale[2]);
                float r2 = dx * dx + dy * dy + dz * dz;
                if (r2 < H2f) sw += (double)spline_w(sqrtf(r2) * iHf);
            });
        }
        h_out[p] = hd;
        omega_out[p] = kSigma * iH * iH * iH * sw;
        H2f_out[p] = (float)(H * H);
    }
    double mn = active ? hd : INFINITY, mx = active ? hd : 0.0;
    warp_minmax(mn, mx);
    double h3 = active ? (kKappa * hd) * (kKappa * hd) * (kKappa * hd) : 0.0;
    for (int o = 16; o > 0; o >>= 1) h3 += __shfl_xor_sync(0xffffffffu, h3, o);
    if ((threadIdx.x & 31) == 0 && mx > 0.0) {
        atomic_min_pos(&hminmax[0], mn);
        atomic_max_pos(&hminmax[1], mx);
        atomicAdd(reinterpret_cast<double*>(&hminmax[4]), h3);
    }
}

// ------------------------------------------------------------------------------------
// a3: symmetric pair lists { j != i : r_ij < max(H_i, H_j) }.  A float test on the
// fixed-point separation decides all pairs except those within 1e-5 of the threshold,
// which are decided by the exact double test (r^2 and H^2 without contraction).
//
// Each particle looks only inside its own support: its list of candidates, or a walk where
// that overflowed.  An entry (i, j) that j does not have in its own support (H_j <= r < H_i) is
// handed to row j as an extra; the row is its own entries merged with its extras, in
// ascending order whatever order the extras arrived in.  Searching out to the largest H_j that
// could reach i instead visits 2.5 times the candidates (0.43 ms on 262,144 particles), and
// on strongly clustered sets no bound is local enough: there every entry and its transpose
// were sorted as 64-bit keys (7.8 of 15.6 ms on 1,000,000 particles).
struct PairParams {
    float scale[3];
};

// extra entries carry this bit beside their index (particle numbers stay below 2^31)
constexpr uint32_t kAsym = 0x80000000u;

// the exact double test of r_pj < H_k (no contraction), as a plain double evaluation would do it;
// a call, because it is rare and its registers would halve the occupancy of the search
__device__ __noinline__ bool inside_exact(const double* __restrict__ xs, double hk, int64_t n, double b0, double b1,
                                          double b2, int periodic, int64_t p, int j) {
    const double H = __dmul_rn(kKappa, hk);
    const double ex = sep_exact(xs[j], xs[p], b0, periodic);
    const double ey = sep_exact(xs[n + j], xs[n + p], b1, periodic);
    const double ez = sep_exact(xs[2 * n + j], xs[2 * n + p], b2, periodic);
    return norm2_exact(ex, ey, ez) < __dmul_rn(H, H);
}

// is r_pj < H of the particle whose float H^2 is H2 and whose h is h[k]?
__device__ __forceinline__ bool inside(const Grid& g, const double* __restrict__ xs, const double* __restrict__ h,
                                       int64_t n, float r2, float H2, int64_t k, int64_t p, int j) {
    if (r2 < H2 * (1.f - 1e-5f)) return true;
    if (r2 > H2 * (1.f + 1e-5f)) return false;
    return inside_exact(xs, h[k], n, g.box[0], g.box[1], g.box[2], g.periodic, p, j);
}

// candidate j of particle p (the whole warp calls): own entry?  asym: not one of j's own
__device__ __forceinline__ bool own_entry(const Grid& g, const double* __restrict__ xs, const uint4* __restrict__ xq,
                                          const double* __restrict__ h, int64_t n, const PairParams& pp, int64_t p,
                                          const uint4& qp, int j, bool valid, bool& asym) {
    asym = false;
    if (!valid || j == p) return false;
    const uint4 qj = xq[j];
    const float dx = fsep(qj.x, qp.x, pp.scale[0]);
    const float dy = fsep(qj.y, qp.y, pp.scale[1]);
    const float dz = fsep(qj.z, qp.z, pp.scale[2]);
    const float r2 = dx * dx + dy * dy + dz * dz;
    if (!inside(g, xs, h, n, r2, __uint_as_float(qp.w), p, p, j)) return false;
    asym = !inside(g, xs, h, n, r2, __uint_as_float(qj.w), j, p, j);
    return true;
}

// extras that a row holds in place; a row that gets more has them filled in a second pass
constexpr int kExtras = 64;

// hands the asymmetric entry (p, j) to row j
__device__ __forceinline__ void hand_extra(int32_t* extra, int32_t* extras, int64_t p, int j) {
    const int k = atomicAdd(&extra[j], 1);
    if (k < kExtras) extras[(int64_t)j * kExtras + k] = (int32_t)p;
}

// One warp per particle: own entries, with their asymmetry bit, over the front of the list
// (each round's reads come before its writes, which lie no further back); their number; and the
// extras of the other rows.  Two rounds of 32 candidates are in flight together.  Particles
// without a list go to `over`, for k_own_walk.
__global__ void __launch_bounds__(256, 5)
k_own_rows(Grid g, const double* __restrict__ xs, const uint4* __restrict__ xq, const double* __restrict__ h,
           int64_t n, PairParams pp, int32_t* list, int cap, const int32_t* __restrict__ list_cnt,
           int32_t* __restrict__ own, int32_t* extra, int32_t* __restrict__ extras, int32_t* over, int* over_n) {
    const int64_t p = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (p >= n) return;
    const int had = list_cnt[p];
    if (had < 0) {
        if (lane == 0) over[atomicAdd(over_n, 1)] = (int32_t)p;
        return;
    }
    const uint4 qp = xq[p];
    int32_t* row = list + p * cap;
    int c = 0;
    for (int t0 = 0; t0 < had; t0 += 64) {
        int j[2];
        bool in[2], asym[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int t = t0 + 32 * u + lane;
            j[u] = t < had ? row[t] : (int)p;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) in[u] = own_entry(g, xs, xq, h, n, pp, p, qp, j[u], true, asym[u]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const unsigned m = __ballot_sync(0xffffffffu, in[u]);
            if (in[u]) {
                row[c + __popc(m & ((1u << lane) - 1u))] = (int32_t)((uint32_t)j[u] | (asym[u] ? kAsym : 0u));
                if (asym[u]) hand_extra(extra, extras, p, j[u]);
            }
            c += __popc(m);
        }
    }
    if (lane == 0) own[p] = c;
}

// The particles without a list, by walks, a warp each: their number of own entries, with room
// for them reserved in the spill (its offset goes to the unused list); FILL writes them there.
template <bool FILL>
__global__ void __launch_bounds__(128)
k_own_walk(Grid g, const double* __restrict__ xs, const uint4* __restrict__ xq, const double* __restrict__ h,
           int64_t n, PairParams pp, int32_t* list, int cap, int32_t* __restrict__ own, int32_t* extra,
           int32_t* __restrict__ extras, const int32_t* __restrict__ over, const int* __restrict__ over_n,
           unsigned long long* spill_n, int32_t* __restrict__ spill) {
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5, m = *over_n;
    for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < m; w += nw) {
        const int64_t p = over[w];
        const uint4 qp = xq[p];
        unsigned long long* where = reinterpret_cast<unsigned long long*>(list + p * cap);
        int32_t* out = FILL ? spill + *where : nullptr;
        int c = 0;
        warp_walk(g, (float)qp.x * pp.scale[0], (float)qp.y * pp.scale[1], (float)qp.z * pp.scale[2],
                  sqrtf(__uint_as_float(qp.w)) * 1.0001f, lane, [&](int j, bool valid) {
                      bool asym;
                      const bool in = own_entry(g, xs, xq, h, n, pp, p, qp, j, valid, asym);
                      const unsigned b = __ballot_sync(0xffffffffu, in);
                      if (in) {
                          if (FILL) out[c + __popc(b & ((1u << lane) - 1u))] = (int32_t)((uint32_t)j | (asym ? kAsym : 0u));
                          else if (asym) hand_extra(extra, extras, p, j);
                      }
                      c += __popc(b);
                      return true;
                  });
        if (!FILL && lane == 0) {
            own[p] = c;
            *where = atomicAdd(spill_n, (unsigned long long)c);
        }
    }
}

// row lengths, own entries and extras; and how many extras the rows have that hold more than
// kExtras (their offsets come from a scan, their sum decides whether the second pass runs)
__global__ void k_row_lengths(const int32_t* __restrict__ own, const int32_t* __restrict__ extra, int64_t n,
                              int32_t* __restrict__ counts, unsigned long long* more) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p > n) return;
    const int e = p < n ? extra[p] : 0;
    counts[p] = p < n ? own[p] + e : 0;
    if (e > kExtras) atomicAdd(more, (unsigned long long)e);
}
__global__ void k_more_extras(const int32_t* __restrict__ extra, int64_t n, int32_t* __restrict__ more) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p <= n) more[p] = p < n && extra[p] > kExtras ? extra[p] : 0;
}

// second pass for those rows: every asymmetric entry (p, j) again, any order
__global__ void __launch_bounds__(256)
k_extras_fill(int64_t n, const int32_t* __restrict__ list, int cap, const int32_t* __restrict__ list_cnt,
              const int32_t* __restrict__ own, const int32_t* __restrict__ extra, const int64_t* __restrict__ off,
              int32_t* fill, const int32_t* __restrict__ spill, int32_t* __restrict__ out) {
    const int64_t p = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (p >= n) return;
    const int32_t* row = list + p * cap;
    if (list_cnt[p] < 0) row = spill + *reinterpret_cast<const unsigned long long*>(row);
    for (int t = lane; t < own[p]; t += 32) {
        const uint32_t v = (uint32_t)row[t];
        if (!(v & kAsym)) continue;
        const int j = (int)(v & ~kAsym);
        if (extra[j] > kExtras) out[off[j] + atomicAdd(&fill[j], 1)] = (int32_t)p;
    }
}

// Row p: own entries (ascending) merged with its extras (any order) by rank, one warp per row; and
// the row's split into lower neighbours j < p and upper ones j > p.  Each unordered pair is the
// upper entry of its lower particle; slot(i, j) numbers those entries.
__global__ void __launch_bounds__(256)
k_rows_merge(int64_t n, const int32_t* __restrict__ list, int cap, const int32_t* __restrict__ list_cnt,
             const int32_t* __restrict__ own, const int32_t* __restrict__ extra, const int32_t* __restrict__ extras,
             const int64_t* __restrict__ more_off, const int32_t* __restrict__ more,
             const int32_t* __restrict__ spill, const int64_t* __restrict__ row_off, int32_t* __restrict__ cols,
             int32_t* __restrict__ n_low, int32_t* __restrict__ n_up) {
    const int64_t p = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (p >= n) return;
    const int32_t* row = list + p * cap;
    if (list_cnt[p] < 0) row = spill + *reinterpret_cast<const unsigned long long*>(row);
    const int m = own[p], E = extra[p];
    const int32_t* ex = E > kExtras ? more + more_off[p] : extras + p * kExtras;
    int32_t* out = cols + row_off[p];
    int low = 0;
    auto below = [&](int v) {     // extras smaller than v
        int c = 0;
        for (int k = 0; k < E; ++k) c += ex[k] < v ? 1 : 0;
        return c;
    };
    for (int t = lane; t < m; t += 32) {
        const int v = (int)((uint32_t)row[t] & ~kAsym);
        low += v < p ? 1 : 0;
        out[t + below(v)] = v;
    }
    for (int k = lane; k < E; k += 32) {
        const int v = ex[k];
        low += v < p ? 1 : 0;
        int b = 0, e = m;         // own entries smaller than v
        while (b < e) {
            const int u = (b + e) >> 1;
            if ((int)((uint32_t)row[u] & ~kAsym) < v) b = u + 1; else e = u;
        }
        out[b + below(v)] = v;
    }
    low = __reduce_add_sync(0xffffffffu, low);
    if (lane == 0) {
        n_low[p] = low;
        n_up[p] = m + E - low;
    }
}

// The two particles of every pair slot, and for every lower entry (i, k), k < i, the slot of the
// pair in k's upper list.  One warp per particle k, its lanes taking the upper entries: the
// slots are written side by side, and k's place among the lower entries of each l is found by a
// binary search.
__global__ void __launch_bounds__(256)
k_pair_slots(const int64_t* __restrict__ row_off, const int32_t* __restrict__ cols,
             const int32_t* __restrict__ n_low, const int64_t* __restrict__ up_off, int64_t n,
             int2* __restrict__ ends, int32_t* __restrict__ low_slot) {
    const int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (k >= n) return;
    const int64_t e0 = row_off[k] + n_low[k], s0 = up_off[k];
    const int m = (int)(up_off[k + 1] - s0);
    for (int t = lane; t < m; t += 32) {
        const int l = cols[e0 + t];
        const int64_t slot = s0 + t, r = row_off[l];
        ends[slot] = make_int2((int)k, l);
        const int32_t* row = cols + r;
        int b = 0, e = n_low[l];
        while (b < e) {
            const int u = (b + e) >> 1;
            if (row[u] < (int32_t)k) b = u + 1; else e = u;
        }
        low_slot[r - up_off[l] + b] = (int32_t)slot;      // r - up_off[l]: lower entries before row l
    }
}

// ------------------------------------------------------------------------------------
// a4: E_i = sum_j psi_j(x_i) d d^T, B_i = E_i^-1 (double), and the per-particle factors used
// by the pair kernels.
template <class T>
__device__ __forceinline__ void sym3_eigs(T a, T b, T c, T d, T e, T f, T ev[3]) {
    // symmetric [[a d e][d b f][e f c]]: trigonometric closed form
    const T p1 = d * d + e * e + f * f;
    const T q = (a + b + c) / T(3);
    if (p1 == T(0)) { ev[0] = a; ev[1] = b; ev[2] = c; return; }
    const T p2 = (a - q) * (a - q) + (b - q) * (b - q) + (c - q) * (c - q) + T(2) * p1;
    const T p = sqrt(p2 / T(6));
    const T ip = T(1) / p;
    const T B00 = (a - q) * ip, B11 = (b - q) * ip, B22 = (c - q) * ip, B01 = d * ip, B02 = e * ip, B12 = f * ip;
    const T detB = B00 * (B11 * B22 - B12 * B12) - B01 * (B01 * B22 - B12 * B02) + B02 * (B01 * B12 - B11 * B02);
    const T phi = acos(fmin_(fmax_(detB / T(2), T(-1)), T(1))) / T(3);
    ev[0] = q + T(2) * p * cos(phi);
    ev[2] = q + T(2) * p * cos(phi + T(2.0943951023931954923));
    ev[1] = T(3) * q - ev[0] - ev[2];
}

// cond_2 from the float eigenvalues of E / tr E (exact to 1e-6 cond) serves all but the largest
// of the set and those above kCondFloat, whose value is taken in double (k_cond): the double
// closed form, an arccosine and two cosines, was most of the geometry's double instructions.
constexpr float kCondFloat = 1e3f;

template <class T>
__device__ __forceinline__ void store_pos(void* pos, int64_t p, const double* xs, const uint4* xq, int64_t n);
template <>
__device__ __forceinline__ void store_pos<float>(void* pos, int64_t p, const double*, const uint4* xq, int64_t n) {
    reinterpret_cast<uint4*>(pos)[p] = xq[p];
}
template <>
__device__ __forceinline__ void store_pos<double>(void* pos, int64_t p, const double* xs, const uint4*, int64_t n) {
    double2* d = reinterpret_cast<double2*>(pos) + 2 * p;
    d[0] = make_double2(xs[p], xs[n + p]);
    d[1] = make_double2(xs[2 * n + p], 0.0);
}

// E_i accumulation over the pair list.  Double path: separations and weights in double.
// Float path: separations from the fixed-point positions, weights in float and a
// compensated (Kahan) float sum, so that E_i keeps ~1e-8 relative accuracy before its
// inversion in double.
//
// E_i, LN lanes a row: eight on the double path's sets too small to fill the GPU with one (a row of 46
// then takes six rounds of loads), else one.  The float path always takes one: its compensated
// sums round at 1e-8 by the order of the row, and E_i is to be the same for every size of set.
struct Sum {
    double v = 0.0;
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void fold(int o) { v += __shfl_xor_sync(0xffffffffu, v, o); }
    __device__ __forceinline__ double value() const { return v; }
};
template <class T, int LN>
__global__ void __launch_bounds__(256)
k_E(const double* __restrict__ xs, const uint4* __restrict__ xq, const double* __restrict__ h,
    const int64_t* __restrict__ row_off, const int32_t* __restrict__ cols, int64_t n, double b0, double b1, double b2,
    int periodic, float s0, float s1, float s2, double* __restrict__ E_out) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t p = t / LN;
    const int lane = (int)(t % LN);
    const bool act = p < n;
    const int64_t pp = act ? p : 0, e1 = act ? row_off[pp + 1] : 0;
    const double H = kKappa * h[pp];
    typename std::conditional<std::is_same<T, float>::value, Kahan, Sum>::type acc[6];
    if constexpr (std::is_same<T, float>::value) {
        const uint4 q = xq[pp];
        const float iH = (float)(1.0 / H), H2 = (float)(H * H);
#pragma unroll 2
        for (int64_t e = row_off[pp] + lane; e < e1; e += LN) {
            const uint4 qj = xq[cols[e]];
            const float dx = fsep(qj.x, q.x, s0), dy = fsep(qj.y, q.y, s1), dz = fsep(qj.z, q.z, s2);
            const float r2 = dx * dx + dy * dy + dz * dz;
            if (!(r2 < H2)) continue;
            const float w = spline_w(sqrtf(r2) * iH);
            acc[0].add(w * dx * dx); acc[1].add(w * dy * dy); acc[2].add(w * dz * dz);
            acc[3].add(w * dx * dy); acc[4].add(w * dx * dz); acc[5].add(w * dy * dz);
        }
    } else {
        const double x = xs[pp], y = xs[n + pp], z = xs[2 * n + pp];
        const double iH = 1.0 / H, H2 = H * H;
        for (int64_t e = row_off[pp] + lane; e < e1; e += LN) {
            const int j = cols[e];
            const double dx = sep_fast(xs[j], x, b0, 0.5 * b0, periodic);
            const double dy = sep_fast(xs[n + j], y, b1, 0.5 * b1, periodic);
            const double dz = sep_fast(xs[2 * n + j], z, b2, 0.5 * b2, periodic);
            const double r2 = dx * dx + dy * dy + dz * dz;
            if (!(r2 < H2)) continue;
            const double w = r2 > 0.0 ? spline_w(sqrt_fast(r2) * iH) : 0.0;
            const double wx = w * dx, wy = w * dy, wz = w * dz;
            acc[0].add(wx * dx); acc[1].add(wy * dy); acc[2].add(wz * dz);
            acc[3].add(wx * dy); acc[4].add(wx * dz); acc[5].add(wy * dz);
        }
    }
    if constexpr (LN == 1) {
        if (!act) return;
#pragma unroll
        for (int k = 0; k < 6; ++k) E_out[k * n + p] = acc[k].value();
    } else {
#pragma unroll
        for (int o = LN / 2; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < 6; ++k) acc[k].fold(o);
        if (!act || lane >= 6) return;
        double v = 0.0;
#pragma unroll
        for (int k = 0; k < 6; ++k) v = k == lane ? acc[k].value() : v;
        E_out[lane * n + p] = v;
    }
}

// Also writes the pair kernels' records: position, {1/H, h, Bp (6)} with
// Bp = V^2 sigma / H^3 B (so that V_i psitilde_j(x_i) = Bp_i d w(q)), and omega; reduces
// max cond_2(E_i) and min V_i into red[2], red[3].
template <class T>
__global__ void k_geometry(const double* __restrict__ xs, const uint4* __restrict__ xq,
                           const double* __restrict__ h, const double* __restrict__ omega,
                           int64_t n, double* V_out, double* B_out, float* cond_out, void* pos_t, T* geo_t, T* om_t,
                           unsigned long long* red, unsigned* cond_max, int* flags) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    float cond = 0.f;
    double V = INFINITY;
    if (p < n) {
        double hi = h[p], H = kKappa * hi, iH = 1.0 / H;
        double om = omega[p];
        double E[6];
        for (int k = 0; k < 6; ++k) E[k] = B_out[k * n + p];     // E_i (k_E), replaced by B_i
        V = 1.0 / om;                              // V, 1/H and bp as in k_set_fields
        const double fac = kSigma * iH * iH * iH * V;   // psi = fac * w
        double e_xx = E[0] * fac, e_yy = E[1] * fac, e_zz = E[2] * fac;
        double e_xy = E[3] * fac, e_xz = E[4] * fac, e_yz = E[5] * fac;
        // cofactor inverse of the symmetric matrix
        double c_xx = e_yy * e_zz - e_yz * e_yz;
        double c_xy = e_xz * e_yz - e_xy * e_zz;
        double c_xz = e_xy * e_yz - e_xz * e_yy;
        double det = e_xx * c_xx + e_xy * c_xy + e_xz * c_xz;
        V_out[p] = V;
        store_pos<T>(pos_t, p, xs, xq, n);
        if (!(det > 0.0) || !(om > 0.0)) {
            atomicExch(&flags[F_GEOM], 1);
            for (int k = 0; k < 6; ++k) B_out[k * n + p] = 0.0;
            for (int k = 0; k < 8; ++k) geo_t[8 * p + k] = (T)0;
            om_t[p] = (T)0;
            cond_out[p] = 0.f;     // the call fails
        } else {
            const double id = rcp_fast(det);
            double B[6];
            B[0] = c_xx * id;
            B[1] = (e_xx * e_zz - e_xz * e_xz) * id;
            B[2] = (e_xx * e_yy - e_xy * e_xy) * id;
            B[3] = c_xy * id;
            B[4] = c_xz * id;
            B[5] = (e_xy * e_xz - e_xx * e_yz) * id;
            const float it = 1.f / (float)(e_xx + e_yy + e_zz);
            float ev[3];
            sym3_eigs((float)e_xx * it, (float)e_yy * it, (float)e_zz * it, (float)e_xy * it, (float)e_xz * it,
                      (float)e_yz * it, ev);
            const float lmin = fminf(ev[0], fminf(ev[1], ev[2])), lmax = fmaxf(ev[0], fmaxf(ev[1], ev[2]));
            cond = lmin > 0.f ? lmax / lmin : INFINITY;
            cond_out[p] = cond;
            const double bp = V * V * kSigma * iH * iH * iH;   // V_i psitilde_j(x_i) = Bp_i d w(q_ij)
            geo_t[8 * p] = (T)iH;
            geo_t[8 * p + 1] = (T)hi;
            for (int k = 0; k < 6; ++k) {
                B_out[k * n + p] = B[k];
                geo_t[8 * p + 2 + k] = (T)(bp * B[k]);
            }
            om_t[p] = (T)om;
        }
    }
    // largest float condition number (non-negative floats order like integers) and smallest V
    const unsigned cm = __reduce_max_sync(0xffffffffu, __float_as_uint(cond));
    for (int o = 16; o > 0; o >>= 1) V = fmin(V, __shfl_xor_sync(0xffffffffu, V, o));
    if ((threadIdx.x & 31) == 0) {
        if (cm) atomicMax(cond_max, cm);
        if (V < INFINITY) atomic_min_pos(&red[3], V);
    }
}

// cond_2(E_i) = cond_2(B_i) in double where the float value is within 2% of the largest or above
// kCondFloat: the largest, the ill-conditioned ones, and a last check that E_i is positive definite
__global__ void k_cond(const float* __restrict__ cond, const double* __restrict__ B, int64_t n,
                       const unsigned* __restrict__ cond_max, unsigned long long* red, int* flags) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n || !(cond[p] >= fminf(0.98f * __uint_as_float(*cond_max), kCondFloat))) return;
    double ev[3];
    sym3_eigs(B[p], B[n + p], B[2 * n + p], B[3 * n + p], B[4 * n + p], B[5 * n + p], ev);
    const double lmin = fmin(ev[0], fmin(ev[1], ev[2])), lmax = fmax(ev[0], fmax(ev[1], ev[2]));
    const double c = lmin > 0 ? lmax / lmin : INFINITY;
    if (!(lmin > 0)) atomicExch(&flags[F_GEOM], 1);
    if (c > 1e10) atomicAdd(&flags[F_ILL], 1);
    atomic_max_pos(&red[2], c);
}

// ------------------------------------------------------------------------------------
// a5 preparation: per source, h_s = eta_s omega_s(h_s)^(-1/3) over gas only (no self term),
// octant sums w_a of psi, mu_a = sum_b w_b / (q_nz w_a), xi = mu_a psi.  One warp per source.
__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The sources' positions as the searches take them.  A periodic one is wrapped into the box, from
// a cell of which the walks start, and whose fixed point the float test measures from (the
// separations themselves wrap once more).  Without walls a source may lie outside.  One that is not
// finite ends the call (F_BADPOS) and is searched from 0 until then.
__global__ void k_src_positions(const double* __restrict__ x, int64_t S, Box b, double* __restrict__ out, int* flags) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= 3 * S) return;
    const double L = b.box[t / S];
    double v = x[t];
    if (!isfinite(v)) {
        atomicExch(&flags[F_BADPOS], 1);
        v = 0.0;
    } else if (b.periodic && !(v >= 0.0 && v <= L)) {
        v = fmin(fmax(v - L * floor(v / L), 0.0), L);
    }
    out[t] = v;
}

struct SrcParams {
    double s_star, eta3, h0, h_cap;   // (kappa eta)^3 / sigma and eta^3 of the sources' eta
    int max_iter;
    int warm;       // start from the h of the last call (in hs_out), else from h0
    int fixed;      // hs_out holds given smoothing lengths: only omega_s at them
};

// One step of the source solve from the sums at h: S(h) = sum w, D = sum q w'(q).  Newton on
// S(h) = S* (see k_h_lists) close to the root, where a step of less than 1e-8 h ends it: the
// next one would be below rounding, and at the root omega is (eta/h)^3.  Farther off on h - eta
// omega^(-1/3), nearly linear in h.  Returns 1 when done, 0 for another evaluation at the new h,
// -1 when h cannot move.
__device__ __forceinline__ int src_newton(const SrcParams& sp, double S, double D, double& h, double& lo, double& hi,
                                          double& om) {
    const double f = S - sp.s_star;
    if (f < 0.0) lo = h; else hi = h;
    double step = -INFINITY;
    if (S > 0.0 && D < 0.0) {
        if (fabs(f) < 1e-3 * sp.s_star) {
            step = -f * h / D;
        } else {
            const double x = cbrt(sp.s_star / S), fp = 1.0 - x - x * D / (3.0 * S);
            step = fp > 0.0 ? h * (1.0 - x) / fp : -INFINITY;
        }
    }
    if (fabs(step) <= 1e-8 * h) {
        h -= step;
        om = sp.eta3 / (h * h * h);
        return 1;
    }
    double hn = h - step;
    if (!(hn > lo && hn < hi)) hn = isinf(hi) ? 1.5 * h : 0.5 * (lo + hi);
    if (hn > sp.h_cap) hn = sp.h_cap;
    if (hn == h) return om > 0.0 ? 1 : -1;
    h = hn;
    return 0;
}

// Sources with a list of candidates (kSrcList of them within 1.1 supports, about 64 of an even
// set): one warp each walks once (warp_walk) and iterates over the stored distances; the count
// and the entries then come from the list.  A source whose candidates overflow it keeps
// src_list_cnt = -1 and goes to k_src_h and k_src_entries, which walk.  One source in 4,096
// particles: 46 + 18 + 43 us with a block of walks per iteration and two more for the entries.
constexpr int kSrcList = 384, kSrcListWarps = 4;

struct QuantParams {
    double mul[3];      // fixed-point units per length, as in k_gather_positions
    float scale[3];
};

__global__ void __launch_bounds__(kSrcListWarps * 32)
k_src_lists(Grid g, const double* __restrict__ xs, const uint4* __restrict__ xq, int64_t n, QuantParams qp,
            const double* __restrict__ xsrc, int64_t S, SrcParams sp, double* hs_out, double* oms_out, int* flags,
            int32_t* __restrict__ list, int32_t* __restrict__ list_cnt) {
    __shared__ double dist[kSrcListWarps][kSrcList];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t s_id = blockIdx.x * (int64_t)kSrcListWarps + wid;
    if (s_id >= S) return;      // whole warps
    const unsigned FULL = 0xffffffffu;
    const double p[3] = {xsrc[s_id], xsrc[S + s_id], xsrc[2 * S + s_id]};
    uint32_t q[3];
    for (int a = 0; a < 3; ++a) q[a] = (uint32_t)fmin(fmax(floor(p[a] * qp.mul[a]), 0.0), 4294967295.0);
    const double half[3] = {0.5 * g.box[0], 0.5 * g.box[1], 0.5 * g.box[2]};
    double h = (sp.warm || sp.fixed) ? hs_out[s_id] : sp.h0, lo = 0.0, hi = INFINITY, om = 0.0, Rs = 0.0;
    if (!(h > 0.0) || !(h < sp.h_cap)) {
        if (sp.fixed && lane == 0) atomicExch(&flags[F_BADH], 1);
        h = sp.h0;
    }
    int c = 0, state = 0;
    for (int it = 0; it < sp.max_iter && state == 0; ++it) {
        const double H = kKappa * h, iH = 1.0 / H;
        if (H > Rs) {
            Rs = H * (sp.fixed ? 1.0 : 1.1);
            const double R2 = Rs * Rs;
            const float R2f = (float)R2 * 1.001f;
            c = 0;
            warp_walk(g, (float)p[0], (float)p[1], (float)p[2], (float)Rs * 1.0001f, lane, [&](int j, bool valid) {
                double r2 = INFINITY;
                if (valid) {
                    const uint4 qj = xq[j];
                    const float ax = fsep(qj.x, q[0], qp.scale[0]), ay = fsep(qj.y, q[1], qp.scale[1]),
                                az = fsep(qj.z, q[2], qp.scale[2]);
                    if (ax * ax + ay * ay + az * az < R2f) {
                        const double dx = sep_fast(xs[j], p[0], g.box[0], half[0], g.periodic);
                        const double dy = sep_fast(xs[n + j], p[1], g.box[1], half[1], g.periodic);
                        const double dz = sep_fast(xs[2 * n + j], p[2], g.box[2], half[2], g.periodic);
                        r2 = dx * dx + dy * dy + dz * dz;
                    }
                }
                const bool in = r2 < R2;
                const unsigned m = __ballot_sync(FULL, in);
                const int pos = c + __popc(m & ((1u << lane) - 1u));
                if (in && pos < kSrcList) {
                    list[s_id * kSrcList + pos] = j;
                    dist[wid][pos] = sqrt(r2);
                }
                c += __popc(m);
                return c <= kSrcList;
            });
            if (c > kSrcList) {
                if (lane == 0) list_cnt[s_id] = -1;
                return;      // hs_out keeps the first guess for k_src_h
            }
            __syncwarp();
        }
        double sw = 0.0, sdw = 0.0;
        for (int k = lane; k < c; k += 32) {
            const double u = dist[wid][k] * iH;
            sw += spline_w(u);
            sdw += u * spline_dw(u);
        }
        for (int o = 16; o > 0; o >>= 1) {
            sw += __shfl_xor_sync(FULL, sw, o);
            sdw += __shfl_xor_sync(FULL, sdw, o);
        }
        om = kSigma * iH * iH * iH * sw;
        if (sp.fixed) {   // given h: omega there, no iteration
            state = om > 0.0 ? 1 : -1;
            break;
        }
        state = src_newton(sp, sw, sdw, h, lo, hi, om);
    }
    if (lane == 0) {
        if (state != 1) atomicExch(&flags[F_SRC_NOCONV], 1);
        hs_out[s_id] = h;
        oms_out[s_id] = om;
        // the last step moves h by less than 1e-8: the list, a tenth longer or exact, covers it
        // unless it ends right at the support
        list_cnt[s_id] = kKappa * h <= Rs ? c : -1;
    }
}

// Count (FILL = false) or write (FILL = true) the gas entries of the sources with a list, one warp
// each; the counterpart of k_src_entries
template <bool FILL>
__global__ void __launch_bounds__(kSrcListWarps * 32)
k_src_list_entries(Grid g, const double* __restrict__ xs, int64_t n, const double* __restrict__ xsrc, int64_t S,
                   const double* __restrict__ hs, const double* __restrict__ oms, const int32_t* __restrict__ list,
                   const int32_t* __restrict__ list_cnt, int32_t* counts, const int64_t* __restrict__ off,
                   int32_t* e_gas, double* e_xi, double* octw_out, const double* __restrict__ octw_given) {
    __shared__ unsigned char oct_of[kSrcListWarps][kSrcList];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t src = blockIdx.x * (int64_t)kSrcListWarps + wid;
    if (src >= S || list_cnt[src] < 0) return;
    const unsigned FULL = 0xffffffffu;
    const double p[3] = {xsrc[src], xsrc[S + src], xsrc[2 * S + src]};
    const double half[3] = {0.5 * g.box[0], 0.5 * g.box[1], 0.5 * g.box[2]};
    const double H = kKappa * hs[src], iH = 1.0 / H, H2 = H * H, fac = kSigma * iH * iH * iH / oms[src];
    const int m = list_cnt[src];
    const int64_t base = FILL ? off[src] : 0;
    double w8[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int c = 0;
    for (int t0 = 0; t0 < m; t0 += 32) {
        const int t = t0 + lane;
        bool in = false;
        int j = 0, oct = 0;
        double ps = 0.0;
        if (t < m) {
            j = list[src * kSrcList + t];
            const double dx = sep_fast(xs[j], p[0], g.box[0], half[0], g.periodic);
            const double dy = sep_fast(xs[n + j], p[1], g.box[1], half[1], g.periodic);
            const double dz = sep_fast(xs[2 * n + j], p[2], g.box[2], half[2], g.periodic);
            const double r2 = dx * dx + dy * dy + dz * dz;
            in = r2 < H2;
            if (FILL && in) {
                ps = fac * spline_w(sqrt(r2) * iH);
                oct = (dx < 0 ? 1 : 0) | (dy < 0 ? 2 : 0) | (dz < 0 ? 4 : 0);
            }
        }
        const unsigned b = __ballot_sync(FULL, in);
        if (FILL && in) {
            const int pos = c + __popc(b & ((1u << lane) - 1u));
            e_gas[base + pos] = j;
            e_xi[base + pos] = ps;
            oct_of[wid][pos] = (unsigned char)oct;
#pragma unroll
            for (int a = 0; a < 8; ++a) w8[a] += a == oct ? ps : 0.0;
        }
        c += __popc(b);
    }
    if (!FILL) {
        if (lane == 0) counts[src] = c;
        return;
    }
    // octant sums; xi = mu_a psi, mu_a = sum_b w_b / (q_nz w_a)
    double wsum = 0.0;
    int qnz = 0;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        w8[a] = octw_given ? octw_given[8 * src + a] : warp_sum(w8[a]);
        wsum += w8[a];
        qnz += (w8[a] > 0.0);
        if (lane == 0) octw_out[8 * src + a] = w8[a];
    }
    __syncwarp();
    const double share = wsum / (double)qnz;
    for (int e = lane; e < c; e += 32) {
        const int oct = oct_of[wid][e];
        double w = 0.0;
#pragma unroll
        for (int a = 0; a < 8; ++a) w = a == oct ? w8[a] : w;
        e_xi[base + e] = share / w * e_xi[base + e];
    }
}

// Rows of the culled walk of for_each_candidate handed out round-robin to the threads of a
// block (thread t takes rows t, t + nt, ...).
template <class F>
__device__ __forceinline__ void strided_rows(const Grid& g, float px, float py, float pz, float R, int t, int nt,
                                             F&& f) {
    const float Rc = R * 1.0001f + 1e-6f * (g.cellf[0] + g.cellf[1] + g.cellf[2]);
    const float R2 = Rc * Rc;
    const float p[3] = {px, py, pz};
    int lo[3], hi[3];
    bool all[3];
    for (int a = 0; a < 3; ++a) {
        lo[a] = (int)floorf((p[a] - Rc) * g.inv_cellf[a]);
        hi[a] = (int)floorf((p[a] + Rc) * g.inv_cellf[a]);
        all[a] = (hi[a] - lo[a] + 1 >= g.nc[a]);
        if (all[a]) {
            lo[a] = 0;
            hi[a] = g.nc[a] - 1;
        } else if (!g.periodic) {
            lo[a] = max(lo[a], 0);
            hi[a] = min(hi[a], g.nc[a] - 1);
        }
    }
    // no rows beside a box without walls
    const int ny = max(hi[1] - lo[1] + 1, 0);
    const int nrows = lo[2] <= hi[2] ? (hi[2] - lo[2] + 1) * ny : 0;
    for (int r = t; r < nrows; r += nt) {
        int z = lo[2] + r / ny, y = lo[1] + r % ny;
        float dz = all[2] ? 0.f : fmaxf(0.f, fmaxf(z * g.cellf[2] - pz, pz - (z + 1) * g.cellf[2]));
        float dy = all[1] ? 0.f : fmaxf(0.f, fmaxf(y * g.cellf[1] - py, py - (y + 1) * g.cellf[1]));
        float rem = R2 - dy * dy - dz * dz;
        if (rem <= 0.f) continue;
        int zz = wrap_cell(z, g.nc[2]), yy = wrap_cell(y, g.nc[1]);
        int64_t base = ((int64_t)zz * g.nc[1] + yy) * g.nc[0];
        int xa, xb;
        if (all[0]) {
            xa = 0;
            xb = g.nc[0] - 1;
        } else {
            float w = sqrtf(rem);
            xa = (int)floorf((px - w) * g.inv_cellf[0]);
            xb = (int)floorf((px + w) * g.inv_cellf[0]);
            if (!g.periodic) {
                xa = max(xa, 0);
                xb = min(xb, g.nc[0] - 1);
            }
        }
        int sl[2], sh[2], ns = 0;
        if (xa < 0) { sl[ns] = xa + g.nc[0]; sh[ns++] = g.nc[0] - 1; sl[ns] = 0; sh[ns++] = xb; }
        else if (xb >= g.nc[0]) { sl[ns] = xa; sh[ns++] = g.nc[0] - 1; sl[ns] = 0; sh[ns++] = xb - g.nc[0]; }
        else { sl[ns] = xa; sh[ns++] = xb; }
        for (int sI = 0; sI < ns; ++sI) {
            int b = g.cell_start[base + sl[sI]];
            int e = g.cell_start[base + sh[sI] + 1];
            for (int j = b; j < e; ++j) f(j);
        }
    }
}

constexpr int kSrcThreads = 128;

// one block per source: Newton on h_s = eta_s omega_s(h_s)^(-1/3) over gas only (no self
// term), omega summed over the rows of all threads in a fixed tree order
__global__ void __launch_bounds__(kSrcThreads) k_src_h(Grid g, const double* __restrict__ xs, int64_t n,
                                                       const double* __restrict__ xsrc, int64_t S, SrcParams sp,
                                                       double* hs_out, double* oms_out, int* flags,
                                                       const int32_t* __restrict__ list_cnt) {
    const int s_id = blockIdx.x;
    const int t = threadIdx.x;
    if (list_cnt[s_id] >= 0) return;     // solved by k_src_lists
    __shared__ double red_w[kSrcThreads], red_dw[kSrcThreads];
    double p[3] = {xsrc[s_id], xsrc[S + s_id], xsrc[2 * S + s_id]};
    const double half[3] = {0.5 * g.box[0], 0.5 * g.box[1], 0.5 * g.box[2]};
    double h = (sp.warm || sp.fixed) ? hs_out[s_id] : sp.h0, lo = 0.0, hi = INFINITY, om = 0.0;
    bool ok = false;
    if (!(h > 0.0) || !(h < sp.h_cap)) {
        if (sp.fixed && t == 0) atomicExch(&flags[F_BADH], 1);
        h = sp.h0;
    }
    __syncthreads();    // every thread has read the first guess before thread 0 overwrites it
    for (int it = 0; it < sp.max_iter; ++it) {
        double H = kKappa * h, iH = 1.0 / H, H2 = H * H;
        double sw = 0.0, sdw = 0.0;
        strided_rows(g, (float)p[0], (float)p[1], (float)p[2], (float)H, t, kSrcThreads, [&](int j) {
            double dx = sep_fast(xs[j], p[0], g.box[0], half[0], g.periodic);
            double dy = sep_fast(xs[n + j], p[1], g.box[1], half[1], g.periodic);
            double dz = sep_fast(xs[2 * n + j], p[2], g.box[2], half[2], g.periodic);
            double r2 = dx * dx + dy * dy + dz * dz;
            if (r2 < H2) {
                double q = sqrt(r2) * iH;
                sw += spline_w(q);
                sdw += q * spline_dw(q);
            }
        });
        red_w[t] = sw;
        red_dw[t] = sdw;
        __syncthreads();
        for (int w = kSrcThreads / 2; w > 0; w >>= 1) {
            if (t < w) {
                red_w[t] += red_w[t + w];
                red_dw[t] += red_dw[t + w];
            }
            __syncthreads();
        }
        sw = red_w[0];
        sdw = red_dw[0];
        __syncthreads();
        om = kSigma * iH * iH * iH * sw;
        if (sp.fixed) {   // given h: omega there, no iteration
            ok = om > 0.0;
            break;
        }
        const int done = src_newton(sp, sw, sdw, h, lo, hi, om);
        if (done) {
            ok = done == 1;
            break;
        }
    }
    if (t == 0) {
        if (!ok) atomicExch(&flags[F_SRC_NOCONV], 1);
        hs_out[s_id] = h;
        oms_out[s_id] = om;
    }
}

// The (z, y) rows of the cell cube [c - k, c + k] around a source, numbered
// z-major; row r's particles are one or two contiguous ranges of the sorted order.
struct CubeRows {
    int lo[3], hi[3];
    int ny, rows;
};

__device__ __forceinline__ CubeRows cube_rows(const Grid& g, const int c0[3], const int k[3]) {
    CubeRows cr;
    for (int a = 0; a < 3; ++a) {
        bool all = (2 * k[a] + 1 >= g.nc[a]);
        cr.lo[a] = all ? 0 : c0[a] - k[a];
        cr.hi[a] = all ? g.nc[a] - 1 : c0[a] + k[a];
        if (!g.periodic && !all) {
            cr.lo[a] = max(cr.lo[a], 0);
            cr.hi[a] = min(cr.hi[a], g.nc[a] - 1);
        }
    }
    cr.ny = cr.hi[1] - cr.lo[1] + 1;
    cr.rows = cr.ny * (cr.hi[2] - cr.lo[2] + 1);
    return cr;
}

// every lane walks row r of the cube, lane l taking every 32nd candidate
template <class F>
__device__ __forceinline__ void warp_row(const Grid& g, const CubeRows& cr, int r, int lane, F&& f) {
    const int zz = wrap_cell(cr.lo[2] + r / cr.ny, g.nc[2]);
    const int yy = wrap_cell(cr.lo[1] + r % cr.ny, g.nc[1]);
    const int64_t base = ((int64_t)zz * g.nc[1] + yy) * g.nc[0];
    const int xa = cr.lo[0], xb = cr.hi[0];
    int sl[2], sh[2], ns = 0;
    if (xa < 0) { sl[ns] = xa + g.nc[0]; sh[ns++] = g.nc[0] - 1; sl[ns] = 0; sh[ns++] = xb; }
    else if (xb >= g.nc[0]) { sl[ns] = xa; sh[ns++] = g.nc[0] - 1; sl[ns] = 0; sh[ns++] = xb - g.nc[0]; }
    else { sl[ns] = xa; sh[ns++] = xb; }
    for (int q = 0; q < ns; ++q) {
        const int b = g.cell_start[base + sl[q]];
        const int e = g.cell_start[base + sh[q] + 1];
        for (int j0 = b; j0 < e; j0 += 32) f(j0 + lane, j0 + lane < e);
    }
}

constexpr int kSrcWarps = 8, kSrcRowsMax = 1024;

// Count (FILL = false) or write (FILL = true) the gas entries of every source, one block of
// kSrcWarps warps per source.  The cube's rows are dealt to the warps (row r to warp
// r mod kSrcWarps); the fill pass first counts every row, scans the counts in row order and
// then writes each row's entries from its offset, so the entries come in the row-major
// candidate order of a single warp's walk.  Cubes of more than kSrcRowsMax rows are walked
// by warp 0 alone.  The fill pass also forms xi, from the octant sums of its own entries or,
// when octw_given is set, from the caller's (a source's owner's, over its whole support).
template <bool FILL>
__global__ void __launch_bounds__(kSrcWarps * 32)
k_src_entries(Grid g, const double* __restrict__ xs, int64_t n, const double* __restrict__ xsrc, int64_t S,
              const double* __restrict__ hs, const double* __restrict__ oms, int32_t* counts,
              const int64_t* __restrict__ off, int32_t* e_gas, double* e_xi, double* octw_out,
              const double* __restrict__ octw_given, const int32_t* __restrict__ list_cnt) {
    __shared__ int row_n[kSrcRowsMax];
    __shared__ double w8s[kSrcWarps][8];
    __shared__ int total;
    const int src = blockIdx.x;
    if (list_cnt[src] >= 0) return;      // k_src_list_entries
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double p[3] = {xsrc[src], xsrc[S + src], xsrc[2 * S + src]};
    int c[3];
    for (int a = 0; a < 3; ++a) c[a] = cell_coord(p[a], g.inv_cell[a], g.nc[a]);
    const double half[3] = {0.5 * g.box[0], 0.5 * g.box[1], 0.5 * g.box[2]};
    const double h = hs[src], H = kKappa * h, iH = 1.0 / H, H2 = H * H;
    const double fac = kSigma * iH * iH * iH / oms[src];
    int k[3];
    for (int a = 0; a < 3; ++a) k[a] = (int)fmin(ceil(H * g.inv_cell[a]), (double)g.nc[a]);
    const CubeRows cr = cube_rows(g, c, k);
    const bool split = cr.rows <= kSrcRowsMax;
    const int nw = split ? kSrcWarps : 1;
    // candidate j of the source's support?  psi and octant when it is
    auto test = [&](int j, bool act, double& ps, int& oct) {
        if (!act) return false;
        const double dx = sep_fast(xs[j], p[0], g.box[0], half[0], g.periodic);
        const double dy = sep_fast(xs[n + j], p[1], g.box[1], half[1], g.periodic);
        const double dz = sep_fast(xs[2 * n + j], p[2], g.box[2], half[2], g.periodic);
        const double r2 = dx * dx + dy * dy + dz * dz;
        if (!(r2 < H2)) return false;
        ps = fac * spline_w(sqrt(r2) * iH);
        oct = (dx < 0 ? 1 : 0) | (dy < 0 ? 2 : 0) | (dz < 0 ? 4 : 0);
        return true;
    };
    // pass 1: entries per row (per warp when the rows are not split)
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    int mine = 0;
    if (wid < nw) {
        for (int r = wid; r < cr.rows; r += nw) {
            int cnt = 0;
            warp_row(g, cr, r, lane, [&](int j, bool act) {
                double ps;
                int oct;
                cnt += __popc(__ballot_sync(0xffffffffu, test(j, act, ps, oct)));
            });
            if (split && lane == 0) row_n[r] = cnt;
            mine += cnt;
        }
        if (lane == 0) atomicAdd(&total, mine);
    }
    __syncthreads();
    if (!FILL) {
        if (threadIdx.x == 0) counts[src] = total;
        return;
    }
    // row offsets in row order (exclusive prefix sums of row_n)
    if (split && threadIdx.x == 0) {
        int acc = 0;
        for (int r = 0; r < cr.rows; ++r) {
            const int v = row_n[r];
            row_n[r] = acc;
            acc += v;
        }
    }
    __syncthreads();
    // pass 2: write the entries (psi for now; mu_a applied below) and the octant sums
    const int64_t base = off[src];
    double w8[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (wid < nw) {
        int run = 0;
        for (int r = wid; r < cr.rows; r += nw) {
            int pos0 = split ? row_n[r] : run;
            warp_row(g, cr, r, lane, [&](int j, bool act) {
                double ps = 0.0;
                int oct = 0;
                const bool in = test(j, act, ps, oct);
                const unsigned bal = __ballot_sync(0xffffffffu, in);
                if (in) {
                    const int pos = pos0 + __popc(bal & ((1u << lane) - 1u));
                    e_gas[base + pos] = j;
                    e_xi[base + pos] = ps;
                    w8[oct] += ps;
                }
                pos0 += __popc(bal);
            });
            run = pos0;
        }
    }
    for (int a = 0; a < 8; ++a) {
        const double v = warp_sum(w8[a]);
        if (lane == 0) w8s[wid][a] = v;
    }
    __syncthreads();
    // octant sums over the warps in warp order; xi = mu_a psi, mu_a = sum_b w_b / (q_nz w_a)
    double ws8[8], wsum = 0.0;
    int qnz = 0;
    for (int a = 0; a < 8; ++a) {
        double v = 0.0;
        for (int w = 0; w < kSrcWarps; ++w) v += w8s[w][a];
        if (octw_given) v = octw_given[8 * src + a];
        ws8[a] = v;
        wsum += v;
        qnz += (v > 0.0);
    }
    if (threadIdx.x == 0)
        for (int a = 0; a < 8; ++a) octw_out[8 * src + a] = ws8[a];
    __syncthreads();   // the entries of pass 2 are visible to every thread
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int j = e_gas[base + e];
        const double dx = sep_fast(xs[j], p[0], g.box[0], half[0], g.periodic);
        const double dy = sep_fast(xs[n + j], p[1], g.box[1], half[1], g.periodic);
        const double dz = sep_fast(xs[2 * n + j], p[2], g.box[2], half[2], g.periodic);
        const int oct = (dx < 0 ? 1 : 0) | (dy < 0 ? 2 : 0) | (dz < 0 ? 4 : 0);
        e_xi[base + e] = wsum / ((double)qnz * ws8[oct]) * e_xi[base + e];
    }
}

// injection entries keyed by (target, source) so that each target sums its sources in
// source order
__global__ void k_inj_keys(const int32_t* __restrict__ e_gas, const int64_t* __restrict__ off, int64_t S,
                           int64_t total, uint64_t* keys, int32_t* vals) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= total) return;
    // source of entry e by binary search in off
    int64_t lo = 0, hi = S;
    while (hi - lo > 1) {
        int64_t mid = (lo + hi) >> 1;
        if (off[mid] <= e) lo = mid; else hi = mid;
    }
    keys[e] = ((uint64_t)(uint32_t)e_gas[e] << 32) | (uint64_t)(uint32_t)lo;
    vals[e] = (int32_t)e;
}

__global__ void k_inj_segments(const uint64_t* __restrict__ keys, const int32_t* __restrict__ vals, int64_t total,
                               const double* __restrict__ e_xi, const double* __restrict__ V,
                               int32_t* head_flag, int32_t* inj_src, double* inj_coef) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= total) return;
    uint32_t g = (uint32_t)(keys[e] >> 32);
    head_flag[e] = (e == 0 || (uint32_t)(keys[e - 1] >> 32) != g) ? 1 : 0;
    inj_src[e] = (int32_t)(uint32_t)(keys[e] & 0xffffffffu);
    inj_coef[e] = e_xi[vals[e]] / V[g];   // xi / V_g: E_g += coef * L dt
}

__global__ void k_inj_targets(const uint64_t* __restrict__ keys, const int32_t* __restrict__ head_flag,
                              const int32_t* __restrict__ head_pos, int64_t total, int32_t* targets,
                              int32_t* inj_off) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= total) return;
    if (head_flag[e]) {
        int t = head_pos[e];
        targets[t] = (int32_t)(keys[e] >> 32);
        inj_off[t] = (int32_t)e;
    }
    if (e == total - 1) inj_off[head_pos[e] + head_flag[e]] = (int32_t)total;
}

static inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// ------------------------------------------------------------------------------------
rt_status build_neighbours(rt_ctx* c, const double* x, const double* m, const double* xsrc, const double* h_in,
                           const double* hs_in, const double* oms_in, const double* octw_in) {
    const int64_t n = c->n, S = c->n_src;
    const rt_config& cfg = c->cfg;
    cudaStream_t st = c->stream;
    const int B = 256;

    // grid: cells of cell_eighths / 8 of the mean-density support radius (default one half)
    double vol = cfg.box[0] * cfg.box[1] * cfg.box[2];
    double h0 = cfg.eta_res * std::cbrt(vol / (double)n);
    double H0 = kKappa * h0;
    const double cell_frac = (c->tune.cell_eighths > 0 ? c->tune.cell_eighths : 4) / 8.0;
    int64_t ncells = 1;
    for (int a = 0; a < 3; ++a) {
        int nca = (int)std::floor(cfg.box[a] / (cell_frac * H0));
        nca = std::max(1, std::min(nca, 1024));
        c->nc[a] = nca;
        c->cell[a] = cfg.box[a] / nca;
        ncells *= nca;
    }
    while (ncells > (int64_t)1 << 27) {   // keep the cell table small
        ncells = 1;
        for (int a = 0; a < 3; ++a) {
            c->nc[a] = std::max(1, c->nc[a] / 2);
            c->cell[a] = cfg.box[a] / c->nc[a];
            ncells *= c->nc[a];
        }
    }
    c->ncells = ncells;
    int bits = 1;
    while (((int64_t)1 << bits) < ncells) ++bits;
    c->key_bits = bits;
    for (int a = 0; a < 3; ++a) c->diag.grid[a] = c->nc[a];

    Grid g;
    for (int a = 0; a < 3; ++a) {
        g.nc[a] = c->nc[a];
        g.cell[a] = c->cell[a];
        g.inv_cell[a] = 1.0 / c->cell[a];
        g.cellf[a] = (float)c->cell[a];
        g.inv_cellf[a] = (float)(1.0 / c->cell[a]);
        g.box[a] = cfg.box[a];
    }
    g.periodic = cfg.periodic;

    // buffers
    RT_TRY(ensure(c, c->keys_in, n * 4, "keys"));
    RT_TRY(ensure(c, c->keys_out, n * 4, "keys"));
    RT_TRY(ensure(c, c->idx_in, n * 4, "idx"));
    RT_TRY(ensure(c, c->perm, n * 4, "perm"));
    RT_TRY(ensure(c, c->inv_perm, n * 4, "inv_perm"));
    RT_TRY(ensure(c, c->cell_start, (ncells + 1) * 4, "cells"));
    RT_TRY(ensure(c, c->xs_d, 3 * n * 8, "positions"));
    RT_TRY(ensure(c, c->xq, 16 * n, "positions"));
    RT_TRY(ensure(c, c->m_s, n * 8, "masses"));
    RT_TRY(ensure(c, c->h_d, n * 8, "h"));
    RT_TRY(ensure(c, c->H2f, n * 4, "h"));
    RT_TRY(ensure(c, c->omega_d, n * 8, "omega"));
    RT_TRY(ensure(c, c->V_d, n * 8, "V"));
    RT_TRY(ensure(c, c->B_d, 6 * n * 8, "B"));
    RT_TRY(ensure(c, c->cond_f, n * 4, "cond"));
    RT_TRY(ensure(c, c->h_sum, 3 * n * 4, "h"));
    size_t ts = c->fp64 ? 8 : 4;
    RT_TRY(ensure(c, c->pos_t, n * 32, "geom"));
    RT_TRY(ensure(c, c->geo_t, 8 * n * ts, "geom"));
    RT_TRY(ensure(c, c->omega_t, n * ts, "geom"));
    RT_TRY(ensure(c, c->counts, (n + 1) * 4, "counts"));
    RT_TRY(ensure(c, c->row_off, (n + 1) * 8, "row_off"));
    const int cap = list_capacity(cfg.eta_res);
    RT_TRY(ensure(c, c->lists, (size_t)n * cap * 4, "candidate lists"));
    RT_TRY(ensure(c, c->list_cnt, (size_t)n * 4, "candidate lists"));
    RT_TRY(ensure(c, c->flags, 64, "flags"));
    RT_TRY(ensure(c, c->red_tmp, 64, "reduction"));

    int* flags = c->flags.as<int>();
    RT_CUDA(c, cudaMemsetAsync(flags, 0, 64, st));
    const bool warm = c->has_h_prev;
    c->has_h_prev = false;       // set again only when this call succeeds
    // reductions: [0] min h, [1] max h, [2] max cond, [3] min V (bit patterns of positive doubles),
    // [4] sum of H^3, [5] spill length, [6] extras of long rows, [7] max float cond
    unsigned long long* red = reinterpret_cast<unsigned long long*>(c->red_tmp.p);
    RT_CUDA(c, cudaMemsetAsync(red, 0, 64, st));
    RT_CUDA(c, cudaMemsetAsync(red, 0xff, 8, st));
    RT_CUDA(c, cudaMemsetAsync(red + 3, 0xff, 8, st));

    // cub scratch: radix sort of N, scans of N+1 and S+1, radix sort of the injection entries
    size_t t1 = 0, t2 = 0, t3 = 0;
    cub::DeviceRadixSort::SortPairs(nullptr, t1, (const uint32_t*)nullptr, (uint32_t*)nullptr,
                                    (const int32_t*)nullptr, (int32_t*)nullptr, (int)n, 0, bits, st);
    cub::DeviceScan::ExclusiveSum(nullptr, t2, (const int32_t*)nullptr, (int64_t*)nullptr,
                                  (int)(std::max<int64_t>(n, S) + 1), st);
    int64_t Smax = std::max<int64_t>(S, 1) * 4096;
    cub::DeviceRadixSort::SortPairs(nullptr, t3, (const uint64_t*)nullptr, (uint64_t*)nullptr,
                                    (const int32_t*)nullptr, (int32_t*)nullptr, (int)Smax, 0, 64, st);
    RT_TRY(ensure(c, c->cub_tmp, std::max(t1, std::max(t2, t3)) + 256, "cub scratch"));

    // a1: keys, sort, cell table, sorted copies
    k_keys<<<nblk(n, B), B, 0, st>>>(x, n, g, c->keys_in.as<uint32_t>(), c->idx_in.as<int32_t>(), flags);
    size_t tb = c->cub_tmp.bytes;
    RT_CUDA(c, cub::DeviceRadixSort::SortPairs(c->cub_tmp.p, tb, c->keys_in.as<uint32_t>(), c->keys_out.as<uint32_t>(),
                                               c->idx_in.as<int32_t>(), c->perm.as<int32_t>(), (int)n, 0, bits, st));
    k_cell_start<<<nblk(ncells + 1, B), B, 0, st>>>(c->keys_out.as<uint32_t>(), n, ncells, c->cell_start.as<int32_t>());
    g.cell_start = c->cell_start.as<int32_t>();
    double qmul[3];
    float qscale[3];
    for (int a = 0; a < 3; ++a) {
        double units = cfg.periodic ? 4294967296.0 : 2147483648.0;
        qmul[a] = units / cfg.box[a];
        qscale[a] = (float)(cfg.box[a] / units);
    }
    const Box box = {{cfg.box[0], cfg.box[1], cfg.box[2]}, cfg.periodic};
    k_gather_positions<<<nblk(n, B), B, 0, st>>>(x, m, c->perm.as<int32_t>(), n, box, qmul[0], qmul[1], qmul[2],
                                                  c->xs_d.as<double>(), c->xq.as<uint4>(), c->m_s.as<double>(),
                                                  c->inv_perm.as<int32_t>());
    RT_CUDA(c, cudaGetLastError());
    c->launches += 3;   // keys, cell table, gather

    // a2: smoothing lengths
    HParams hp;
    hp.eta = cfg.eta_res;
    hp.eta3 = cfg.eta_res * cfg.eta_res * cfg.eta_res;
    hp.s_star = kKappa * kKappa * kKappa / kSigma * hp.eta3;
    hp.h0 = h0;
    double minbox = std::min(cfg.box[0], std::min(cfg.box[1], cfg.box[2]));
    hp.h_cap = cfg.periodic ? 0.5 * minbox / kKappa : 1e30;
    for (int a = 0; a < 3; ++a) hp.scale[a] = qscale[a];
    hp.max_iter = cfg.h_max_iter > 0 ? cfg.h_max_iter : 100;
    hp.tol32 = (float)std::max(cfg.h_tol, 2e-6);
    // the FP64 path refines every h in double; the float path only those of particles with a
    // candidate near their support radius, which is enough for the exact roots' pair lists
    hp.refine64 = c->fp64 ? 1 : 0;
    int* refine_count = flags + F_REFINE;
    const size_t st_bytes = (size_t)kListParticles * cap * sizeof(float);
    if (h_in) {
        hp.refine64 = c->fp64 ? 1 : 0;   // omega in the working path's arithmetic
        k_h_given<<<nblk(n, 128), 128, 0, st>>>(g, c->xs_d.as<double>(), c->xq.as<uint4>(), n, hp, h_in,
                                                 c->perm.as<int32_t>(), c->h_d.as<double>(), c->omega_d.as<double>(),
                                                 c->H2f.as<float>(), red, flags);
    } else {
        k_h_lists<true><<<nblk(n, kListParticles), kListWarps * 32, st_bytes, st>>>(
            g, c->xs_d.as<double>(), c->xq.as<uint4>(), n, hp, warm ? c->h_prev.as<double>() : nullptr,
            c->perm.as<int32_t>(), nullptr, c->h_sum.as<float>(), flags, c->idx_in.as<int32_t>(), refine_count,
            c->lists.as<int32_t>(), c->list_cnt.as<int32_t>(), cap);
    }
    RT_CUDA(c, cudaGetLastError());
    if (h_in)
        k_h_lists<false><<<nblk(n, kListParticles), kListWarps * 32, st_bytes, st>>>(
            g, c->xs_d.as<double>(), c->xq.as<uint4>(), n, hp, nullptr, nullptr, c->h_d.as<double>(), nullptr, flags,
            nullptr, nullptr, c->lists.as<int32_t>(), c->list_cnt.as<int32_t>(), cap);
    k_h_finish<<<nblk(n, 256), 256, 0, st>>>(h_in ? nullptr : c->h_sum.as<float>(), n, hp.refine64 ? 0 : 1,
                                             c->h_d.as<double>(), c->omega_d.as<double>(), c->H2f.as<float>(),
                                             c->xq.as<uint4>(), red);
    if (!h_in) {
        // the number of flagged particles is on the device: grids of resident blocks (FP64: all)
        int32_t* rest = c->keys_in.as<int32_t>();     // the keys are done with
        int* rest_n = flags + F_SCRATCH;
        RT_CUDA(c, cudaMemsetAsync(rest_n, 0, 4, st));
        const bool few = !c->fp64 && n < (int64_t)c->sm_count * 256;
        const int64_t nbr = std::min<int64_t>(nblk(n * (few ? 32 : 8), 128), c->sm_count * (c->fp64 ? 64 : 8));
        (few ? k_h_refine<32, 4> : k_h_refine<8, 12>)<<<(unsigned)nbr, 128, 0, st>>>(
            g, c->xs_d.as<double>(), c->xq.as<uint4>(), n, hp, c->fp64 ? nullptr : c->idx_in.as<int32_t>(),
            refine_count, c->lists.as<int32_t>(), c->list_cnt.as<int32_t>(), cap, c->h_d.as<double>(),
            c->omega_d.as<double>(), c->H2f.as<float>(), c->xq.as<uint4>(), red, flags, rest, rest_n);
        k_h_refine_walk<<<(unsigned)std::min<int64_t>(nblk(n, kRestWarps), c->sm_count * 6), kRestWarps * 32, 0, st>>>(
            g, c->xs_d.as<double>(), c->xq.as<uint4>(), n, hp, rest, rest_n, c->list_cnt.as<int32_t>(),
            c->h_d.as<double>(), c->omega_d.as<double>(), c->H2f.as<float>(), c->xq.as<uint4>(), red,
            c->fp64 ? 1 : 0, flags);
        c->launches += 1;
    }
    RT_CUDA(c, cudaGetLastError());
    c->launches += 3;

    // a3: symmetric pair lists; every particle finds the entries of its own support, and the
    // sizes of the rows come back with the flags of everything before (one synchronisation)
    PairParams pp;
    for (int a = 0; a < 3; ++a) pp.scale[a] = qscale[a];
    RT_TRY(ensure(c, c->own_cnt, (size_t)n * 4, "pair rows"));
    RT_TRY(ensure(c, c->extra_cnt, (size_t)n * 4, "pair rows"));
    RT_TRY(ensure(c, c->extras, (size_t)n * kExtras * 4, "pair rows"));
    unsigned long long *spill_n = red + 5, *more_n = red + 6;
    int* over_n = flags + F_OVER;
    int32_t* over = c->idx_in.as<int32_t>();      // the flagged particles' list is done with
    RT_CUDA(c, cudaMemsetAsync(c->extra_cnt.p, 0, (size_t)n * 4, st));
    k_own_rows<<<nblk(n * 32, 256), 256, 0, st>>>(g, c->xs_d.as<double>(), c->xq.as<uint4>(), c->h_d.as<double>(), n,
                                                   pp, c->lists.as<int32_t>(), cap, c->list_cnt.as<int32_t>(),
                                                   c->own_cnt.as<int32_t>(), c->extra_cnt.as<int32_t>(),
                                                   c->extras.as<int32_t>(), over, over_n);
    k_own_walk<false><<<(unsigned)c->sm_count * 4, 128, 0, st>>>(
        g, c->xs_d.as<double>(), c->xq.as<uint4>(), c->h_d.as<double>(), n, pp, c->lists.as<int32_t>(), cap,
        c->own_cnt.as<int32_t>(), c->extra_cnt.as<int32_t>(), c->extras.as<int32_t>(), over, over_n, spill_n, nullptr);
    k_row_lengths<<<nblk(n + 1, 256), 256, 0, st>>>(c->own_cnt.as<int32_t>(), c->extra_cnt.as<int32_t>(), n,
                                                     c->counts.as<int32_t>(), more_n);
    RT_CUDA(c, cudaGetLastError());
    tb = c->cub_tmp.bytes;
    RT_CUDA(c, cub::DeviceScan::ExclusiveSum(c->cub_tmp.p, tb, c->counts.as<int32_t>(), c->row_off.as<int64_t>(),
                                             (int)(n + 1), st));
    c->launches += 3;
    int hflags[8];
    struct {
        double hmin, hmax, cond, vmin, h3;
        unsigned long long spill, more;
    } hred;
    static_assert(sizeof(hred) == 56, "layout of the reduction buffer");
    int64_t P2 = 0;
    RT_CUDA(c, cudaMemcpyAsync(hflags, flags, sizeof(hflags), cudaMemcpyDeviceToHost, st));
    RT_CUDA(c, cudaMemcpyAsync(&hred, red, sizeof(hred), cudaMemcpyDeviceToHost, st));
    RT_CUDA(c, cudaMemcpyAsync(&P2, c->row_off.as<int64_t>() + n, 8, cudaMemcpyDeviceToHost, st));
    RT_CUDA(c, cudaStreamSynchronize(st));
    if (hflags[F_BADPOS]) return fail(c, RT_ERR_INVALID, "positions must be finite and inside [0, box)");
    if (hflags[F_NOCONV]) return fail(c, RT_ERR_NOCONV, "smoothing-length iteration did not converge");
    if (hflags[F_BADH]) return fail(c, RT_ERR_INVALID, "given smoothing lengths must be finite, > 0 and below the "
                                                       "quarter of the periodic box over the support ratio");
    c->diag.h_refined = h_in ? 0 : (c->fp64 ? n : (int64_t)hflags[F_REFINE]);
    c->diag.h_min = hred.hmin;
    c->diag.h_max = hred.hmax;
    const double Hmax = kKappa * hred.hmax;
    if (cfg.periodic && Hmax >= 0.5 * minbox)
        return fail(c, RT_ERR_GEOMETRY, "support radius reaches half the periodic box");
    if (P2 >= ((int64_t)1 << 31)) return fail(c, RT_ERR_INVALID, "more than 2^31 neighbour entries");
    // the spread of the supports, H_max^3 over the mean H^3
    c->diag.pair_build = Hmax * Hmax * Hmax / std::max(hred.h3 / (double)n, 1e-300) > 12.0 ? 1 : 0;
    RT_TRY(ensure(c, c->cols, std::max<int64_t>(P2, 1) * 4, "pair lists", true));
    RT_TRY(ensure(c, c->n_low, (n + 1) * 4, "pair split"));
    RT_TRY(ensure(c, c->n_up, (n + 1) * 4, "pair split"));
    if (hred.spill > 0) {     // own entries of the particles without a list
        RT_TRY(ensure(c, c->spill, (size_t)hred.spill * 4, "pair rows", true));
        k_own_walk<true><<<(unsigned)c->sm_count * 4, 128, 0, st>>>(
            g, c->xs_d.as<double>(), c->xq.as<uint4>(), c->h_d.as<double>(), n, pp, c->lists.as<int32_t>(), cap,
            c->own_cnt.as<int32_t>(), nullptr, nullptr, over, over_n, nullptr, c->spill.as<int32_t>());
        c->launches += 1;
    }
    if (hred.more > 0) {      // rows with more extras than they hold in place
        RT_TRY(ensure(c, c->more, (size_t)hred.more * 4, "pair rows", true));
        RT_TRY(ensure(c, c->more_off, (size_t)(n + 1) * 8, "pair rows"));
        int32_t* cnt = c->counts.as<int32_t>();
        k_more_extras<<<nblk(n + 1, 256), 256, 0, st>>>(c->extra_cnt.as<int32_t>(), n, cnt);
        tb = c->cub_tmp.bytes;
        RT_CUDA(c, cub::DeviceScan::ExclusiveSum(c->cub_tmp.p, tb, cnt, c->more_off.as<int64_t>(), (int)(n + 1), st));
        RT_CUDA(c, cudaMemsetAsync(cnt, 0, (size_t)n * 4, st));
        k_extras_fill<<<nblk(n * 32, 256), 256, 0, st>>>(
            n, c->lists.as<int32_t>(), cap, c->list_cnt.as<int32_t>(), c->own_cnt.as<int32_t>(),
            c->extra_cnt.as<int32_t>(), c->more_off.as<int64_t>(), cnt, c->spill.as<int32_t>(), c->more.as<int32_t>());
        c->launches += 2;
    }
    k_rows_merge<<<nblk(n * 32, 256), 256, 0, st>>>(
        n, c->lists.as<int32_t>(), cap, c->list_cnt.as<int32_t>(), c->own_cnt.as<int32_t>(),
        c->extra_cnt.as<int32_t>(), c->extras.as<int32_t>(), c->more_off.as<int64_t>(), c->more.as<int32_t>(),
        c->spill.as<int32_t>(), c->row_off.as<int64_t>(), c->cols.as<int32_t>(), c->n_low.as<int32_t>(),
        c->n_up.as<int32_t>());
    c->launches += 1;
    RT_CUDA(c, cudaGetLastError());
    c->n_directed = P2;
    c->launches += 1;   // geometry below

    // the slots of the pairs
    RT_TRY(ensure(c, c->up_off, (n + 1) * 8, "pair split"));
    RT_TRY(ensure(c, c->low_slot, std::max<int64_t>(P2 / 2, 1) * 4, "pair split", true));
    RT_CUDA(c, cudaMemsetAsync(c->n_up.as<int32_t>() + n, 0, 4, st));
    tb = c->cub_tmp.bytes;
    RT_CUDA(c, cub::DeviceScan::ExclusiveSum(c->cub_tmp.p, tb, c->n_up.as<int32_t>(), c->up_off.as<int64_t>(),
                                             (int)(n + 1), st));
    RT_TRY(ensure(c, c->pair_ends, std::max<int64_t>(P2 / 2, 1) * 8, "pair split", true));
    k_pair_slots<<<nblk(n * 32, 256), 256, 0, st>>>(c->row_off.as<int64_t>(), c->cols.as<int32_t>(),
                                                     c->n_low.as<int32_t>(), c->up_off.as<int64_t>(), n,
                                                     c->pair_ends.as<int2>(), c->low_slot.as<int32_t>());
    c->launches += 1;
    RT_CUDA(c, cudaGetLastError());

    // a4: geometry
    unsigned* cond_max = reinterpret_cast<unsigned*>(red + 7);
    double* Bd = c->B_d.as<double>();
    if (c->fp64) {
        const bool few = n < (int64_t)c->sm_count * 1024;
        (few ? k_E<double, 8> : k_E<double, 1>)<<<nblk(few ? n * 8 : n, 256), 256, 0, st>>>(
            c->xs_d.as<double>(), c->xq.as<uint4>(), c->h_d.as<double>(), c->row_off.as<int64_t>(),
            c->cols.as<int32_t>(), n, cfg.box[0], cfg.box[1], cfg.box[2], cfg.periodic, qscale[0], qscale[1],
            qscale[2], Bd);
        k_geometry<double><<<nblk(n, 128), 128, 0, st>>>(
            c->xs_d.as<double>(), c->xq.as<uint4>(), c->h_d.as<double>(), c->omega_d.as<double>(), n,
            c->V_d.as<double>(), Bd, c->cond_f.as<float>(), c->pos_t.p, c->geo_t.as<double>(), c->omega_t.as<double>(),
            red, cond_max, flags);
    } else {
        k_E<float, 1><<<nblk(n, 256), 256, 0, st>>>(
            c->xs_d.as<double>(), c->xq.as<uint4>(), c->h_d.as<double>(), c->row_off.as<int64_t>(),
            c->cols.as<int32_t>(), n, cfg.box[0], cfg.box[1], cfg.box[2], cfg.periodic, qscale[0], qscale[1],
            qscale[2], Bd);
        k_geometry<float><<<nblk(n, 128), 128, 0, st>>>(
            c->xs_d.as<double>(), c->xq.as<uint4>(), c->h_d.as<double>(), c->omega_d.as<double>(), n,
            c->V_d.as<double>(), Bd, c->cond_f.as<float>(), c->pos_t.p, c->geo_t.as<float>(), c->omega_t.as<float>(),
            red, cond_max, flags);
    }
    c->launches += 1;
    k_cond<<<nblk(n, 256), 256, 0, st>>>(c->cond_f.as<float>(), c->B_d.as<double>(), n, cond_max, red, flags);
    c->launches += 1;
    RT_CUDA(c, cudaGetLastError());

    // a5 preparation: sources
    c->n_inj_entries = 0;
    c->n_inj_targets = 0;
    if (S > 0) {
        RT_TRY(ensure(c, c->xsrc_d, 3 * S * 8, "sources"));
        RT_TRY(ensure(c, c->hs_d, S * 8, "sources"));
        RT_TRY(ensure(c, c->omegas_d, S * 8 + 64 * S, "sources"));
        RT_TRY(ensure(c, c->src_counts, (S + 1) * 4, "sources"));
        RT_TRY(ensure(c, c->src_off, (S + 1) * 8, "sources"));
        k_src_positions<<<nblk(3 * S, 128), 128, 0, st>>>(xsrc, S, box, c->xsrc_d.as<double>(), flags);
        SrcParams sp;
        sp.eta3 = cfg.eta_res_star * cfg.eta_res_star * cfg.eta_res_star;
        sp.s_star = kKappa * kKappa * kKappa / kSigma * sp.eta3;
        sp.h0 = cfg.eta_res_star * std::cbrt(vol / (double)n);
        sp.h_cap = hp.h_cap;
        sp.max_iter = std::max(hp.max_iter, 200);
        sp.warm = c->has_hs_prev ? 1 : 0;
        sp.fixed = hs_in ? 1 : 0;
        c->has_hs_prev = false;     // set again only when this call succeeds
        if (hs_in) RT_CUDA(c, cudaMemcpyAsync(c->hs_d.p, hs_in, S * 8, cudaMemcpyDeviceToDevice, st));
        const unsigned sb = (unsigned)S;   // one block of kSrcWarps warps per source
        RT_TRY(ensure(c, c->src_list, (size_t)S * kSrcList * 4, "sources"));
        RT_TRY(ensure(c, c->src_list_cnt, (size_t)S * 4, "sources"));
        int32_t* slist = c->src_list.as<int32_t>();
        int32_t* scnt = c->src_list_cnt.as<int32_t>();
        QuantParams qp;
        for (int a = 0; a < 3; ++a) {
            qp.mul[a] = qmul[a];
            qp.scale[a] = qscale[a];
        }
        const unsigned sw = nblk(S, kSrcListWarps);
        k_src_lists<<<sw, kSrcListWarps * 32, 0, st>>>(g, c->xs_d.as<double>(), c->xq.as<uint4>(), n, qp,
                                                       c->xsrc_d.as<double>(), S, sp, c->hs_d.as<double>(),
                                                       c->omegas_d.as<double>(), flags, slist, scnt);
        k_src_h<<<(unsigned)S, kSrcThreads, 0, st>>>(g, c->xs_d.as<double>(), n, c->xsrc_d.as<double>(), S, sp,
                                                     c->hs_d.as<double>(), c->omegas_d.as<double>(), flags, scnt);
        if (hs_in && oms_in)   // the sources' own omega_s, from their owners
            RT_CUDA(c, cudaMemcpyAsync(c->omegas_d.p, oms_in, S * 8, cudaMemcpyDeviceToDevice, st));
        k_src_list_entries<false><<<sw, kSrcListWarps * 32, 0, st>>>(
            g, c->xs_d.as<double>(), n, c->xsrc_d.as<double>(), S, c->hs_d.as<double>(), c->omegas_d.as<double>(),
            slist, scnt, c->src_counts.as<int32_t>(), nullptr, nullptr, nullptr, nullptr, nullptr);
        k_src_entries<false><<<sb, kSrcWarps * 32, 0, st>>>(g, c->xs_d.as<double>(), n, c->xsrc_d.as<double>(), S,
                                                 c->hs_d.as<double>(), c->omegas_d.as<double>(),
                                                 c->src_counts.as<int32_t>(), nullptr, nullptr, nullptr, nullptr,
                                                 nullptr, scnt);
        RT_CUDA(c, cudaMemsetAsync(c->src_counts.as<int32_t>() + S, 0, 4, st));
        tb = c->cub_tmp.bytes;
        RT_CUDA(c, cub::DeviceScan::ExclusiveSum(c->cub_tmp.p, tb, c->src_counts.as<int32_t>(),
                                                 c->src_off.as<int64_t>(), (int)(S + 1), st));
        c->launches += 5;
        int64_t NE = 0;
        RT_CUDA(c, cudaMemcpyAsync(&NE, c->src_off.as<int64_t>() + S, 8, cudaMemcpyDeviceToHost, st));
        RT_CUDA(c, cudaMemcpyAsync(hflags, flags, sizeof(hflags), cudaMemcpyDeviceToHost, st));
        RT_CUDA(c, cudaStreamSynchronize(st));
        if (hflags[F_BADPOS]) return fail(c, RT_ERR_INVALID, "source positions must be finite");
        if (hflags[F_BADH]) return fail(c, RT_ERR_INVALID, "given source smoothing lengths must be finite and > 0");
        if (hflags[F_SRC_NOCONV]) return fail(c, RT_ERR_NOCONV, "source smoothing-length iteration did not converge");
        if (NE > Smax) return fail(c, RT_ERR_INVALID, "too many injection entries");
        c->n_inj_entries = NE;
        const int64_t NEa = std::max<int64_t>(NE, 1);
        RT_TRY(ensure(c, c->src_entry_gas, NEa * 4, "injection", true));
        RT_TRY(ensure(c, c->src_entry_xi, NEa * 8, "injection", true));
        RT_TRY(ensure(c, c->inj_key, NEa * 8, "injection", true));
        RT_TRY(ensure(c, c->inj_key_out, NEa * 8, "injection", true));
        RT_TRY(ensure(c, c->inj_val, NEa * 4, "injection", true));
        RT_TRY(ensure(c, c->inj_val_out, NEa * 4, "injection", true));
        RT_TRY(ensure(c, c->inj_src, NEa * 4, "injection", true));
        RT_TRY(ensure(c, c->inj_coef, NEa * 8, "injection", true));
        RT_TRY(ensure(c, c->inj_targets, NEa * 4, "injection", true));
        RT_TRY(ensure(c, c->inj_off, (NEa + 1) * 4, "injection", true));
        double* octw = c->omegas_d.as<double>() + S;   // 8 per source after omega_s
        k_src_list_entries<true><<<sw, kSrcListWarps * 32, 0, st>>>(
            g, c->xs_d.as<double>(), n, c->xsrc_d.as<double>(), S, c->hs_d.as<double>(), c->omegas_d.as<double>(),
            slist, scnt, nullptr, c->src_off.as<int64_t>(), c->src_entry_gas.as<int32_t>(),
            c->src_entry_xi.as<double>(), octw, hs_in ? octw_in : nullptr);
        k_src_entries<true><<<sb, kSrcWarps * 32, 0, st>>>(g, c->xs_d.as<double>(), n, c->xsrc_d.as<double>(), S,
                                                c->hs_d.as<double>(), c->omegas_d.as<double>(), nullptr,
                                                c->src_off.as<int64_t>(), c->src_entry_gas.as<int32_t>(),
                                                c->src_entry_xi.as<double>(), octw, hs_in ? octw_in : nullptr, scnt);
        c->launches += 2;
        if (NE > 0) {
            c->launches += 3;
            k_inj_keys<<<nblk(NE, B), B, 0, st>>>(c->src_entry_gas.as<int32_t>(), c->src_off.as<int64_t>(), S, NE,
                                                   c->inj_key.as<uint64_t>(), c->inj_val.as<int32_t>());
            tb = c->cub_tmp.bytes;
            RT_CUDA(c, cub::DeviceRadixSort::SortPairs(c->cub_tmp.p, tb, c->inj_key.as<uint64_t>(),
                                                       c->inj_key_out.as<uint64_t>(), c->inj_val.as<int32_t>(),
                                                       c->inj_val_out.as<int32_t>(), (int)NE, 0, 64, st));
            // head flags into idx_in (free now), positions via scan into counts-sized scratch
            int32_t* head = c->inj_val.as<int32_t>();       // reuse: NE int32
            k_inj_segments<<<nblk(NE, B), B, 0, st>>>(c->inj_key_out.as<uint64_t>(), c->inj_val_out.as<int32_t>(), NE,
                                                       c->src_entry_xi.as<double>(), c->V_d.as<double>(), head,
                                                       c->inj_src.as<int32_t>(), c->inj_coef.as<double>());
            int32_t* hpos = reinterpret_cast<int32_t*>(c->inj_key.as<uint64_t>());   // reuse: NE int32
            tb = c->cub_tmp.bytes;
            RT_CUDA(c, cub::DeviceScan::ExclusiveSum(c->cub_tmp.p, tb, head, hpos, (int)NE, st));
            k_inj_targets<<<nblk(NE, B), B, 0, st>>>(c->inj_key_out.as<uint64_t>(), head, hpos, NE,
                                                      c->inj_targets.as<int32_t>(), c->inj_off.as<int32_t>());
            int32_t lastpos = 0, lasthead = 0;
            RT_CUDA(c, cudaMemcpyAsync(&lastpos, hpos + NE - 1, 4, cudaMemcpyDeviceToHost, st));
            RT_CUDA(c, cudaMemcpyAsync(&lasthead, head + NE - 1, 4, cudaMemcpyDeviceToHost, st));
            RT_CUDA(c, cudaStreamSynchronize(st));
            c->n_inj_targets = lastpos + lasthead;
        }
    }

    // finish: flags, counters (one synchronisation)
    double cv[2];
    RT_CUDA(c, cudaMemcpyAsync(hflags, flags, sizeof(hflags), cudaMemcpyDeviceToHost, st));
    RT_CUDA(c, cudaMemcpyAsync(cv, red + 2, sizeof(cv), cudaMemcpyDeviceToHost, st));
    RT_CUDA(c, cudaStreamSynchronize(st));
    if (hflags[F_GEOM]) return fail(c, RT_ERR_GEOMETRY, "singular E_i: a particle has fewer than 3 non-coplanar neighbours");
    c->diag.n_ill_conditioned = hflags[F_ILL];
    c->diag.n_directed = P2;
    c->diag.n_pairs = P2 / 2;
    c->diag.n_injection = c->n_inj_entries;
    c->diag.cond_max = cv[0];
    c->diag.dx_min = std::cbrt(cv[1] / (4.0 * M_PI / 3.0));
    // keep h in caller order as the first guess of the next call
    RT_TRY(ensure(c, c->h_prev, n * 8, "h"));
    RT_TRY(field_out(c, c->h_d.as<double>(), c->h_prev.as<double>(), 1));
    c->has_h_prev = true;
    c->has_hs_prev = S > 0;
    return RT_OK;
}

}  // namespace rt
