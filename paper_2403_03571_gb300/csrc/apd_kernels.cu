// Seed preparation, the dual value/gradient of eqs. (2.7)-(2.8) from integer
// moments, the discrete centroids of Algorithm 3, and the vector kernels of
// the L-BFGS weight solve (Algorithm 2).
#include <float.h>
#include <math.h>
#include <stddef.h>
#include <string.h>

#include <algorithm>

#include "apd_common.cuh"

namespace apd {

namespace {

// Counts a block in: the caller's earlier writes (and those a barrier made visible to it)
// are visible to whoever counts in later.
__device__ __forceinline__ unsigned count_in(unsigned *counter) {
    unsigned old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(counter) : "memory");
    return old;
}

__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }


// Start of an evaluation whose records' positions and matrices are unchanged
// (same x, A, n as the last seed preparation): zeroed moments and queue count,
// the trial weights (w = W0 + t p into Wt when p is given, else w = W0), their
// copies in the scored records (scan order) and both rescoring record arrays,
// the reference weight wref = max w (per-block maxima reduced by the last block
// to finish), and each 32-seed group's largest weight and gap wref - wmax.  One
// thread per scan position; a warp covers one group.
// With coef (the first trial of a new L-BFGS direction), the direction itself
// is formed first, p = -gamma gf + sum_k (cy_k y_k + cs_k s_k) from the
// coefficients the direction kernels left (written to pdir), with <gf, p>
// reduced by the last block into sc->gp0: one launch instead of two.
//
// Bound: latency (memory round trips, the FP64 chain of p's terms); each warp is a block of
// its own, so that no two share an SM's FP64 unit while there are SMs, maxima go through
// ordered integer keys (an FP64 maximum and shuffle step take 127 clocks), twelve pairs'
// loads are in flight at a time, the stores follow the count of the blocks.  n = 1000, ten
// pairs: 11.5 us -> 7.9 us.  <gf, p> is summed as blocks of `vw` warps, then over the blocks.
__global__ void __launch_bounds__(32)
    eval_begin_kernel(const int n, const int n_pad, const int vw, const long long n_mom, const double *__restrict__ W0,
                      const double t, double *__restrict__ pdir, double *__restrict__ Wt,
                      const int32_t *__restrict__ perm, SeedRec *__restrict__ recs,
                      SeedRec32 *__restrict__ recs32, SeedRec32 *__restrict__ recs32s,
                      GroupBound *__restrict__ groups, unsigned long long *__restrict__ mom,
                      double *__restrict__ part, DevScalars *__restrict__ sc, const LbfgsCoef *__restrict__ coef,
                      const double *__restrict__ S, const double *__restrict__ Y, const double *__restrict__ gfv,
                      const double *__restrict__ w0, const unsigned long long *__restrict__ wref0,
                      const unsigned *__restrict__ g3_hist, const unsigned full_max,
                      float2 *__restrict__ drift, const PushState push, PushState *__restrict__ push_to) {
    __shared__ double ccy[32], ccs[32];
    __shared__ int cslot[32];
    const int lane = threadIdx.x;
    const int i = blockIdx.x * 32 + lane;
    const int src = i < n_pad ? (perm ? perm[i] : i) : n;
    const bool real = src < n;
    double wi = real ? W0[src] : 0.0;
    int hist = 0;
    double gam = 0.0;
    if (coef) {
        hist = min(coef->hist, 31);
        gam = coef->gamma;
        ccy[lane] = coef->cy[lane];
        ccs[lane] = coef->cs[lane];
        cslot[lane] = coef->slot[lane];
        __syncwarp();
    }
    double gp = 0.0;
    double dhi = -DBL_MAX, dlo = DBL_MAX;  // range of w - w0 (with w0)
    unsigned long long wkey = dkey(-DBL_MAX);
    double pv = 0.0;
    if (real) {
        if (pdir) {
            if (coef) {
                const double g = gfv[src];
                pv = -gam * g;
                constexpr int kAhead = 12;
                for (int k0 = 0; k0 < hist; k0 += kAhead) {
                    double yk[kAhead], sk[kAhead];
#pragma unroll
                    for (int e = 0; e < kAhead; ++e) {
                        const size_t o = (size_t)cslot[min(k0 + e, hist - 1)] * n + src;
                        yk[e] = Y[o];
                        sk[e] = S[o];
                    }
#pragma unroll
                    for (int e = 0; e < kAhead; ++e)
                        if (k0 + e < hist) pv += ccy[k0 + e] * yk[e] + ccs[k0 + e] * sk[e];
                }
                gp = g * pv;
            } else {
                pv = pdir[src];
            }
            wi = fma(t, pv, wi);
        }
        if (finite_bits(wi)) wkey = dkey(wi);
        if (w0) {  // rounded outwards, so that the range covers the exact drift
            dhi = __dsub_ru(wi, w0[src]);
            dlo = __dsub_rd(wi, w0[src]);
        }
    }
    const unsigned long long wmax = warp_max_key(wkey);
    if (coef) gp = warp_sum(gp);
    double hi = dhi, lo = dlo;
    if (w0) {
        hi = warp_max(dhi);
        lo = warp_min(dlo);
    }
    unsigned last = 0;
    if (lane == 0) {
        double *row = part + (size_t)blockIdx.x * kPartStride;
        row[0] = __longlong_as_double((long long)wmax);
        if (coef) row[1] = gp;
        if (w0) {
            row[2] = hi;
            row[3] = lo;
        }
        last = count_in(&sc->dual_done) == gridDim.x - 1;
    }
    // the seeds' and the pass's stores after the count: the fence before it would wait for them
    if (real) {
        if (pdir) {
            if (coef) pdir[src] = pv;
            Wt[src] = wi;
        }
        if (!finite_bits(wi)) atomicOr(&sc->status, ST_NONFINITE);
        recs[i].w = wi;
        float wh, wl;
        split_f32(wi, wh, wl);
        recs32[src].wh = wh;
        recs32[src].wl = wl;
        if (recs32s) {
            recs32s[i].wh = wh;
            recs32s[i].wl = wl;
        }
        if (w0 && drift) drift[src] = make_float2(__double2float_rd(dlo), __double2float_ru(dhi));
    }
    for (long long e = i; e < n_mom; e += (long long)gridDim.x * 32) mom[e] = 0ull;
    if (i == 0) {
        sc->flag_count = 0u;
        sc->band_count = 0u;
        if (push_to) *push_to = push;
    }
    if (groups && lane == 0 && i < n) groups[blockIdx.x].wmax = dkey_inv(wmax);
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __syncwarp();
    // the warps' maxima (a warp is a 32-seed group), loaded in parallel
    const volatile double *rows = part;
    unsigned long long top = 0ull;
#pragma unroll 4
    for (unsigned k = lane; k < gridDim.x; k += 32)
        top = max(top, (unsigned long long)__double_as_longlong(rows[(size_t)k * kPartStride]));
    double gsum = 0.0;  // <gf, p>: blocks of vw warps, lane-strided, then a fixed tree
    if (coef)
        for (unsigned k = lane; k * vw < gridDim.x; k += 32) {
            double b = 0.0;
#pragma unroll 2
            for (int e = 0; e < vw; ++e) b += rows[(size_t)(k * vw + e) * kPartStride + 1];
            gsum += b;
        }
    const double wref = dkey_inv(warp_max_key(top));
    if (groups) {
#pragma unroll 4
        for (unsigned k = lane; k * 32 < (unsigned)n; k += 32) {
            const double wm = dkey_inv((unsigned long long)__double_as_longlong(rows[(size_t)k * kPartStride]));
            groups[k].wgap = __double2float_rd(wref - wm);
        }
    }
    if (w0 && threadIdx.x < 32) {  // the drift range (max and min are order-independent)
        double x = -DBL_MAX, m = DBL_MAX;
        for (unsigned k = threadIdx.x; k < gridDim.x; k += 32) {
            x = fmax(x, *(volatile double *)&part[(size_t)k * kPartStride + 2]);
            m = fmin(m, *(volatile double *)&part[(size_t)k * kPartStride + 3]);
        }
        x = warp_max(x);
        m = warp_min(m);
        // the pixels a re-decision would settle in full have g3 <= D: bound their
        // count by the record's histogram (every bin up to D's); bin 0 (no
        // certified margin: FP64 near ties) costs a recording as much
        const float bD = __double2float_ru(__dsub_ru(x, m));
        const unsigned eD = bD > 0.f ? min(__float_as_uint(bD) >> 21, (unsigned)kIncBins - 1u) : 0u;
        unsigned cnt = 0u;
        if (g3_hist)
            for (unsigned e = threadIdx.x; e < (unsigned)kIncBins; e += 32u)
                cnt += (e > 0u && e <= eD) ? g3_hist[e] : 0u;
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (threadIdx.x == 0) {
            sc->drift_max = x;
            sc->drift_min = m;
            sc->drift_hi = __double2float_ru(x);
            sc->inc_go = (sc->inc_valid && g3_hist && cnt <= full_max) ? 1 : 0;
            // the incremental pass's band width and excluded-seed shift, rounded outwards
            sc->band_D = bD;
            // (less 2^-40 (|w_ref| + |w_ref0|): the scorers take w_ref as a float pair)
            const double wr0 = wref0 ? dkey_inv(*wref0) : wref;
            const double slack = ldexp(fabs(wref) + fabs(wr0), -40);
            sc->band_shift = __double2float_rd(__dsub_rd(__dsub_rd(__dsub_rd(wref, wr0), x), slack));
        }
    }
    if (coef) {
        gsum = warp_sum(gsum);
        if (lane == 0) sc->gp0 = gsum;
    }
    if (threadIdx.x == 0) {
        sc->wref_key = dkey(wref);
        split_f32(wref, sc->wref_h, sc->wref_l);
        sc->dual_done = 0u;
    }
}

// Seed records at new positions, one seed per thread, with the scalars of the pass: the
// blocks' maxima (w, ||A||_F, -lambda bound as ordered keys: no FP64 comparisons) go to
// `part`, the last block to finish reduces them and clears the pass's counters; mom's
// words are cleared on the way.  Bound: the FP64 chain of a seed (SPD test and
// eigenvalue bound, about 100 dependent operations of 64 clocks), so the blocks are
// small.  One launch where there were a clear, a reset and a 36 us kernel: 5 us.
template <int D>
__global__ void seed_prep_kernel(const GridDev g, const int n, const int n_pad,
                                 const double *__restrict__ x, const double *__restrict__ A,
                                 const double *__restrict__ w, SeedRec *__restrict__ recs,
                                 SeedRec32 *__restrict__ recs32, uint32_t *__restrict__ codes,
                                 unsigned long long *__restrict__ mom, const long long n_mom,
                                 unsigned long long *__restrict__ part, DevScalars *__restrict__ sc,
                                 const PtsGeo *__restrict__ box) {
    __shared__ unsigned long long sk[3];
    __shared__ bool last;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (threadIdx.x < 3) sk[threadIdx.x] = 0ull;
    for (long long e = i; e < n_mom; e += (long long)gridDim.x * blockDim.x) mom[e] = 0ull;
    SeedRec r;
    SeedRec32 r32;
    double wkey, frob, lam;
    int bad;
    build_seed<D>(i, n, x, A, w, r, r32, wkey, frob, lam, bad);
    const bool active = i < n;
    if (bad) atomicOr(&sc->status, bad);
    if (i < n_pad) {
        recs[i] = r;
        recs32[i] = r32;
        if (codes) codes[i] = seed_code<D>(g, r, active, box);
    }
    __syncthreads();
    const unsigned long long kw = warp_max_key(active ? dkey(wkey) : 0ull);
    const unsigned long long kf = warp_max_key(active ? (unsigned long long)__double_as_longlong(frob) : 0ull);
    const unsigned long long kl = warp_max_key(active ? ~(unsigned long long)__double_as_longlong(lam) : 0ull);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&sk[0], kw);
        atomicMax(&sk[1], kf);
        atomicMax(&sk[2], kl);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long *p = part + (size_t)blockIdx.x * kPartStride;
        p[0] = sk[0];
        p[1] = sk[1];
        p[2] = sk[2];
        __threadfence();
        last = atomicAdd(&sc->dual_done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    unsigned long long a = 0ull, b = 0ull, c = 0ull;
    for (unsigned k = threadIdx.x; k < gridDim.x; k += 32) {
        const volatile unsigned long long *p = part + (size_t)k * kPartStride;
        a = max(a, p[0]);
        b = max(b, p[1]);
        c = max(c, p[2]);
    }
    a = warp_max_key(a);
    b = warp_max_key(b);
    c = warp_max_key(c);
    if (threadIdx.x == 0) {
        sc->flag_count = 0u;
        sc->wref_key = a;
        split_f32(dkey_inv(a), sc->wref_h, sc->wref_l);
        sc->lam_abs_bits = b;
        sc->lam_min_bits = ~c;
        sc->dual_done = 0u;
        sc->inc_go = 0;     // a full pass: it records (incremental solves) ...
        sc->inc_valid = 0;  // ... and no earlier record holds for its records
    }
}

// Morton order of the seeds by counting: a block ranks 32 seeds (lane = seed), its
// eight warps counting an eighth of the codes each (code, then index, below the
// seed's), then copies their records to their scan positions.  n^2 / 32 warp steps over
// all SMs instead of a sort in one block (10^4 seeds: 190 us with the gather -> 12 us;
// 1000 seeds: 17 -> 4 us); the order is the same, by (code, index).
constexpr int kRankThreads = 256;
constexpr int kRankPiece = 4096;
__global__ void __launch_bounds__(kRankThreads)
    rank_kernel(const int n, const uint32_t *__restrict__ codes, uint32_t *__restrict__ scodes,
                int32_t *__restrict__ perm, const SeedRec *__restrict__ src, SeedRec *__restrict__ dst,
                const SeedRec32 *__restrict__ src32, SeedRec32 *__restrict__ dst32, const int n_pad) {
    __shared__ uint4 piece[kRankPiece / 4];
    __shared__ int part[kRankThreads / 32][32];
    __shared__ int rank[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 32, i = i0 + lane;
    const uint32_t ci = codes[i];
    // the codes in pieces of 4096 through shared memory; warp w counts an eighth of each
    int below = 0;
    for (int base = 0; base < n; base += kRankPiece) {
        const int m = min(kRankPiece, n_pad - base);  // a multiple of 256
        __syncthreads();
        for (int e = threadIdx.x; e < m / 4; e += kRankThreads)
            piece[e] = reinterpret_cast<const uint4 *>(codes + base)[e];
        __syncthreads();
        if (i0 >= n) continue;
        const int len = m / (kRankThreads / 32);
        int j = base + wid * len;
        const uint4 *c4 = piece + (wid * len >> 2);
#pragma unroll 4
        for (int e = 0; e < len / 4; ++e, j += 4) {  // padding codes count for no seed
            const uint4 c = c4[e];
            if (j + 4 <= i0) {
                below += (c.x <= ci) + (c.y <= ci) + (c.z <= ci) + (c.w <= ci);
            } else if (j >= i0 + 32) {
                below += (c.x < ci) + (c.y < ci) + (c.z < ci) + (c.w < ci);
            } else {
                below += (c.x < ci || (c.x == ci && j < i)) + (c.y < ci || (c.y == ci && j + 1 < i)) +
                         (c.z < ci || (c.z == ci && j + 2 < i)) + (c.w < ci || (c.w == ci && j + 3 < i));
            }
        }
    }
    part[wid][lane] = below;
    __syncthreads();
    if (wid == 0) {
        int r = 0;
#pragma unroll
        for (int k = 0; k < kRankThreads / 32; ++k) r += part[k][lane];
        if (i >= n) r = i;  // padding stays behind, in its order
        rank[lane] = r;
        scodes[r] = ci;
        perm[r] = i;
    }
    __syncthreads();
    const int e = threadIdx.x >> 3, c = threadIdx.x & 7;  // record, 16-byte piece
    const int to = rank[e];
    if (c < 4)
        reinterpret_cast<float4 *>(dst + to)[c] = reinterpret_cast<const float4 *>(src + i0 + e)[c];
    else
        reinterpret_cast<float4 *>(dst32 + to)[c - 4] = reinterpret_cast<const float4 *>(src32 + i0 + e)[c - 4];
}

template <int D>
__global__ void group_bounds_kernel(const int n, const SeedRec *__restrict__ recs, GroupBound *__restrict__ groups,
                                    const DevScalars *__restrict__ sc) {
    const int grp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (grp * 32 < n) group_bound_warp<D>(recs, n, grp, groups, dkey_inv(sc->wref_key));
}

// Pair p (of D (D + 1) / 2, a <= b in row order) of the upper triangle.
template <int D>
__device__ __forceinline__ void pair_ab(const int p, int &a, int &b) {
    if (D == 3) {
        a = p < 3 ? 0 : (p < 5 ? 1 : 2);
        b = p < 3 ? p : (p < 5 ? p - 2 : 2);
    } else {
        a = p < 2 ? 0 : 1;
        b = p < 2 ? p : 1;
    }
}
__device__ __forceinline__ double sel3(const double (&v)[3], const int a) {
    return a == 0 ? v[0] : (a == 1 ? v[1] : v[2]);
}

// The pair term of Q_i = sum_j (y_j - x_i)^T A_i (y_j - x_i) over cell i's pixels (|P| Q_i
// is the integral term of eq. (2.7)) that lane q of the cell's eight lanes takes: pair q,
// its factors A and M.  Q_ab = A_ab M_ab (A_ab + A_ba off the diagonal) with
// M_ab = sum_j (y - x)_a (y - x)_b written through the integer moments m, S1 = sum u,
// S2 = sum u u^T (u = 2k + 1, y = lo + h u / 2):
// M_ab = h_a h_b / 4 (S2_ab - S1_a S1_b / m) + m e_a e_b, e = centroid - x (lane a's).
template <int D>
__device__ __forceinline__ void dual_pair_term(const GridDev &g, const unsigned long long *__restrict__ mo,
                                               const double *__restrict__ xi, const double *__restrict__ Ai,
                                               const int q, const int a, const int b, double &Aab, double &Mab) {
    constexpr int NP = D * (D + 1) / 2;
    const int ax = min(q, D - 1);
    // no early exit on an empty cell: every load is issued before the first result
    // is needed (one memory round trip), and an empty cell's terms are dropped at the end
    const unsigned long long m0 = mo[0], s1 = mo[1 + ax], s2 = mo[1 + D + min(q, NP - 1)];
    const double xa = xi[ax], Aa = Ai[a * D + b], Ab = Ai[b * D + a];
    const double hh = 0.5 * sel3(g.h, ax), cc = 0.25 * sel3(g.h, a) * sel3(g.h, b);
    const double m = (double)m0;
    const double inv_m = 1.0 / m;  // one division; products with it differ from quotients by a few ulp
    const double S1 = (double)s1;
    const double e = __dsub_rn(__fma_rn(hh, __dmul_rn(S1, inv_m), sel3(g.lo, ax)), xa);
    const int base = threadIdx.x & 24;
    const double S1a = __shfl_sync(0xffffffffu, S1, base + a), S1b = __shfl_sync(0xffffffffu, S1, base + b);
    const double ea = __shfl_sync(0xffffffffu, e, base + a), eb = __shfl_sync(0xffffffffu, e, base + b);
    const double Cab = __fma_rn(-__dmul_rn(S1a, S1b), inv_m, (double)s2);
    Mab = __fma_rn(__dmul_rn(m, ea), eb, __dmul_rn(cc, Cab));
    Aab = a == b ? Aa : Aa + Ab;
    if (m0 == 0ull) Aab = Mab = 0.0;
}

// The same from FP64 element-measure moments (non-uniform discretisation):
// m = sum |P_j|, S1 = sum |P_j| y_j, S2 = sum |P_j| y_j y_j^T, and
// Q_ab = A_ab (S2_ab - S1_a x_b - x_a S1_b + m x_a x_b).
template <int D>
__device__ __forceinline__ void points_pair_term(const double *__restrict__ mo, const double *__restrict__ xi,
                                                 const double *__restrict__ Ai, const int q, const int a, const int b,
                                                 double &Aab, double &Mab) {
    constexpr int NP = D * (D + 1) / 2;
    const double m = mo[0];
    Mab = mo[1 + D + min(q, NP - 1)] - mo[1 + a] * xi[b] - xi[a] * mo[1 + b] + m * xi[a] * xi[b];
    Aab = a == b ? Ai[a * D + a] : Ai[a * D + b] + Ai[b * D + a];
}

// Partial results of the dual over some cells, spread over eight lanes (position p =
// lane & 7): g, <grad f, p> and sum v in `a` of positions 0, 1, 2, the smallest v as an
// ordered key in `a` of position 5; the largest |grad_k| / v_k as the pair (en, ed) of its
// cell in every position, compared through one product each in positions 3 and 4.
// One FP64 addition and one product join two rows: an FP64 instruction occupies a warp's
// scheduler for 64 clocks however few lanes it serves, and eight of them a step (one lane
// holding all) made the trees half of the kernel's time.
struct DualRow {
    double a, en, ed;
    __device__ static DualRow none(int p) {
        DualRow t;
        t.a = p == 5 ? __longlong_as_double((long long)dkey(DBL_MAX)) : 0.0;
        t.en = 0.0;
        t.ed = 1.0;
        return t;
    }
    __device__ void ratio(double on, double od, int p) {  // all products >= 0: ordered as integers
        const double prod = __dmul_rn(p == 4 ? en : on, p == 4 ? od : ed);
        const double other = __shfl_xor_sync(0xffffffffu, prod, 7);
        const long long mine = __double_as_longlong(prod), theirs = __double_as_longlong(other);
        if (p == 4 ? theirs > mine : mine > theirs) {
            en = on;
            ed = od;
        }
    }
    __device__ static double smaller(double x, double y) {
        const unsigned long long a = (unsigned long long)__double_as_longlong(x),
                                 b = (unsigned long long)__double_as_longlong(y);
        return a < b ? x : y;
    }
    __device__ void join(const DualRow &o, int p) {
        const double s = __dadd_rn(a, o.a);
        a = p == 5 ? smaller(a, o.a) : s;
        ratio(o.en, o.ed, p);
    }
    __device__ void join_lanes(int off, int p) {
        DualRow o;
        o.a = __shfl_xor_sync(0xffffffffu, a, off);
        o.en = __shfl_xor_sync(0xffffffffu, en, off);
        o.ed = __shfl_xor_sync(0xffffffffu, ed, off);
        join(o, p);
    }
    __device__ double value(int p) const { return p == 3 ? en : p == 4 ? ed : a; }  // a stored row's word p
    __device__ static DualRow load(const volatile double *row, int p) {
        DualRow t;
        t.a = row[min(p, 5)];
        t.en = row[3];
        t.ed = row[4];
        return t;
    }
};
static_assert(kPartStride == 6, "words of a stored row");

// Rows 4 / J lane groups apart: group k = lane / 8 holds the rows J k + j, j < J (J a power
// of two); joined in a fixed tree over neighbouring rows, `rows` of them (a power of two).
template <int MAXJ>
__device__ __forceinline__ void join_rows(DualRow (&t)[MAXJ], const int J, const int rows, const int p) {
#pragma unroll
    for (int w = 1; w < MAXJ; w <<= 1)
        if (w < J && w < rows) {
#pragma unroll
            for (int j = 0; j + w < MAXJ; j += 2 * w) t[j].join(t[j + w], p);
        }
    if (rows > J) t[0].join_lanes(8, p);
    if (rows > 2 * J) t[0].join_lanes(16, p);
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// address of this block's shared location in the cluster's block `rank`
__device__ __forceinline__ uint32_t cluster_map(const void *p, uint32_t rank) {
    uint32_t to;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return to;
}
__device__ __forceinline__ void cluster_store(uint32_t to, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(to), "d"(v) : "memory");
}
__device__ __forceinline__ int pow2_at_least(int v) { return v <= 1 ? 1 : 1 << (32 - __clz(v - 1)); }

// Per-cell dual terms, eight lanes per cell, then a deterministic reduction: a cluster's 64
// cells through fixed trees, the clusters' rows by the last cluster to finish.
//   g_i = (v_i - m_i |P|) w_i + |P| Q_i,  grad_i = v_i - m_i |P|  (eqs. (2.7), (2.8))
// kPoints: FP64 element-measure moments of a non-uniform discretisation
// (mom_pts), g_i = (v_i - m_i) w_i + Q_i, grad_i = v_i - m_i.
// The largest relative volume error max_i |grad_i| / v_i is tracked as the
// pair (|grad_k|, v_k) of its cell and divided once at the end.
//
// Bound: FP64 instructions, 64 clocks each in a warp's scheduler, and memory round trips of
// 600 to 1300 clocks (loads, the count of the clusters, the fence before the host's word).
// So the work is spread over schedulers, four warps a block (one each), four blocks a
// cluster, and no instruction serves one value alone.  Eight warps of 64 cells on one SM,
// a lane of each joining all six values: 13.4 us at n = 1000, 11 at n = 20; so 9.3 and 7.0.
constexpr int kDualBlocks = 4;                     // blocks of a cluster
constexpr int kDualThreads = 128;                  // four warps of four cells
constexpr int kDualCells = kDualBlocks * kDualThreads / 8;  // cells of a cluster's round

template <int D, bool kPoints = false>
__global__ void __launch_bounds__(kDualThreads) __cluster_dims__(kDualBlocks, 1, 1)
    dual_kernel(const GridDev g, const int n, const double *__restrict__ x,
                const double *__restrict__ A, const double *__restrict__ w,
                const double *__restrict__ v, const double *__restrict__ p_dir,
                const unsigned long long *__restrict__ mom, double *__restrict__ part,
                DevScalars *__restrict__ sc, double *g_out, double *grad_out, double *gf_out,
                double *err_out, DevScalars *__restrict__ host, const double *__restrict__ mom_pts = nullptr) {
    constexpr int K = moment_width(D), NP = D * (D + 1) / 2;
    constexpr int kWarps = kDualThreads / 32 * kDualBlocks;  // rows of a cluster
    __shared__ double rows[kWarps][kPartStride];
    const int lane = threadIdx.x & 31, p = lane & 7;
    const int rank = blockIdx.x % kDualBlocks, blk = blockIdx.x / kDualBlocks, nblk = gridDim.x / kDualBlocks;
    const int row = rank * (kDualThreads / 32) + (int)(threadIdx.x >> 5);
    cluster_arrive();  // waited for before the write into the first block's shared memory
    int a, b;
    pair_ab<D>(min(p, NP - 1), a, b);
    DualRow t = DualRow::none(p);
    // the last round's gradient is stored after the sums have been counted in: the fence
    // before that waits for a warp's earlier stores
    int i_last = -1;
    double gr_last = 0.0;
    auto put_gradient = [&]() {
        if (i_last < 0) return;
        if (p == 0 && grad_out) grad_out[i_last] = gr_last;
        if (p == 1 && gf_out) gf_out[i_last] = -gr_last;
    };
    const int i0 = blk * kDualCells + row * 4;  // the warp's first cell
    for (int c0 = i0; c0 < n; c0 += nblk * kDualCells) {
        const int cell = c0 + (lane >> 3);
        const bool real = cell < n;
        const int i = real ? cell : c0;
        const double vi = v[i], wi = w[i], pd = p_dir ? p_dir[i] : 0.0;
        const double mi = kPoints ? mom_pts[(size_t)i * K] : (double)mom[(size_t)i * K];
        double Aab, Mab;
        if (kPoints) points_pair_term<D>(mom_pts + (size_t)i * K, x + (size_t)i * D, A + (size_t)i * D * D, p, a, b, Aab, Mab);
        else dual_pair_term<D>(g, mom + (size_t)i * K, x + (size_t)i * D, A + (size_t)i * D * D, p, a, b, Aab, Mab);
        const double gr = kPoints ? __dsub_rn(vi, mi) : __dsub_rn(vi, __dmul_rn(mi, g.cell));
        // pairs q and q + 4 first, then q ^ 1, q ^ 2
        const double P = p < NP ? __dmul_rn(Aab, Mab) : 0.0;
        double Q = P;
        if (NP > 4) {
            const double F = __fma_rn(Aab, Mab, __shfl_xor_sync(0xffffffffu, P, 4));
            const double up = __shfl_xor_sync(0xffffffffu, F, 4);
            if (p + 4 < NP) Q = up;
        }
        Q += __shfl_xor_sync(0xffffffffu, Q, 1);
        Q += __shfl_xor_sync(0xffffffffu, Q, 2);
        const double u = __dmul_rn(gr, wi);
        const double f = kPoints ? __fma_rn(p == 1 ? -gr : gr, p == 1 ? pd : wi, p == 1 ? t.a : Q) : __fma_rn(p == 1 ? -gr : g.cell, p == 1 ? pd : Q, p == 1 ? t.a : u);
        const double s = __dadd_rn(t.a, p == 2 ? vi : f);
        const DualRow old = t;
        if (p == 5) t.a = DualRow::smaller(t.a, __longlong_as_double((long long)dkey(vi)));
        else t.a = p == 1 ? f : s;
        t.ratio(fabs(gr), vi, p);
        if (!real) {
            t = old;
        } else {
            if (p == 0 && (!(vi > 0.0) || !isfinite(vi))) atomicOr(&sc->status, ST_BAD_VOLUME);
            put_gradient();
            i_last = i;
            gr_last = gr;
        }
    }
    if (i0 < n) {
        t.join_lanes(8, p);
        t.join_lanes(16, p);
    }
    cluster_wait();
    if (lane < kPartStride && i0 < n) cluster_store(cluster_map(&rows[row][lane], 0), t.value(lane));
    cluster_arrive();
    if (row != 0) {
        put_gradient();
        cluster_wait();
        return;
    }
    cluster_wait();
    {  // the cluster's 16 rows, those of warps that hold cells
        constexpr int J = kWarps / 4;
        const int used = (min(n - i0, kDualCells) + 3) / 4;
        DualRow z[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int k = (lane >> 3) * J + j;
            z[j] = k < used ? DualRow::load(rows[k], p) : DualRow::none(p);
        }
        join_rows<J>(z, J, pow2_at_least(used), p);
        t = z[0];
    }
    constexpr int kWords = sizeof(DevScalars) / 4, kPer = (kWords + 31) / 32;
    unsigned word[kPer];
    if (nblk > 1) {
        if (lane < kPartStride) part[(size_t)blk * kPartStride + lane] = t.value(lane);
        __syncwarp();
        unsigned last = 0;
        if (lane == 0) last = count_in(&sc->dual_done) == nblk - 1;
        if (!__shfl_sync(0xffffffffu, last, 0)) {
            put_gradient();
            return;
        }
        __syncwarp();
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k)
        word[k] = reinterpret_cast<const volatile unsigned *>(sc)[min(k * 32 + lane, kWords - 1)];
    if (nblk > 1) {
        // the last cluster: 32 columns take the clusters in order (c, c + 32, ...), then a fixed tree
        constexpr int MJ = 8;
        const int cols = min(32, pow2_at_least(nblk)), J = max(1, cols / 4);
        DualRow z[MJ];
#pragma unroll
        for (int j = 0; j < MJ; ++j) {
            const int c = (lane >> 3) * J + j;
            z[j] = j < J && c < nblk ? DualRow::load(part + (size_t)c * kPartStride, p) : DualRow::none(p);
        }
        for (int c0 = 32; c0 < nblk; c0 += 32) {
#pragma unroll
            for (int j = 0; j < MJ; ++j) {
                const int c = c0 + (lane >> 3) * J + j;
                const DualRow o = j < J && c < nblk ? DualRow::load(part + (size_t)c * kPartStride, p) : DualRow::none(p);
                z[j].join(o, p);
            }
        }
        join_rows<MJ>(z, J, cols, p);
        t = z[0];
    }
    if (p == 3) t.a = __ddiv_rn(t.en, t.ed);
    if (p == 5) t.a = dkey_inv((unsigned long long)__double_as_longlong(t.a));
    if (lane < kPartStride && lane != 4) {
        // position -> field (g, dot_gp, sum_v, max_rel_err, -, min_v)
        const int field = lane == 0 ? 0 : lane == 1 ? 2 : lane == 2 ? 3 : lane == 3 ? 1 : 4;
        (&sc->g)[field] = t.a;
        if (lane == 0 && g_out) *g_out = t.a;
        if (lane == 3 && err_out) *err_out = t.a;
        if (host) (&host->g)[field] = t.a;
    }
    if (lane == 0) sc->dual_done = 0u;
    if (host) {  // the other scalars, then the pass's number, which the host waits for
        constexpr int w0 = offsetof(DevScalars, g) / 4, w1 = offsetof(DevScalars, sy) / 4, ws = offsetof(DevScalars, seq) / 4;
        static_assert(w1 - w0 == 10, "g, max_rel_err, dot_gp, sum_v, min_v in a row");
        unsigned seq = 0u;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int e = k * 32 + lane;
            if (k == ws / 32) seq = __shfl_sync(0xffffffffu, word[k], ws % 32) + 1u;
            if (e < kWords && e != ws && (e < w0 || e >= w1)) reinterpret_cast<volatile unsigned *>(host)[e] = word[k];
        }
        __syncwarp();
        if (lane == 0) {
            sc->seq = seq;
            __threadfence_system();
            *(volatile unsigned *)&host->seq = seq;
        }
    }
    put_gradient();
}

template <int D>
__global__ void centroid_kernel(const GridDev g, const int n, const double *__restrict__ x,
                                const unsigned long long *__restrict__ mom, double *x_out) {
    constexpr int K = moment_width(D);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const unsigned long long *mo = mom + (size_t)i * K;
    const double m = (double)mo[0];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const double xa = x[(size_t)i * D + a];
        x_out[(size_t)i * D + a] = mo[0] > 0ull ? g.lo[a] + 0.5 * g.h[a] * ((double)mo[1 + a] / m) : xa;
    }
}

__global__ void axpy_kernel(const int n, const double *a, const double t, const double *b, double *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = a[i] + t * b[i];
}

// The L-BFGS pairs (s_k, y_k) live in slots of a ring of `cap`; beside them the
// Gram entries gram[0][i][j] = s_i . y_j and gram[1][i][j] = y_i . y_j (slot
// indices), filled by the push kernel for every pair of slots that can be in
// the history together.  With them the two-loop recursion of the L-BFGS
// direction (Nocedal and Wright, Algorithm 7.4) needs only the 2 hist dot
// products s_k . g, y_k . g over the seeds; its scalar recursion then runs on
// the Gram entries and p is assembled in one pass as
//   p = -gamma g + sum_k gamma alpha_k y_k - sum_k (alpha_k - beta_k) s_k,
// the same vector as the two-loop form in exact arithmetic.
//
// FP64 runs at a few operations per clock per SM and every dependent global
// load costs about a microsecond of latency, so the dot products are spread
// over up to one block per SM (32 seeds per block range, a warp per dot, all
// of a block's loads in flight together) and the last block to finish reduces
// the per-block sums in block order (deterministic) and runs the scalar part
// in one warp, column by column (one shuffle per step).  The push kernel also
// forms the next direction's dot products (for both outcomes of its curvature
// test), so an accepted step costs two launches: push-and-coefficients, then p.
constexpr int kLbfgsMax = 32;    // ring capacity the kernels below support
static_assert(kLbfgsDots >= 5 + 5 * (kLbfgsMax - 1), "partial-sum rows hold the push's products");
constexpr int kLbT = 1024;       // threads per block of the dot-product kernels
constexpr int kLbR = 32;         // seeds per block range
constexpr int kLbP = 64;         // threads per block of the p kernel

// Sum over the warp of five values, each by warp_sum's tree (pairs 16, 8, ... apart), in 8
// additions where five trees take 25: after a step that pairs two values, half of the
// lanes carry on with each.  The sum of value c is returned in the lanes where
// dot_of_lane() is c.
__device__ __forceinline__ double warp_sum5(const double (&v)[5]) {
    const int lane = threadIdx.x & 31;
    auto both = [&](double a, double b, int off) {  // lanes without the bit go on with a, those with it b
        const bool hi = lane & off;
        const double keep = hi ? b : a, send = hi ? a : b;
        return keep + __shfl_xor_sync(0xffffffffu, send, off);
    };
    const double r01 = both(v[0], v[1], 16), r23 = both(v[2], v[3], 16);
    double r4 = v[4] + __shfl_xor_sync(0xffffffffu, v[4], 16);
    const double r03 = both(r01, r23, 8);
    r4 += __shfl_xor_sync(0xffffffffu, r4, 8);
    double r = both(r03, r4, 4);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    return r;
}
__device__ __forceinline__ int dot_of_lane(int lane) { return lane & 4 ? 4 : ((lane >> 3) & 1) * 2 + ((lane >> 4) & 1); }

// Partial dot products of one block over its ranges of 32 seeds (range r
// starts at (blockIdx.x + r gridDim.x) 32): dot d (of nd) is sum_i f(d, i),
// warp w takes the dots d = w mod 32.  part[blockIdx.x * kLbfgsDots + d]
// receives the block's sums.
template <class F>
__device__ void block_partial_dots(const int nd, const int n, F f, double *part) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int d = wid; d < nd; d += kLbT / 32) {
        double v = 0.0;
        for (int r0 = blockIdx.x * kLbR; r0 < n; r0 += gridDim.x * kLbR)
            if (r0 + lane < n) v += f(d, r0 + lane);
        v = warp_sum(v);
        if (lane == 0) part[(size_t)blockIdx.x * kLbfgsDots + d] = v;
    }
}

// Called by every block after its partial sums are stored: true in the last
// block to arrive (which then sees every block's sums).
__device__ bool lbfgs_last_block(DevScalars *sc) {
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&sc->lbfgs_done, 1u) == gridDim.x * gridDim.y - 1;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// out[d] = sum over blocks (lane-strided, then the warp tree) of part[.][d], d < nd.
__device__ void reduce_partials(const int nd, const double *part, double *out) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int d = wid; d < nd; d += (int)(blockDim.x >> 5)) {
        double v = 0.0;
        for (unsigned b = lane; b < gridDim.x; b += 32) v += *(const volatile double *)(part + (size_t)b * kLbfgsDots + d);
        v = warp_sum(v);
        if (lane == 0) out[d] = v;
    }
    __syncthreads();
}

// Shared state of the scalar part: the history's Gram entries (padded rows:
// the column-wise steps read one column across the lanes), 1 / s.y, s_k . g,
// y_k . g and the slots, k = 0 the newest pair.
struct LbfgsScalars {
    double sy[kLbfgsMax][kLbfgsMax + 1];  // s_k . y_j
    double yy[kLbfgsMax][kLbfgsMax + 1];  // y_k . y_j
    double rh[kLbfgsMax], sg[kLbfgsMax], yg[kLbfgsMax];
    int slot[kLbfgsMax];
};

// The last block's gather of the history's Gram entries and 1 / s.y.
__device__ void load_gram(LbfgsScalars &L, const int hist, const int cap, const double *__restrict__ gram,
                          const double *__restrict__ rho) {
    for (int e = threadIdx.x; e < hist * hist; e += blockDim.x) {
        const int k = e / hist, j = e % hist;
        L.sy[k][j] = gram[(size_t)L.slot[k] * cap + L.slot[j]];
        L.yy[k][j] = gram[(size_t)cap * cap + (size_t)L.slot[k] * cap + L.slot[j]];
    }
    for (int k = threadIdx.x; k < hist; k += blockDim.x) L.rh[k] = rho[L.slot[k]];
    __syncthreads();
}

// The two-loop recursion on the Gram entries, by warp 0, column by column:
// alpha_k = rho_k (s_k . g - sum_{j<k} alpha_j s_k . y_j)          (newest first)
// c_k = alpha_k - rho_k (gamma y_k . q + sum_{j>k} c_j s_j . y_k)   (oldest first)
// with y_k . q = y_k . g - sum_j alpha_j y_k . y_j (summed beside the alphas: the chain of
// an alpha leaves the FP64 unit idle); then the coefficients of p.  Pair k lies in row
// k + base of L.
__device__ void lbfgs_coefficients(const LbfgsScalars &L, const int base, const int hist, const double gamma,
                                   LbfgsCoef *coef) {
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    const bool halves = hist <= 16;  // lanes 16 .. 31 sum y_k . q beside lanes 0 .. 15, by the same instruction
    const int k0 = halves ? lane & 15 : lane, row = min(k0 + base, kLbfgsMax - 1);
    const double rh = L.rh[row], sg = L.sg[row];
    double t = 0.0, al = 0.0, yq = L.yg[row];
    if (halves) {
        const bool up = lane >= 16;
        double acc = up ? yq : 0.0;
        const double(*M)[kLbfgsMax + 1] = up ? L.yy : L.sy;
#pragma unroll 2
        for (int k = 0; k < hist; ++k) {
            const double mk = M[row][k + base];
            double a = rh * (sg - acc);
            a = __shfl_sync(0xffffffffu, a, k);
            if (lane == k) al = a;
            acc = __fma_rn(up ? -a : a, mk, acc);
        }
        yq = __shfl_sync(0xffffffffu, acc, lane | 16);
    } else {
#pragma unroll 2
        for (int k = 0; k < hist; ++k) {
            const double sy = L.sy[row][k + base], yy = L.yy[row][k + base];
            double a = rh * (sg - t);
            a = __shfl_sync(0xffffffffu, a, k);
            if (lane == k) al = a;
            if (lane > k && lane < hist) t += a * sy;
            yq -= a * yy;
        }
    }
    double u = 0.0, c = 0.0;
#pragma unroll 2
    for (int k = hist - 1; k >= 0; --k) {
        const double sy = L.sy[k + base][row];
        double ck = al - rh * (gamma * yq + u);
        ck = __shfl_sync(0xffffffffu, ck, k);
        if (lane == k) c = ck;
        if (lane < k) u += ck * sy;
    }
    // p = -gamma g + sum_k gamma alpha_k y_k - sum_k (alpha_k - beta_k) s_k
    if (lane < hist) {
        coef->cs[lane] = -c;
        coef->cy[lane] = gamma * al;
        coef->slot[lane] = L.slot[row];
    }
    if (lane == 0) {
        coef->hist = hist;
        coef->gamma = gamma;
    }
}

// Coefficients of p = -H gf (H0 = gamma I, the stored pairs newest at slot
// `newest`).  With use_pair, the pair just pushed (slot newest_acc) is used if
// it passed the push kernel's curvature test: then hist_acc pairs and
// gamma = s.y / y.y.
__global__ void __launch_bounds__(kLbT)
    lbfgs_dots_kernel(const int n, int hist, int newest, const int cap, double gamma, const int use_pair,
                      const int hist_acc, const int newest_acc, const double *__restrict__ S,
                      const double *__restrict__ Y, const double *__restrict__ rho,
                      const double *__restrict__ gram, const double *__restrict__ gf, double *part,
                      LbfgsCoef *coef, DevScalars *sc) {
    __shared__ LbfgsScalars L;
    __shared__ double dots[2 * kLbfgsMax];
    if (use_pair && sc->pair_ok) {
        hist = hist_acc;
        newest = newest_acc;
        gamma = sc->sy / sc->yy;
    }
    hist = min(hist, kLbfgsMax - 1);
    for (int k = threadIdx.x; k < hist; k += blockDim.x) L.slot[k] = (newest - k + cap) % cap;
    __syncthreads();
    // dots 2k: s_k . g, 2k + 1: y_k . g
    block_partial_dots(2 * hist, n, [&](int d, int i) {
        return ((d & 1) ? Y : S)[(size_t)L.slot[d >> 1] * n + i] * gf[i];
    }, part);
    if (!lbfgs_last_block(sc)) return;
    reduce_partials(2 * hist, part, dots);
    for (int k = threadIdx.x; k < hist; k += blockDim.x) {
        L.sg[k] = dots[2 * k];
        L.yg[k] = dots[2 * k + 1];
    }
    load_gram(L, hist, cap, gram, rho);
    lbfgs_coefficients(L, 0, hist, gamma, coef);
    if (threadIdx.x == 0) sc->lbfgs_done = 0u;
}

// p = -gamma gf + sum_k (cy_k y_k + cs_k s_k) and <gf, p> into sc->gp0.
__global__ void __launch_bounds__(kLbP)
    lbfgs_pdir_kernel(const int n, const LbfgsCoef *__restrict__ coef, const double *__restrict__ S,
                      const double *__restrict__ Y, const double *__restrict__ gf, double *__restrict__ p,
                      double *part, DevScalars *sc) {
    __shared__ double cy[kLbfgsMax], cs[kLbfgsMax];
    __shared__ int slot[kLbfgsMax];
    __shared__ double red[kLbP / 32];
    const int hist = coef->hist;
    const double gamma = coef->gamma;
    for (int k = threadIdx.x; k < hist; k += blockDim.x) {
        cy[k] = coef->cy[k];
        cs[k] = coef->cs[k];
        slot[k] = coef->slot[k];
    }
    __syncthreads();
    double d = 0.0;
    for (int i = blockIdx.x * kLbP + threadIdx.x; i < n; i += gridDim.x * kLbP) {
        const double g = gf[i];
        double v = -gamma * g;
#pragma unroll 8
        for (int k = 0; k < hist; ++k) {
            const size_t o = (size_t)slot[k] * n + i;
            v += cy[k] * Y[o] + cs[k] * S[o];
        }
        p[i] = v;
        d += g * v;
    }
    d = warp_sum(d);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = d;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kLbP / 32; ++w) t += red[w];
        part[(size_t)blockIdx.x * kLbfgsDots] = t;
    }
    if (!lbfgs_last_block(sc)) return;
    if (threadIdx.x < 32) {
        double t = 0.0;
        for (unsigned b = threadIdx.x; b < gridDim.x; b += 32) t += *(const volatile double *)(part + (size_t)b * kLbfgsDots);
        t = warp_sum(t);
        if (threadIdx.x == 0) {
            sc->gp0 = t;
            sc->lbfgs_done = 0u;
        }
    }
}

// Store the pair s = Wt - W, y = gft - gf in the slot after `newest`; sy, yy, ss, the
// curvature test and 1 / s.y into sc and rho; the Gram entries of the new pair with
// itself and with the pairs that are kept beside it.  With dir, also the coefficients of
// the next direction for the gradient gft: the pair taken (then hist_acc = min(hist + 1,
// history) pairs newest first from the new slot, gamma = s.y / y.y) if it passes the
// test, else the hist pairs before it with the given gamma.
// The state, written by the trial's first kernel: with pend, the pair pushed before (slot p_slot) has not been looked at by
// the host: it is part of the history if its test passed.  The push follows each trial of
// a line search before the host knows the trial's value, so that the device does not wait
// for the host; the slot written is in no history, so a push that
// the search does not accept leaves nothing behind.  Nothing is formed at an evaluation
// that met eps; Wbest takes Wt where the evaluation's error is below best_err.
//
// Unit u = 0 is the new pair (s.y, y.y, s.s, s.g, y.g), unit u > 0 the pair j = u - 1
// before it (s.y_j, s_j.y, y.y_j, s_j.g, y_j.g): a warp takes a unit over 32 seeds (lane =
// seed, s and y formed in registers), the units of a range spread over gridDim.y blocks.
// Bound: latency; memory round trips and the recursion's chain of 4 FP64 operations a pair
// and direction.  A warp per dot product with a tree each, the pair read back from memory
// and the Gram entries gathered at the end: 20.8 us at n = 1000 and ten pairs; so 8.9 us.
__global__ void __launch_bounds__(kLbT)
    lbfgs_push_kernel(const int n, const int cap, const PushState *__restrict__ state, const double *__restrict__ W,
                      const double *__restrict__ Wt, const double *__restrict__ gf, const double *__restrict__ gft,
                      double *S, double *Y, double *__restrict__ rho, double *__restrict__ gram, double *part,
                      DevScalars *sc, const int dir, LbfgsCoef *coef, double *__restrict__ Wbest) {
    __shared__ LbfgsScalars L;
    __shared__ double dots[kLbfgsMax][5];
    __shared__ bool pair_ok, last;
    __shared__ double gamma_new;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const double err = sc->max_rel_err;
    const PushState ps = *state;
    const double psy = sc->sy, pyy = sc->yy;  // of the pair before; the last block replaces them
    const bool taken = ps.pend && sc->pair_ok;
    const int newest = taken ? ps.p_slot : ps.newest;
    const int hist = taken ? ps.hist_acc : ps.hist;
    const int slot = (newest + 1) % cap, hist_acc = min(hist + 1, ps.history);
    if (Wbest && err < ps.best_err && blockIdx.y == gridDim.y - 1 && wid == nw - 1)
        for (int i = blockIdx.x * kLbR + lane; i < n; i += gridDim.x * kLbR) Wbest[i] = Wt[i];
    if (Wbest && err < ps.eps) return;
    const int np = min(hist_acc - 1, kLbfgsMax - 1);
    const int nh = dir ? min(hist, kLbfgsMax - 1) : 0;
    const int m = max(np, nh), units = m + 1;
    double *gsy = gram, *gyy = gram + (size_t)cap * cap;
    auto prev = [&](int j) {  // slot of the j-th pair before the new one
        const int q = slot - 1 - j;
        return q < 0 ? q + cap : q;
    };
    // the old pairs' Gram entries, needed by the last block: on their way early (row 0 of L is
    // the new pair); a warp takes a row, a lane a column (there is a warp for every pair)
    const bool old = dir && wid < m && lane < m;
    const size_t og = old ? (size_t)prev(wid) * cap + prev(lane) : 0;
    const double osy = old ? gsy[og] : 0.0, oyy = old ? gyy[og] : 0.0;
    const double orh = wid == 0 && lane < m ? rho[prev(lane)] : 0.0;
    const size_t rows = gridDim.x;
    for (int u = wid * gridDim.y + blockIdx.y; u < units; u += gridDim.y * nw) {
        const double *sj = S + (size_t)(u ? prev(u - 1) : 0) * n, *yj = Y + (size_t)(u ? prev(u - 1) : 0) * n;
        double v[5];
        bool first = true;
        for (int i0 = blockIdx.x * kLbR; i0 < n; i0 += gridDim.x * kLbR) {
            const int i = min(i0 + lane, n - 1);
            const bool in = i0 + lane < n;
            const double s = Wt[i] - W[i], g = gft[i], y = g - gf[i];
            const double a = u ? sj[i] : s, b = u ? yj[i] : y;
            // new pair: a = s, b = y; else a = s_j, b = y_j
            const double d[5] = {__dmul_rn(s, b), __dmul_rn(u ? a : y, y), __dmul_rn(u ? y : s, u ? b : s), __dmul_rn(a, g),
                                 __dmul_rn(b, g)};
#pragma unroll
            for (int c = 0; c < 5; ++c) v[c] = first ? (in ? d[c] : 0.0) : in ? __dadd_rn(v[c], d[c]) : v[c];
            first = false;
        }
        const double r = warp_sum5(v);
        if ((lane & 3) == 0 && (lane == 4 || !(lane & 4)))
            part[(size_t)(u * 5 + dot_of_lane(lane)) * rows + blockIdx.x] = r;
    }
    __syncthreads();
    if (threadIdx.x == 0) last = count_in(&sc->lbfgs_done) == gridDim.x * gridDim.y - 1;
    if (blockIdx.y == 0 && wid == nw - 1)  // the pair itself, after the count (the fence before it would wait)
        for (int i = blockIdx.x * kLbR + lane; i < n; i += gridDim.x * kLbR) {
            S[(size_t)slot * n + i] = Wt[i] - W[i];
            Y[(size_t)slot * n + i] = gft[i] - gf[i];
        }
    if (dir) {
        if (old) {
            L.sy[wid + 1][lane + 1] = osy;
            L.yy[wid + 1][lane + 1] = oyy;
        }
        if (wid == 0 && lane <= m) L.slot[lane] = lane == 0 ? slot : prev(lane - 1);
        if (wid == 0 && lane < m) L.rh[lane + 1] = orh;
    }
    __syncthreads();
    if (!last) return;
    for (int u = wid; u < units; u += nw) {
        double v[5];
        const volatile double *pp = part + (size_t)u * 5 * rows;
#pragma unroll
        for (int c = 0; c < 5; ++c) v[c] = lane < (int)rows ? pp[(size_t)c * rows + lane] : 0.0;
        for (unsigned b = lane + 32; b < rows; b += 32)
#pragma unroll
            for (int c = 0; c < 5; ++c) v[c] += pp[(size_t)c * rows + b];
        if (rows > 1) {
            const double r = warp_sum5(v);
            if ((lane & 3) == 0 && (lane == 4 || !(lane & 4))) dots[u][dot_of_lane(lane)] = r;
        } else if (lane == 0) {
#pragma unroll
            for (int c = 0; c < 5; ++c) dots[u][c] = v[c];
        }
    }
    __syncthreads();
    const double vsy = dots[0][0], vyy = dots[0][1], vss = dots[0][2];
    // the test in one warp, the new pair's quotients in another, its Gram entries in the rest
    if (threadIdx.x == 0) {
        // vsy > 1e-12 sqrt(vss vyy): by the squares where they decide it clearly
        const double prod = vss * vyy, sq = vsy * vsy;
        const bool clear = vsy > 0.0 && sq > 1e-290 && prod < 1e290 && sq > 1.0001e-24 * prod;
        const bool ok = (clear || vsy > 1e-12 * sqrt(prod)) && vyy > 0.0;
        sc->pair_ok = ok ? 1 : 0;
        pair_ok = ok;
    }
    if (wid == 1 && lane < 2) {  // 1 / s.y and s.y / y.y side by side
        const double num = lane == 0 ? 1.0 : vsy, den = lane == 0 ? vsy : vyy;
        const double r = lane == 1 || vsy != 0.0 ? num / den : 0.0;
        if (lane == 0) {
            rho[slot] = r;
            L.rh[0] = r;
        } else {
            gamma_new = r;
        }
    }
    if ((int)threadIdx.x == (int)blockDim.x - 1) {
        gsy[(size_t)slot * cap + slot] = vsy;
        gyy[(size_t)slot * cap + slot] = vyy;
        sc->sy = vsy;
        sc->yy = vyy;
        sc->ss = vss;
        L.sy[0][0] = vsy;
        L.yy[0][0] = vyy;
        L.sg[0] = dots[0][3];
        L.yg[0] = dots[0][4];
    }
    for (int j = threadIdx.x; j < m; j += blockDim.x) {
        const double *d = dots[j + 1];
        L.sy[0][j + 1] = d[0];
        L.sy[j + 1][0] = d[1];
        L.yy[0][j + 1] = L.yy[j + 1][0] = d[2];
        L.sg[j + 1] = d[3];
        L.yg[j + 1] = d[4];
        if (j < np) {
            const int q = prev(j);
            gsy[(size_t)slot * cap + q] = d[0];
            gsy[(size_t)q * cap + slot] = d[1];
            gyy[(size_t)slot * cap + q] = d[2];
            gyy[(size_t)q * cap + slot] = d[2];
        }
    }
    if (dir) {
        __syncthreads();
        const bool ok = pair_ok;
        lbfgs_coefficients(L, ok ? 0 : 1, ok ? min(hist_acc, kLbfgsMax - 1) : nh, ok ? gamma_new : taken ? psy / pyy : ps.gamma, coef);
    }
    if (threadIdx.x == 0) sc->lbfgs_done = 0u;
}

}  // namespace

// Threads per block of the seed preparation: 64 (two warps, spreading the FP64 work over
// more SMs) while the blocks fit the workspace's partial-sum rows, else 256.  The same
// blocks are the units in which an evaluation's first kernel sums <gf, p>.
static int prep_threads(int n_pad, const Workspace &ws) { return n_pad / 64 <= ws.part_rows ? 64 : 256; }

cudaError_t launch_eval_begin(int n, const double *W0, double t, const double *pdir, double *Wt,
                              unsigned long long *mom, Workspace &ws, cudaStream_t st, bool form_p,
                              const double *w0, unsigned full_max, const PushState *push) {
    const unsigned long long *wref0 = w0 ? ws.inc_aux : nullptr;
    const unsigned *hist = w0 ? ws.inc_hist : nullptr;
    const int n_pad = ((n + kChunk - 1) / kChunk) * kChunk;
    const long long n_mom = (long long)n * moment_width(ws.dim);
    if (n_pad == 0) return cudaSuccess;
    const bool fp = form_p && pdir;
    eval_begin_kernel<<<n_pad / 32, 32, 0, st>>>(n, n_pad, prep_threads(n_pad, ws) / 32, n_mom, W0, t, const_cast<double *>(pdir), Wt,
                                                   ws.sorted ? ws.perm : nullptr, ws.recs, ws.recs32,
                                                   ws.sorted ? ws.recs32s : nullptr, ws.groups, mom, ws.part, ws.sc,
                                                   fp ? ws.lb_coef : nullptr, ws.S, ws.Y, ws.gf, w0, wref0,
                                                   hist, full_max, w0 ? ws.inc_drift : nullptr, push ? *push : PushState{},
                                                   push ? ws.push_state : nullptr);
    return cudaGetLastError();
}

const void *eval_begin_kernel_fn() { return reinterpret_cast<const void *>(eval_begin_kernel); }

// The same launch as launch_eval_begin, written into a kernel node of an
// instantiated graph (only the trial step t changes between replays).
cudaError_t set_eval_begin_node(cudaGraphExec_t exec, cudaGraphNode_t node, int n, const double *W0, double t,
                                const double *pdir, double *Wt, unsigned long long *mom, Workspace &ws,
                                bool form_p, const double *w0, unsigned full_max, const PushState *push) {
    const unsigned long long *wref0 = w0 ? ws.inc_aux : nullptr;
    const unsigned *hist = w0 ? ws.inc_hist : nullptr;
    float2 *drift = w0 ? ws.inc_drift : nullptr;
    PushState ps = push ? *push : PushState{}, *to = push ? ws.push_state : nullptr;
    int n_pad = ((n + kChunk - 1) / kChunk) * kChunk;
    long long n_mom = (long long)n * moment_width(ws.dim);
    const int32_t *perm = ws.sorted ? ws.perm : nullptr;
    SeedRec *recs = ws.recs;
    SeedRec32 *recs32 = ws.recs32, *recs32s = ws.sorted ? ws.recs32s : nullptr;
    GroupBound *groups = ws.groups;
    double *part = ws.part;
    DevScalars *sc = ws.sc;
    double *pd = const_cast<double *>(pdir);
    const LbfgsCoef *coef = form_p && pdir ? ws.lb_coef : nullptr;
    const double *S = ws.S, *Y = ws.Y, *gfv = ws.gf;
    int vw = prep_threads(n_pad, ws) / 32;
    void *args[] = {&n,      &n_pad,   &vw,    &n_mom,  &W0,  &t,    &pd, &Wt,   &perm, &recs, &recs32,
                    &recs32s, &groups, &mom, &part, &sc, &coef, &S, &Y, &gfv, &w0, &wref0, &hist, &full_max,
                    &drift, &ps, &to};
    cudaKernelNodeParams p{};
    p.func = reinterpret_cast<void *>(eval_begin_kernel);
    p.gridDim = dim3(n_pad / 32);
    p.blockDim = dim3(32);
    p.sharedMemBytes = 0;
    p.kernelParams = args;
    p.extra = nullptr;
    return cudaGraphExecKernelNodeSetParams(exec, node, &p);
}

// Incremental pass, before scoring: a re-decision starts from the recorded
// moments; a recording clears the margin histogram its scorer fills.
__global__ void inc_prepare_kernel(const long long n_mom, unsigned long long *__restrict__ mom,
                                   const unsigned long long *__restrict__ mom0, unsigned *__restrict__ hist,
                                   const DevScalars *__restrict__ sc) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (sc->inc_go) {
        for (long long e = i; e < n_mom; e += stride) mom[e] = mom0[e];
    } else {
        for (long long e = i; e < kIncBins; e += stride) hist[e] = 0u;
    }
}

// Incremental pass, after rescoring: a recording keeps its moments, weights and
// w_ref for the re-decisions that follow.
__global__ void inc_commit_kernel(const int n, const long long n_mom, const unsigned long long *__restrict__ mom,
                                  const double *__restrict__ w, unsigned long long *__restrict__ mom0,
                                  double *__restrict__ w0, unsigned long long *__restrict__ aux,
                                  DevScalars *__restrict__ sc) {
    if (sc->inc_go) return;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long e = i; e < n_mom; e += (long long)gridDim.x * blockDim.x) mom0[e] = mom[e];
    for (long long e = i; e < n; e += (long long)gridDim.x * blockDim.x) w0[e] = w[e];
    if (i == 0) {
        aux[0] = sc->wref_key;
        sc->inc_valid = 1;
    }
}

cudaError_t launch_inc_prepare(int n, unsigned long long *mom, Workspace &ws, cudaStream_t st) {
    const long long n_mom = (long long)n * moment_width(ws.dim);
    const int blocks = (int)std::max<long long>(1, std::min<long long>((n_mom + 255) / 256, 4 * ws.sms));
    inc_prepare_kernel<<<blocks, 256, 0, st>>>(n_mom, mom, ws.inc_mom0, ws.inc_hist, ws.sc);
    return cudaGetLastError();
}

cudaError_t launch_inc_commit(int n, const unsigned long long *mom, const double *w, Workspace &ws,
                              cudaStream_t st) {
    const long long n_mom = (long long)n * moment_width(ws.dim);
    const int blocks = (int)std::max<long long>(1, std::min<long long>((n_mom + 255) / 256, 4 * ws.sms));
    inc_commit_kernel<<<blocks, 256, 0, st>>>(n, n_mom, mom, w, ws.inc_mom0, ws.inc_w0, ws.inc_aux, ws.sc);
    return cudaGetLastError();
}

cudaError_t launch_seed_prep(const GridDev &g, int n, const double *x, const double *A,
                             const double *w, Workspace &ws, unsigned long long *mom, long long n_mom,
                             cudaStream_t st, const PtsGeo *box) {
    const int n_pad = ((n + kChunk - 1) / kChunk) * kChunk;
    // Morton order for the scoring scan when the workspace has the buffers
    ws.sorted = ws.recs_tmp && ws.codes && ws.scodes && ws.perm && ws.recs32s && n_pad <= kSortMax;
    SeedRec *dst = ws.sorted ? ws.recs_tmp : ws.recs;
    uint32_t *codes = ws.sorted ? ws.codes : nullptr;
    unsigned long long *part = reinterpret_cast<unsigned long long *>(ws.part);
    const int tpb = prep_threads(n_pad, ws);
    if (g.dim == 3)
        seed_prep_kernel<3><<<n_pad / tpb, tpb, 0, st>>>(g, n, n_pad, x, A, w, dst, ws.recs32, codes, mom, n_mom, part,
                                                         ws.sc, box);
    else
        seed_prep_kernel<2><<<n_pad / tpb, tpb, 0, st>>>(g, n, n_pad, x, A, w, dst, ws.recs32, codes, mom, n_mom, part,
                                                         ws.sc, box);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (ws.cond_read) {  // the host waits for this copy while the ranking runs
        e = cudaMemcpyAsync(&ws.sc_host->lam_abs_bits, &ws.sc->lam_abs_bits, 2 * sizeof(unsigned long long),
                            cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaEventRecord(ws.cond_ev, st);
        if (e != cudaSuccess) return e;
    }
    if (!ws.sorted) return cudaSuccess;
    rank_kernel<<<n_pad / 32, kRankThreads, 0, st>>>(n, ws.codes, ws.scodes, ws.perm, ws.recs_tmp, ws.recs, ws.recs32,
                                                     ws.recs32s, n_pad);
    return cudaGetLastError();
}

cudaError_t launch_group_bounds(int n, Workspace &ws, cudaStream_t st) {
    if (!ws.groups) return cudaSuccess;
    const int groups = (n + 31) / 32;
    const int blocks = (groups * 32 + 255) / 256;
    if (ws.dim == 3) group_bounds_kernel<3><<<blocks, 256, 0, st>>>(n, ws.recs, ws.groups, ws.sc);
    else group_bounds_kernel<2><<<blocks, 256, 0, st>>>(n, ws.recs, ws.groups, ws.sc);
    return cudaGetLastError();
}

// Clusters of the dual kernel: 64 cells each, at most the workspace's partial rows.
static int dual_blocks(int n, const Workspace &ws) {
    return std::max(1, std::min((n + kDualCells - 1) / kDualCells, ws.part_rows));
}

cudaError_t launch_dual(const GridDev &g, int n, const double *x, const double *A, const double *w,
                        const double *v, const double *p_dir, const unsigned long long *moments,
                        Workspace &ws, double *g_out, double *grad_out, double *gf_out,
                        double *err_out, cudaStream_t st, DevScalars *host) {
    const int blocks = dual_blocks(n, ws);
    if (g.dim == 3)
        dual_kernel<3><<<blocks * kDualBlocks, kDualThreads, 0, st>>>(g, n, x, A, w, v, p_dir, moments, ws.part, ws.sc, g_out,
                                                   grad_out, gf_out, err_out, host);
    else
        dual_kernel<2><<<blocks * kDualBlocks, kDualThreads, 0, st>>>(g, n, x, A, w, v, p_dir, moments, ws.part, ws.sc, g_out,
                                                   grad_out, gf_out, err_out, host);
    return cudaGetLastError();
}

cudaError_t launch_points_dual(int dim, int n, const double *x, const double *A, const double *w, const double *v,
                               const double *mom_pts, Workspace &ws, double *g_out, double *grad_out,
                               double *err_out, cudaStream_t st) {
    const int blocks = dual_blocks(n, ws);
    GridDev g;
    memset(&g, 0, sizeof g);
    g.dim = dim;
    if (dim == 3)
        dual_kernel<3, true><<<blocks * kDualBlocks, kDualThreads, 0, st>>>(g, n, x, A, w, v, nullptr, nullptr, ws.part, ws.sc, g_out,
                                                         grad_out, nullptr, err_out, nullptr, mom_pts);
    else
        dual_kernel<2, true><<<blocks * kDualBlocks, kDualThreads, 0, st>>>(g, n, x, A, w, v, nullptr, nullptr, ws.part, ws.sc, g_out,
                                                         grad_out, nullptr, err_out, nullptr, mom_pts);
    return cudaGetLastError();
}

cudaError_t launch_centroids(const GridDev &g, int n, const double *x,
                             const unsigned long long *moments, double *x_out, cudaStream_t st) {
    const int blocks = (n + 255) / 256;
    if (g.dim == 3)
        centroid_kernel<3><<<blocks, 256, 0, st>>>(g, n, x, moments, x_out);
    else
        centroid_kernel<2><<<blocks, 256, 0, st>>>(g, n, x, moments, x_out);
    return cudaGetLastError();
}

cudaError_t launch_axpy(int n, const double *a, double t, const double *b, double *out,
                        cudaStream_t st) {
    axpy_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, a, t, b, out);
    return cudaGetLastError();
}

// The dot-product kernels take one block per 32 seeds, the p kernel one per 64,
// each at most one block per SM (the workspace's partial-sum rows).
static int lbfgs_blocks(int n, int per, const Workspace &ws) {
    return std::max(1, std::min((n + per - 1) / per, ws.lb_rows));
}

cudaError_t launch_lbfgs_direction(int n, int hist, int newest, int cap, double gamma, bool use_pair,
                                   int hist_acc, int newest_acc, Workspace &ws, cudaStream_t st) {
    if (cap > kLbfgsMax || hist > cap || hist_acc > cap || !ws.lb_part || !ws.lb_coef || ws.lb_rows < 1)
        return cudaErrorInvalidValue;
    const cudaError_t e = launch_lbfgs_coefficients(n, hist, newest, cap, gamma, use_pair, hist_acc, newest_acc, ws, st);
    return e != cudaSuccess ? e : launch_lbfgs_pdir(n, ws, st);
}

cudaError_t launch_lbfgs_coefficients(int n, int hist, int newest, int cap, double gamma, bool use_pair,
                                      int hist_acc, int newest_acc, Workspace &ws, cudaStream_t st) {
    if (cap > kLbfgsMax || hist > cap || hist_acc > cap || !ws.lb_part || !ws.lb_coef || ws.lb_rows < 1)
        return cudaErrorInvalidValue;
    lbfgs_dots_kernel<<<lbfgs_blocks(n, kLbR, ws), kLbT, 0, st>>>(n, hist, newest, cap, gamma, use_pair ? 1 : 0,
                                                                  hist_acc, newest_acc, ws.S, ws.Y, ws.rho, ws.gram,
                                                                  ws.gf, ws.lb_part, ws.lb_coef, ws.sc);
    return cudaGetLastError();
}

cudaError_t launch_lbfgs_pdir(int n, Workspace &ws, cudaStream_t st) {
    if (!ws.lb_part || !ws.lb_coef || ws.lb_rows < 1) return cudaErrorInvalidValue;
    lbfgs_pdir_kernel<<<lbfgs_blocks(n, kLbP, ws), kLbP, 0, st>>>(n, ws.lb_coef, ws.S, ws.Y, ws.gf, ws.p,
                                                                  ws.lb_part, ws.sc);
    return cudaGetLastError();
}

cudaError_t launch_lbfgs_push(int n, int cap, int history, const PushState *state, bool dir, double *Wbest,
                              Workspace &ws, cudaStream_t st) {
    if (cap > kLbfgsMax || history >= cap || history < 1 || !state || !ws.lb_part || !ws.lb_coef || !ws.gram ||
        ws.lb_rows < 1)
        return cudaErrorInvalidValue;
    // a warp per pair and the new one; the pairs of one range over up to four SMs
    const int ranges = lbfgs_blocks(n, kLbR, ws), warps = std::max(2, std::min(kLbT / 32, history + 1));
    const int split = std::max(1, std::min({4, ws.lb_rows / ranges, (history + 2) / 2}));
    lbfgs_push_kernel<<<dim3(ranges, split), warps * 32, 0, st>>>(n, cap, state, ws.W, ws.Wt, ws.gf, ws.gft, ws.S, ws.Y,
                                                                  ws.rho, ws.gram, ws.lb_part, ws.sc, dir ? 1 : 0,
                                                                  ws.lb_coef, Wbest);
    return cudaGetLastError();
}

}  // namespace apd
