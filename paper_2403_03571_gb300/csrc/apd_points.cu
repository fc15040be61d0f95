// Algorithm 1 on a non-uniform discretisation (Section 2.3): sample points y_j
// (loaded, not generated) with element measures |P_j|, fused with the
// measure-weighted moments m_i = sum |P_j|, S1_i = sum |P_j| y_j,
// S2_i = sum |P_j| y_j y_j^T of each cell.
//
// Tiled form.  The points' box is cut into tiles (about 32 per seed, no more than one
// per two points), every tile gets its candidate list as the grid's tiles do
// (apd_region.cuh: the difference of two costs over the tile's box), stored as
// polynomials; a thread per point finds its tile, evaluates the few polynomials there
// and settles near ties in FP64 itself.  The points need no order.
//   points_box_kernel    the boxes and the tilings, on the device (high words of the
//                        coordinates: 20 bits are enough for a box): one tiling, or a fine
//                        one around the seeds and a coarse one of the whole box
//   points_lists_kernel  a block per 2 x 2 (x 2) tiles, eight warps listing, a warp
//                        per tile storing
//   points_score_kernel  labels and moments
// Bounds: the scoring kernel reads 32 (2D: 24) bytes a point from memory, a 16-byte
// header and about three 48-byte polynomials a point from L2, issues nine FP64
// products a point (16 clocks of an SM per warp each) and ten FP64 additions to the
// cell's words, which are what it waits for (in shared memory 275 us per 4 M points, as
// global reductions 610 us).  1000 seeds, 4 M random points in 3D: the call took
// 13.6 ms with the direct form below and takes 0.41 ms (box 26, preparation 21, lists
// 81, scoring 275 us).
//
// Direct form (few seeds or points, or more seeds than region lists take): the seeds
// stream through shared memory in chunks of
// 256 FP32 direct-form records (coordinates and weights split into FP32 high
// and low parts).  Pass 1 takes the smallest FP32 cost plus its rounding bound
// over all seeds as a threshold; pass 2 recomputes every seed whose FP32 cost
// minus its bound lies below it in FP64 with the reference operation order, and
// the smallest FP64 cost wins (lowest index on ties): the label equals the
// FP64 argmin over all seeds (the rescoring argument of the grid path).  Points whose
// tile's list did not fit its store, or that are not finite, take the same two passes a
// warp at a time.  The
// moments are FP64 sums accumulated with atomics (their rounding depends on
// the order of the additions).
#include <algorithm>

#include "apd_common.cuh"
#include "apd_cost.cuh"
#include "apd_region.cuh"

namespace apd {

namespace {

using namespace region;

constexpr int kPtThreads = 256;
constexpr int kMaxTiles = 1024;  // per axis
constexpr int kPtManyPoints = 320;  // points per SM from which block sums pay
constexpr size_t kPtShared = 200 * 1024;  // block sums of the moments

// One tile: 2 max E of its list, the reference seed (natural index; -1: no list, the
// points are searched in full), where its polynomials start and how many there are.
struct TileHead {
    float gap;
    int ref;
    unsigned first, count;
};

// The moment words of one point, and their addition to its cell.
template <int D>
__device__ __forceinline__ void point_words(double mj, const double (&yy)[D], double (&v)[moment_width(D)]) {
    v[0] = mj;
    int e = 1 + D;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        v[1 + a] = mj * yy[a];
#pragma unroll
        for (int b = a; b < D; ++b) v[e++] = v[1 + a] * yy[b];
    }
}
template <int D>
__device__ __forceinline__ void add_point(double *mom, int label, double mj, const double (&yy)[D]) {
    double v[moment_width(D)];
    point_words<D>(mj, yy, v);
    double *o = mom + (size_t)label * moment_width(D);
#pragma unroll
    for (int k = 0; k < moment_width(D); ++k) atomicAdd(&o[k], v[k]);
}

// High and low FP32 parts of a double by integer operations (the FP64 pipe converts a
// warp in 16 clocks of the SM): hi is v truncated to 24 bits, lo the rounded remainder,
// |v - hi - lo| <= 2^-47 |v|.  Values beyond FP32's normal range give 0 or infinity.
__device__ __forceinline__ void split_trunc(double v, float &hi, float &lo) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned h = (unsigned)(b >> 32), l = (unsigned)b;
    const int e = (int)((h >> 20) & 0x7ffu) - 1023 + 127;  // FP32 exponent
    const unsigned sign = h & 0x80000000u;
    if (e <= 30 || e >= 255) {
        hi = e >= 255 ? __uint_as_float(sign | 0x7f800000u) : 0.f;
        lo = 0.f;
        return;
    }
    hi = __uint_as_float(sign | ((unsigned)e << 23) | ((h & 0xfffffu) << 3) | (l >> 29));
    const float r = (float)(l & 0x1fffffffu);  // units of 2^(e - 127 - 52)
    const float scale = __uint_as_float((unsigned)(e - 29) << 23) * 0x1p-23f;
    lo = __uint_as_float(__float_as_uint(r * scale) | sign);
}

// About `want` tiles of near-cubic shape over the box lo .. lo + ext.
template <int D>
__device__ void make_tiling(const float (&lo)[3], const float (&box)[3], const long long want, PtsGeo *geo) {
    float ext[3] = {box[0], box[1], box[2]}, big = 1e-30f;
#pragma unroll
    for (int a = 0; a < D; ++a) big = fmaxf(big, ext[a]);
    float vol = 1.f;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        ext[a] = fmaxf(ext[a], 1e-4f * big);
        vol *= ext[a] / big;
    }
    float side = D == 3 ? cbrtf(vol / (float)want) : sqrtf(vol / (float)want);  // in units of big
    int t[3] = {1, 1, 1};
    for (int it = 0; it < 64; ++it) {  // shrink until the product fits
        long long n = 1;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            t[a] = max(1, min(kMaxTiles, (int)(ext[a] / big / side + 0.5f)));
            n *= t[a];
        }
        if (n <= want) break;
        side *= 1.03f;
    }
    long long n = 1;
    for (int a = 0; a < D; ++a) n *= t[a];
    if (n > want) t[0] = t[1] = t[2] = 1;
    geo->n_regions = 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const bool ax = a < D;
        const float h = ax ? __fmul_ru(__fdiv_ru(0.5f * ext[a], (float)t[a]), 1.f + 0x1p-20f) : 1.f;
        geo->gf.loh[a] = ax ? lo[a] : 0.f;
        geo->gf.lol[a] = 0.f;
        geo->gf.hh[a] = h;
        geo->gf.hl[a] = 0.f;
        geo->gf.ymax[a] = ax ? fmaxf(fabsf(lo[a]), fabsf(lo[a]) + ext[a]) * (1.f + 1e-6f) : 0.f;
        geo->t[a] = t[a];
        geo->regions[a] = (t[a] + 1) / 2;
        geo->n_regions *= geo->regions[a];
        geo->inv[a] = 0.5f / h;
        geo->r[a] = h * (1.f + 0x1p-9f);
        geo->ext[a] = ext[a];
    }
}

// The points' and the seeds' boxes from the high words of their coordinates, then (last
// block) the tilings.  geo[0] tiles the points' box with all `want` tiles, unless that box
// is more than four times the seeds' neighbourhood on an axis (an outlier among the points,
// or seeds in one place): uniform tiles would then be as large as many cells, their lists
// all seeds and their gaps beyond any difference.  geo[0] then tiles that neighbourhood (half
// the seeds' extent more on every side) with three quarters of the tiles and geo[1] the
// whole box with the rest.  MEASURED, us per call, one tiling / two (direct form): 1000
// seeds, 10^6 points in 3D, one of them at 1000 box lengths 60756 / 332 (3691), at 10
// 2199 / 333 (3689); 5000 seeds, 3000 points 14538 / 596 (969).
template <int D>
__global__ void __launch_bounds__(kPtThreads)
    points_box_kernel(const long long count, const double *__restrict__ y, const int n, const double *__restrict__ x,
                      const int point_blocks, const long long want, unsigned *__restrict__ part,
                      PtsGeo *__restrict__ geo) {
    __shared__ unsigned smn[D], smx[D];
    __shared__ bool last;
    if (threadIdx.x < D) {
        smn[threadIdx.x] = 0xffffffffu;
        smx[threadIdx.x] = 0u;
    }
    __syncthreads();
    unsigned mn[D], mx[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        mn[a] = 0xffffffffu;
        mx[a] = 0u;
    }
    // the blocks behind the points' take the seeds
    const bool seeds = (int)blockIdx.x >= point_blocks;
    const uint2 *v2 = reinterpret_cast<const uint2 *>(seeds ? x : y);
    const long long m = seeds ? n : count;
    const int blk = (int)blockIdx.x - (seeds ? point_blocks : 0), nblk = seeds ? (int)gridDim.x - point_blocks : point_blocks;
#pragma unroll 4
    for (long long j = (long long)blk * kPtThreads + threadIdx.x; j < m; j += (long long)nblk * kPtThreads)
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const unsigned h = v2[j * D + a].y;
            if ((h & 0x7ff00000u) == 0x7ff00000u) continue;  // not finite
            const unsigned k = h ^ ((h >> 31) ? 0xffffffffu : 0x80000000u);
            mn[a] = min(mn[a], k);
            mx[a] = max(mx[a], k);
        }
#pragma unroll
    for (int a = 0; a < D; ++a) {
        mn[a] = __reduce_min_sync(0xffffffffu, mn[a]);
        mx[a] = __reduce_max_sync(0xffffffffu, mx[a]);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&smn[a], mn[a]);
            atomicMax(&smx[a], mx[a]);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int a = 0; a < D; ++a) {
            part[(size_t)blockIdx.x * 6 + a] = smn[a];
            part[(size_t)blockIdx.x * 6 + 3 + a] = smx[a];
        }
        __threadfence();
        last = atomicAdd(&geo->done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    float lo[2][3] = {}, hi[2][3] = {};  // points, seeds
    bool some[2] = {true, true};
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int a = 0; a < D; ++a) {
            unsigned m = 0xffffffffu, v = 0u;
            for (int b = (q ? point_blocks : 0) + (int)threadIdx.x; b < (q ? (int)gridDim.x : point_blocks); b += 32) {
                m = min(m, __ldcg(&part[(size_t)b * 6 + a]));
                v = max(v, __ldcg(&part[(size_t)b * 6 + 3 + a]));
            }
            m = __reduce_min_sync(0xffffffffu, m);
            v = __reduce_max_sync(0xffffffffu, v);
            // outward: the dropped low words all zeros or all ones
            const unsigned hm = (m >> 31) ? m ^ 0x80000000u : ~m, hx = (v >> 31) ? v ^ 0x80000000u : ~v;
            const double dl = __longlong_as_double((long long)(((unsigned long long)hm << 32) | ((hm >> 31) ? 0xffffffffull : 0ull)));
            const double dh = __longlong_as_double((long long)(((unsigned long long)hx << 32) | ((hx >> 31) ? 0ull : 0xffffffffull)));
            const bool any = m <= v;
            some[q] = some[q] && any;
            lo[q][a] = any ? __double2float_rd(dl) : 0.f;
            hi[q][a] = any ? __double2float_ru(dh) : 1.f;
        }
    if (threadIdx.x != 0) return;
    float ext[3] = {0.f, 0.f, 0.f}, near_lo[3] = {0.f, 0.f, 0.f}, near_ext[3] = {0.f, 0.f, 0.f}, margin = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a) margin = fmaxf(margin, 0.5f * (hi[1][a] - lo[1][a]));
    bool wide = false, meet = some[0] && some[1];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        ext[a] = __fsub_ru(hi[0][a], lo[0][a]);
        near_lo[a] = fmaxf(lo[0][a], lo[1][a] - margin);
        near_ext[a] = __fsub_ru(fminf(hi[0][a], hi[1][a] + margin), near_lo[a]);
        wide = wide || ext[a] > 4.f * near_ext[a];
        meet = meet && near_ext[a] >= 0.f;
    }
    const bool two = wide && meet && want >= 8;
    if (two) {
        make_tiling<D>(near_lo, near_ext, want - want / 4, geo);
        make_tiling<D>(lo[0], ext, want / 4, geo + 1);
    } else {
        make_tiling<D>(lo[0], ext, want, geo);
        geo[1].n_regions = 0;
    }
    geo->pool = 0u;
    geo->done = 0u;
}

// Candidate lists of the tiles, stored.
template <int D>
__global__ void __launch_bounds__(kThreads, 4)
    points_lists_kernel(const __grid_constant__ Src src, PtsGeo *__restrict__ geo, TileHead *__restrict__ all_heads,
                        const int second, const int first_blocks, float4 *__restrict__ polys, const unsigned pool_cap) {
    using G = Geom<D>;
    constexpr int NP = G::NP;
    constexpr int PV = D == 3 ? 3 : 2;  // float4s of a polynomial
    __shared__ Shared<D> sm;
    __shared__ Src s;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned full = 0xffffffffu;
    const bool other = (int)blockIdx.x >= first_blocks;  // the blocks of the second tiling
    const PtsGeo *const ge = geo + (other ? 1 : 0);
    TileHead *const heads = all_heads + (other ? second : 0);
    const int nr = ge->n_regions;
    if (nr == 0) return;
    for (int i = tid; i < (int)(sizeof(Src) / 4); i += kThreads)
        reinterpret_cast<int *>(&s)[i] = reinterpret_cast<const int *>(&src)[i];
    const int stride = other ? (int)gridDim.x - first_blocks : first_blocks;
    __syncthreads();
    if (tid == 0) s.gf = ge->gf;
    __syncthreads();
    const float hh[3] = {s.gf.hh[0], s.gf.hh[1], s.gf.hh[2]};
    float tr[3], rr[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        tr[a] = a < D ? ge->r[a] : 0.f;
        rr[a] = a < D ? hh[a] + tr[a] : 0.f;
    }
    for (int reg = (int)blockIdx.x - (other ? first_blocks : 0); reg < nr; reg += stride) {
        const int q = reg / ge->regions[0];
        const int rb[3] = {reg % ge->regions[0], D == 3 ? q % ge->regions[1] : q, D == 3 ? q / ge->regions[1] : 0};
        float ch[3] = {0.f, 0.f, 0.f}, cl[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < D; ++a) axis_point(s.gf, a, 4 * rb[a] + 2, ch[a], cl[a]);
        float r0h, r0l;
        const unsigned total = region_list<D>(sm, s, ch, cl, rr, r0h, r0l);
        const int tc[3] = {wid & 1, (wid >> 1) & 1, wid >> 2};
        int ti[3];
        float toff[3] = {0.f, 0.f, 0.f};
        bool real = D == 3 || wid < 4;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            ti[a] = a < D ? 2 * rb[a] + tc[a] : 0;
            if (a < D) toff[a] = tc[a] ? hh[a] : -hh[a];
            real = real && ti[a] < ge->t[a];
        }
        if (real) {
            const bool scan = total > (unsigned)kListCap;
            const int n_src = scan ? s.n_groups : (int)((total + 31u) / 32u);
            auto source = [&](int c) -> int {
                const int e = c * 32 + lane;
                if (scan) return (sm.mask[c] >> lane) & 1u ? e : -1;
                return e < (int)total ? (int)sm.list[e] : -1;
            };
            unsigned best = 0xffffffffu;
            int best_pos = 0x7fffffff;
            Local<D> L;
            for (int c = 0; c < n_src; ++c) {
                const int p = source(c);
                unsigned ck = 0xffffffffu;
                if (p >= 0) {
                    local_terms<D>(s.recs[p], ch, cl, toff, tr, s.gf, L);
                    ck = min(okey(L.q - ((L.wh - r0h) + (L.wl - r0l))), 0xfffffffeu);
                }
                const unsigned cm = __reduce_min_sync(full, ck);
                const int who = (int)__reduce_min_sync(full, ck == cm && p >= 0 ? (unsigned)p : 0x7fffffffu);
                if (cm < best || (cm == best && who < best_pos)) {
                    best = cm;
                    best_pos = who;
                    if (p == who && p >= 0) store_local<D>(sm.ref[wid], L, s.perm ? s.perm[p] : p);
                }
            }
            __syncwarp();
            Local<D> R;
            int ref_id = 0;
            if (best != 0xffffffffu) load_local<D>(sm.ref[wid], R, ref_id);
            // counted first (the pool is taken in one piece), then stored
            auto test = [&](int c, Diff<D> &F) -> bool {
                const int p = source(c);
                if (p < 0 || p == best_pos) return false;
                local_terms<D>(s.recs[p], ch, cl, toff, tr, s.gf, L);
                difference<D>(L, R, F);
                return can_win<D>(F, tr);
            };
            unsigned keep_bits = 0u;  // of the first 32 chunks
            unsigned count = 0u;
            float Emax = 0.f;
            for (int c = 0; c < n_src; ++c) {
                Diff<D> F;
                const bool keep = test(c, F);
                if (keep) Emax = fmaxf(Emax, F.E);
                if (keep && c < 32) keep_bits |= 1u << c;
                count += (unsigned)__popc(__ballot_sync(full, keep));
            }
            Emax = __uint_as_float(__reduce_max_sync(full, __float_as_uint(Emax)));
            unsigned first = 0u;
            if (lane == 0 && count) first = atomicAdd(&geo->pool, count);
            first = __shfl_sync(full, first, 0);
            const bool fits = best != 0xffffffffu && first <= pool_cap && count <= pool_cap - first;
            if (lane == 0) {
                TileHead h;
                h.gap = 2.f * Emax;
                h.ref = fits ? ref_id : -1;
                h.first = first;
                h.count = count;
                heads[(size_t)ti[0] + (size_t)ge->t[0] * ((size_t)ti[1] + (size_t)ge->t[1] * (size_t)ti[2])] = h;
            }
            if (fits && count) {
                unsigned at = first;
                for (int c = 0; c < n_src; ++c) {
                    const bool maybe = c >= 32 || ((keep_bits >> c) & 1u);
                    if (!__any_sync(full, maybe)) continue;
                    Diff<D> F;
                    const bool keep = maybe && test(c, F);
                    const unsigned km = __ballot_sync(full, keep);
                    if (keep) {
                        const int p = source(c);
                        const int id = s.perm ? s.perm[p] : p;
                        float4 *o = polys + (size_t)(at + (unsigned)__popc(km & ((1u << lane) - 1u))) * PV;
                        o[0] = make_float4(F.d0, F.g[0], F.g[1], D == 3 ? F.g[D - 1] : __int_as_float(id));
                        if (D == 3) {
                            o[1] = make_float4(F.a[0], 2.f * F.a[1], 2.f * F.a[2], F.a[NP - 3]);
                            o[2] = make_float4(2.f * F.a[NP - 2], F.a[NP - 1], __int_as_float(id), 0.f);
                        } else {
                            o[1] = make_float4(F.a[0], 2.f * F.a[1], F.a[2], 0.f);
                        }
                    }
                    at += (unsigned)__popc(km);
                }
            }
        }
        __syncthreads();  // the list is read until here
    }
}

// Labels and moments from the tiles' lists.  SHARED: the block sums its moments in
// shared memory (n K doubles) and adds them to the global ones at the end; a warp whose
// points lie in one cell sums them first.
template <int D, bool SHARED, int T>
__global__ void __launch_bounds__(T)
    points_score_kernel(const long long count, const double *__restrict__ y, const double *__restrict__ mass,
                        const int n, const double *__restrict__ x, const double *__restrict__ A,
                        const double *__restrict__ w, const SeedRec32 *__restrict__ r32, const PtsGeo *__restrict__ geo,
                        const TileHead *__restrict__ heads, const int second, const float4 *__restrict__ polys,
                        DevScalars *__restrict__ sc, double *__restrict__ mom, int32_t *__restrict__ labels) {
    constexpr int PV = D == 3 ? 3 : 2;
    constexpr int K = moment_width(D);
    __shared__ PtsGeo tilings[2];
    extern __shared__ double acc[];
    for (int i = threadIdx.x; i < (int)(2 * sizeof(PtsGeo) / 4); i += T)
        reinterpret_cast<int *>(tilings)[i] = reinterpret_cast<const int *>(geo)[i];
    if (SHARED)
        for (int i = threadIdx.x; i < n * K; i += T) acc[i] = 0.0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const float finf = __int_as_float(0x7f800000);
    for (long long j0 = (long long)blockIdx.x * T; j0 < count; j0 += (long long)gridDim.x * T) {
        const long long j = j0 + threadIdx.x;
        const bool active = j < count;
        double yy[D];
        float yh[3] = {0.f, 0.f, 0.f}, yl[3] = {0.f, 0.f, 0.f}, e[3] = {0.f, 0.f, 0.f};
        size_t tile = 0;
#pragma unroll
        for (int a = D - 1; a >= 0; --a) {
            yy[a] = active ? y[j * D + a] : 0.0;
            split_trunc(yy[a], yh[a], yl[a]);
        }
        auto locate = [&](const PtsGeo &ge) -> bool {  // the point's tile and its offset from the centre
            bool in = active;
            tile = 0;
#pragma unroll
            for (int a = D - 1; a >= 0; --a) {
                const float d = (yh[a] - ge.gf.loh[a]) + yl[a];
                const int t = min(max((int)(d * ge.inv[a]), 0), ge.t[a] - 1);
                float ch, cl;
                axis_point(ge.gf, a, 2 * t + 1, ch, cl);
                e[a] = (yh[a] - ch) + (yl[a] - cl);
                in = in && fabsf(e[a]) <= ge.r[a];  // false for a NaN
                tile = tile * (size_t)ge.t[a] + (size_t)t;
            }
            return in;
        };
        bool inside = locate(tilings[0]);
        if (!inside && tilings[1].n_regions) {
            inside = locate(tilings[1]);
            tile += (size_t)second;
        }
        const double mj = active ? mass[j] : 0.0;
        TileHead h{0.f, -1, 0u, 0u};
        if (inside) h = heads[tile];
        const bool listed = h.ref >= 0;
        auto value = [&](unsigned k, int &id) -> float {
            const float4 *o = polys + (size_t)(h.first + k) * PV;
            const float4 v0 = o[0], v1 = o[1];
            if (D == 3) {
                const float4 v2 = o[2];
                id = __float_as_int(v2.z);
                const float b = fmaf(v1.z, e[2], fmaf(v1.y, e[1], v0.y));
                const float t1 = fmaf(v2.x, e[2], fmaf(v1.w, e[1], v0.z));
                const float t2 = fmaf(v2.y, e[2], v0.w);
                return fmaf(fmaf(v1.x, e[0], b), e[0], fmaf(e[2], t2, fmaf(e[1], t1, v0.x)));
            }
            id = __float_as_int(v0.w);
            return fmaf(fmaf(v1.x, e[0], fmaf(v1.y, e[1], v0.y)), e[0], fmaf(e[1], fmaf(v1.z, e[1], v0.z), v0.x));
        };
        int bi = h.ref;
        if (listed) {
            float v1 = 0.f, v2 = finf;
            for (unsigned k = 0; k < h.count; ++k) {
                int id;
                const float v = value(k, id);
                v2 = fminf(v2, fmaxf(v1, v));
                bi = v < v1 ? id : bi;
                v1 = fminf(v1, v);
            }
            const float thr = v1 + h.gap;
            if (!(v2 > thr)) {  // near tie: FP64 among the seeds within the gap
                double best = __longlong_as_double(0x7ff0000000000000ll);
                bi = 0x7fffffff;
                for (int k = -1; k < (int)h.count; ++k) {
                    int id = h.ref;
                    const float v = k < 0 ? 0.f : value((unsigned)k, id);
                    if (v > thr) continue;
                    const double c = cost64<D>(yy, x + (size_t)id * D, A + (size_t)id * D * D, w[id]);
                    if (c < best || (c == best && id < bi)) {
                        best = c;
                        bi = id;
                    }
                }
            }
        }
        // points without a list, a warp per point: both passes over every seed
        unsigned todo = __ballot_sync(full, active && !listed);
        while (todo) {
            const int p = __ffs(todo) - 1;
            todo &= todo - 1u;
            double py[D];
            float ph[3] = {0.f, 0.f, 0.f}, pl[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int a = 0; a < D; ++a) {
                py[a] = __shfl_sync(full, yy[a], p);
                split_f32(py[a], ph[a], pl[a]);
            }
            const float wrh = sc->wref_h, wrl = sc->wref_l;
            float thr = finf;
            for (int s = lane; s < n; s += 32) {
                float c, E;
                cost32_bound<D>(r32[s], ph, pl, wrh, wrl, c, E);
                thr = fminf(thr, c + E);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) thr = fminf(thr, __shfl_xor_sync(full, thr, off));
            double best = __longlong_as_double(0x7ff0000000000000ll);
            int ib = 0x7fffffff;
            for (int s = lane; s < n; s += 32) {
                float c, E;
                cost32_bound<D>(r32[s], ph, pl, wrh, wrl, c, E);
                if (!(c - E <= thr)) continue;
                const double c64 = cost64<D>(py, x + (size_t)s * D, A + (size_t)s * D * D, w[s]);
                if (c64 < best) {
                    best = c64;
                    ib = s;
                }
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const double ob = __shfl_xor_sync(full, best, off);
                const int oi = __shfl_xor_sync(full, ib, off);
                if (ob < best || (ob == best && oi < ib)) {
                    best = ob;
                    ib = oi;
                }
            }
            if (lane == p) bi = ib;
        }
        const bool good = active && bi >= 0 && bi < n;
        if (active && !good) atomicOr(&sc->status, ST_BAD_LABEL);
        if (good && labels) labels[j] = bi;
        if (SHARED) {
            const int b0 = __shfl_sync(full, bi, 0);
            if (__all_sync(full, good && bi == b0)) {  // points in spatial order: one cell
                double v[K];
                point_words<D>(mj, yy, v);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const double t = warp_sum(v[k]);
                    if (lane == 0) atomicAdd(&acc[(size_t)b0 * K + k], t);
                }
                continue;
            }
        }
        if (good) add_point<D>(SHARED ? acc : mom, bi, mj, yy);
    }
    if (SHARED) {
        __syncthreads();
        for (int i = threadIdx.x; i < n * K; i += T)
            if (acc[i] != 0.0) atomicAdd(&mom[i], acc[i]);
    }
}

template <int D>
__global__ void __launch_bounds__(kPtThreads)
    points_assign_kernel(const long long count, const double *__restrict__ y, const double *__restrict__ mass,
                         const int n, const double *__restrict__ x, const double *__restrict__ A,
                         const double *__restrict__ w, const SeedRec32 *__restrict__ r32,
                         DevScalars *__restrict__ sc, double *__restrict__ mom, int32_t *__restrict__ labels) {
    constexpr int K = moment_width(D);
    __shared__ SeedRec32 sr[kPtThreads];
    const double wref = dkey_inv(sc->wref_key);
    float wrh, wrl;
    split_f32(wref, wrh, wrl);
    for (long long j0 = (long long)blockIdx.x * kPtThreads; j0 < count; j0 += (long long)gridDim.x * kPtThreads) {
        const long long j = j0 + threadIdx.x;
        const bool active = j < count;
        double yy[D];
        float yh[3] = {0.f, 0.f, 0.f}, yl[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < D; ++a) {
            yy[a] = active ? y[j * D + a] : 0.0;
            split_f32(yy[a], yh[a], yl[a]);
        }
        // pass 1: threshold = min_k (C_k + E_k)
        float thr = __int_as_float(0x7f800000);
        for (int c0 = 0; c0 < n; c0 += kPtThreads) {
            const int m = min(kPtThreads, n - c0);
            __syncthreads();
            if ((int)threadIdx.x < m) sr[threadIdx.x] = r32[c0 + threadIdx.x];
            __syncthreads();
            for (int k = 0; k < m; ++k) {
                float c, E;
                cost32_bound<D>(sr[k], yh, yl, wrh, wrl, c, E);
                thr = fminf(thr, c + E);
            }
        }
        // pass 2: FP64 reference cost of the candidates
        double best = __longlong_as_double(0x7ff0000000000000ll);
        int bi = 0x7fffffff;
        for (int c0 = 0; c0 < n; c0 += kPtThreads) {
            const int m = min(kPtThreads, n - c0);
            __syncthreads();
            if ((int)threadIdx.x < m) sr[threadIdx.x] = r32[c0 + threadIdx.x];
            __syncthreads();
            if (!active) continue;
            for (int k = 0; k < m; ++k) {
                float c, E;
                cost32_bound<D>(sr[k], yh, yl, wrh, wrl, c, E);
                if (!(c - E <= thr)) continue;
                const int s = c0 + k;
                const double c64 = cost64<D>(yy, x + (size_t)s * D, A + (size_t)s * D * D, w[s]);
                if (c64 < best || (c64 == best && s < bi)) {
                    best = c64;
                    bi = s;
                }
            }
        }
        if (!active) continue;
        if (bi < 0 || bi >= n) {
            atomicOr(&sc->status, ST_BAD_LABEL);
            continue;
        }
        if (labels) labels[j] = bi;
        add_point<D>(mom, bi, mass[j], yy);
    }
}

template <int D>
cudaError_t launch_t(long long count, const double *y, const double *mass, int n, const double *x, const double *A,
                     const double *w, double *mom, int32_t *labels, Workspace &ws, cudaStream_t st) {
    const long long n_mom = (long long)n * moment_width(D);
    unsigned long long *m64 = reinterpret_cast<unsigned long long *>(mom);
    GridDev none{};
    none.dim = D;
    none.res[0] = none.res[1] = none.res[2] = 1;
    none.h32[0] = none.h32[1] = none.h32[2] = 1.f;
    const bool tiled = points_tiled(count, n, ws);
    const long long want_blocks = (count + kPtThreads - 1) / kPtThreads;
    if (tiled) {
        const int blocks = (int)std::min<long long>(want_blocks, (long long)ws.sms * 8);
        // about 32 tiles a seed, no more than one per two points or the store holds
        const long long cap = (long long)(ws.pts_bytes / (sizeof(TileHead) + 8 * 48));
        const long long tiles = std::max<long long>(1, std::min<long long>(std::min<long long>(32ll * n, count / 2), cap));
        const int second = (int)(tiles - tiles / 4);  // first tile of the second tiling
        const int sblocks = std::min((n + kPtThreads - 1) / kPtThreads, 64);
        // the blocks' boxes (24 bytes each) go where the tiles' headers follow
        points_box_kernel<D><<<blocks + sblocks, kPtThreads, 0, st>>>(
            count, y, n, x, blocks, tiles, reinterpret_cast<unsigned *>(ws.pts_tiles), ws.pts_geo);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        e = launch_seed_prep(none, n, x, A, w, ws, m64, n_mom, st, ws.pts_geo);
        if (e != cudaSuccess) return e;
        e = launch_group_bounds(n, ws, st);
        if (e != cudaSuccess) return e;
        Src src{};
        src.n = n;
        src.n_groups = (n + kGroup - 1) / kGroup;
        src.recs = ws.sorted ? ws.recs32s : ws.recs32;
        src.perm = ws.sorted ? ws.perm : nullptr;
        src.groups = ws.groups;
        src.sc = ws.sc;
        TileHead *heads = reinterpret_cast<TileHead *>(ws.pts_tiles);
        float4 *polys = reinterpret_cast<float4 *>(ws.pts_tiles + ((size_t)tiles * sizeof(TileHead) + 255) / 256 * 256);
        const size_t rest = ws.pts_bytes - ((size_t)tiles * sizeof(TileHead) + 255) / 256 * 256;
        const unsigned pool = (unsigned)std::min<size_t>(rest / ((D == 3 ? 3 : 2) * sizeof(float4)), 0x7fffffffu);
        const int lb = (int)std::min<long long>(4ll * ws.sms, tiles);
        const int lb2 = (int)std::min<long long>(ws.sms, std::max<long long>(1, tiles / 32));  // most calls need none
        points_lists_kernel<D><<<lb + lb2, kThreads, 0, st>>>(src, ws.pts_geo, heads, second, lb, polys, pool);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        // Block sums where n K doubles fit (one block of 1024 per SM) and a block gets
        // several points per word it then adds to the global moments: those additions, by
        // every block to the same n K words, cost 60 to 110 us whatever the count.
        // MEASURED, us shared / global sums, 3D: n = 24, 20000 points 106 / 83, 80000 110 / 207;
        // n = 80, 40000 81 / 82; n = 1000, 4 M (scoring alone) 275 / 610.
        const size_t smem = (size_t)n_mom * sizeof(double);
        if (smem <= kPtShared && count >= (long long)std::max(kPtManyPoints, 4 * n) * ws.sms) {
            constexpr int T = 1024;
            constexpr unsigned bit = D == 3 ? kAttrPoints3 : kAttrPoints2;
            if (!(ws.attr_done & bit)) {
                e = cudaFuncSetAttribute(points_score_kernel<D, true, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kPtShared);
                if (e != cudaSuccess) return e;
                ws.attr_done |= bit;
            }
            const int per_sm = smem <= kPtShared / 2 ? 2 : 1;
            points_score_kernel<D, true, T><<<per_sm * ws.sms, T, smem, st>>>(
                count, y, mass, n, x, A, w, ws.recs32, ws.pts_geo, heads, second, polys, ws.sc, mom, labels);
        } else {
            const int sb = (int)std::min<long long>(want_blocks, (long long)ws.sms * 8);
            points_score_kernel<D, false, kPtThreads><<<sb, kPtThreads, 0, st>>>(
                count, y, mass, n, x, A, w, ws.recs32, ws.pts_geo, heads, second, polys, ws.sc, mom, labels);
        }
        return cudaGetLastError();
    }
    // the seeds in their own order: no ranking (4 us of a 25 us call)
    uint32_t *const codes = ws.codes;
    ws.codes = nullptr;
    cudaError_t e = launch_seed_prep(none, n, x, A, w, ws, m64, n_mom, st);
    ws.codes = codes;
    if (e != cudaSuccess) return e;
    const int blocks = (int)std::min<long long>(want_blocks, (long long)ws.sms * 8);
    points_assign_kernel<D><<<blocks, kPtThreads, 0, st>>>(count, y, mass, n, x, A, w, ws.recs32, ws.sc, mom, labels);
    return cudaGetLastError();
}

}  // namespace

// The tiled form's six launches and lists against two passes over all seeds a point.
// MEASURED, us direct / tiled: 2D n = 20, 20000 points 56 / 60, n = 30 66 / 64, n = 45 62 / 56,
// n = 3000, 5000 points 438 / 57; 3D n = 8, 3000 points 50 / 54, n = 16, 5000 62 / 55 (direct
// with the ranking it no longer makes); few seeds gain where the block sums do (n = 8,
// 100000 points: 2D 338 / 167, 3D 492 / 173).
bool points_tiled(long long count, int n, const Workspace &ws) {
    if (!ws.groups || !ws.pts_tiles || (n + kGroup - 1) / kGroup > kMaxGroups || count < 256) return false;
    return n >= (ws.dim == 2 ? 40 : 12) || (n >= 8 && count >= (long long)kPtManyPoints * ws.sms);
}

cudaError_t launch_points_assign(int dim, long long count, const double *y, const double *mass, int n,
                                 const double *x, const double *A, const double *w, double *mom,
                                 int32_t *labels, Workspace &ws, cudaStream_t st) {
    return dim == 3 ? launch_t<3>(count, y, mass, n, x, A, w, mom, labels, ws, st)
                    : launch_t<2>(count, y, mass, n, x, A, w, mom, labels, ws, st);
}

}  // namespace apd
