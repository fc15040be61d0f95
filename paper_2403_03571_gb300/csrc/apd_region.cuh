// Algorithm 1 over one region of a regular grid from candidate lists, fused with
// the per-cell integer moments: the pruned scorer of the one-instance calls and of
// the batches.
//
// Lists.  Inside a box of half-widths r around c the difference of two costs of
// eq. (2.1) is a quadratic whose linear part dominates: with d = c - x, y = c + e,
//     C_i - C_a = D0 + G.e + e^T (A_i - A_a) e,
//     D0 = (q_i - w_i) - (q_a - w_a),  q = d^T A d,  G = 2 (A_i d_i - A_a d_a).
// Seed i is nowhere the argmin in the box when the lower bound
//     D0 - sum |G_b| r_b - 2 sum_{b<c} |dA_bc| r_b r_c + sum_b min(dA_bb, 0) r_b^2 - E
// is positive (E: the FP32 rounding, below).  Separate bounds of C_i and C_a differ
// by the variation of the cost over the box, several cell widths times the box's;
// here only what differs between the two seeds counts, so the lists hold hardly
// more than the cells that meet the box (3.2 of 1000 seeds per 8^3 tile at 256^3,
// against 33 with separate bounds).
//   * Region (16^3 voxels / 64^2 pixels, one block): the 32-seed groups' cost lower
//     bounds, one group per lane; the seed a of least cost at the centre among the
//     warps' nearest groups; the seeds of the groups that can beat a's largest cost
//     are tested against a and listed in shared memory (past 1024: as a bit per seed).
//   * Tile (8^3 / 32 x 16, one warp): the same test over the tile against the listed
//     seed of least cost at the tile's centre.  Up to 48 polynomials stay in shared
//     memory; of a longer list the positions stay, and its polynomials are formed again
//     32 at a time (see tile_cap).
// Measured (1000 seeds, 256^3, solve-sized weights): 99 us, 61.0 M warp
// instructions (region lists 33 %, tile lists 23 %, pixels 27 %, moments 17 %) at half
// of the issue slots; the tensor-core scorer with separate bounds took 456 us after a
// 92 us list pre-pass, and 14 us of rescoring followed.  10^4 seeds, 200^3, axis
// ratios up to 3.3 (the alpha = 0.7 law): 6.2 ms -> 0.79 ms, since the bound E is local
// (the FP32 kernel's grows with the largest condition number of all seeds).
// Scoring.  What is left is a handful of polynomials D_i(e) per tile (a itself is 0
// everywhere): a lane owns two rows of eight pixels, the two row coefficients cost
// nine operations and each pixel two packed FMAs and five selections per listed
// seed.  No contraction is left for the tensor cores: a 32-seed MMA step would be
// nine tenths padding.  Bound: issue (the pixel loop and the moments take about two
// thirds of a block's instructions, the lists one third); memory traffic is the
// labels alone.
// Moments.  Per tile and label the lanes' row masks become sums of local
// coordinates by a 256-entry table, two sums to a word, reduced over the warp in 5
// (2D: 3) integer reductions and shifted to the grid's coordinates in 64 bits; a
// tile or region of one cell adds its sums in closed form.
//
// Rounding.  With u = 2^-24, p_b = |d_b| + r_b + 2^-24 (|x_b| + |y|_max,b) and
// S = sum_bc |A_bc| p_b p_c: a difference d is two FP32 subtractions of pairs (one
// rounding of c - x, one of the sum) and the tile's offset o (two roundings) added, so it
// errs by at most 3 u |d| + 4 u |o|, and a pixel's own offset by 2 u r.  |o| <= 8/7 r in
// 3D, 3.2 r on the second axis in 2D (tiles 24 h from the centre, r = 7.5 h): 6.6 u p and
// 14.8 u p.  The cost of one seed then errs by at most 21 u S in 3D (A's own rounding 1,
// the differences 2 x 6.6, the dot products 6), 35 u S in 2D (1, 2 x 14.8, 4); forming D0,
// G and dA adds 3 u (S_i + S_a + |dw| + ...), the row coefficients and the two FMAs 9 u,
// in 2D 5 u, of the same: 33 u (3D) and 43 u (2D) in all, and the list test's sums no more
// than the pixels'.  kCoef = 64 is used for both the list test and the certificate.  A
// pixel is labelled when its two smallest values are more than 2 max_i E_i apart,
// E_i = 64 u (S_i + S_a + W), W = |dw| + 2^-24 (|w_i| + |w_a|); every other pixel is settled
// by its warp in FP64 with the reference arithmetic over the seeds within the gap, a
// lane per pixel: no rescoring launch follows.
#pragma once

#include <float.h>

#include "apd_cost.cuh"
#include "apd_internal.cuh"

namespace apd {
namespace region {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kListCap = 1024;  // listed seeds of a region; beyond it the tiles take the groups that hold any
constexpr int kBuf = 48;        // polynomials a warp keeps at a time
constexpr int kFast = 8;        // polynomials of a tile whose labels fit the byte masks
constexpr int kTilePix = 512;
constexpr float kCoef = 64.f * 5.9604644775390625e-8f;
constexpr float kEta = 5.9604644775390625e-8f;
constexpr int kMaxGroups = kSortMax / kGroup;  // 512: two groups per lane and warp

// Seeds of a tile's list kept by their scan position, in dynamic shared memory (16 bytes a
// seed for a block): what does not fit the polynomials' buffer is formed again from there,
// a list beyond it from the region's.  512 leave the caches their room; where the regions
// are fewer than the SMs hold, or cells are so small that lists are long, a block gets more.
// MEASURED, us per call, lists formed again from the region's only / from the tile's: 3D
// n = 10000 on 96^3 1326 / 347, n = 3000 on 60^3 441 / 223; 2D n = 5000 on 300^2 601 / 245.
constexpr int kTileCap = 512, kTileCapMax = 12032;
inline int tile_cap(long long regions, long long pixels, int n, int sms) {
    const int cap = regions <= sms ? kTileCapMax
                    : regions <= 2ll * sms ? 4864
                    : regions <= 3ll * sms || pixels < 128ll * n ? 2560 : kTileCap;
    const int all = (n + 31) / 32 * 32;
    return all < cap ? all : cap;
}
inline size_t tile_bytes(int cap) { return (size_t)kWarps * cap * sizeof(uint16_t); }
inline int blocks_per_sm(int cap) { return cap <= 1472 ? 4 : cap <= 2560 ? 3 : cap <= 4864 ? 2 : 1; }

template <int D>
struct Geom;
template <>
struct Geom<3> {
    static constexpr int RX = 16, RY = 16, RZ = 16;  // region
    static constexpr int TX = 8, TY = 8, TZ = 8;     // tile
    static constexpr int NP = 6;                     // entries of a symmetric matrix
};
template <>
struct Geom<2> {
    static constexpr int RX = 64, RY = 64, RZ = 1;
    static constexpr int TX = 32, TY = 16, TZ = 1;
    static constexpr int NP = 3;
};

// One scoring problem.
struct Src {
    GridDev g;
    GridF gf;
    int n, n_groups;
    int tile_cap;              // seeds a tile keeps by position
    const SeedRec32 *recs;     // scan order
    const int32_t *perm;       // scan position -> seed index (null: identity)
    const GroupBound *groups;  // bounds of the scan-order groups
    const double *x, *A, *w;   // the FP64 seeds (natural order)
    unsigned long long *gmom;  // [n][K]
    int32_t *labels;           // [J] or null
    DevScalars *sc;
    unsigned long long *pairs_scored;
    // MASKED: only the pixels of marked coarse pixels (r pixels per axis each)
    const uint8_t *mask;       // [product of cres]
    int r, cres[3];
};

// A seed's cost around a point: q = d^T A d, h = A d, S (see Rounding).
template <int D>
struct Local {
    float q, S, wh, wl;
    float h[D];
    float a[Geom<D>::NP];
};

template <int D>
struct Shared {
    float4 poly[kWarps][kBuf][3];
    float4 ref[kWarps][5];             // the warp's best seed (region), then its tile's reference
    uint16_t list[kListCap];           // scan positions
    unsigned mask[kMaxGroups];         // a group's listed seeds (where there are more than kListCap)
    uint16_t queue[kWarps][kTilePix];  // the tile's near ties: pixel of the tile
    unsigned lut[256];  // row mask -> count | sum x << 8 | sum x^2 << 16
    unsigned key[kWarps];
    unsigned count;     // listed seeds
    unsigned pairs;
    unsigned queued;    // pixels settled in FP64
};

__device__ __forceinline__ unsigned okey(float v) {  // order-preserving float -> unsigned
    const unsigned u = __float_as_uint(v);
    return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}

// Index of the upper-triangle entry (a, b), a <= b, in row order.
template <int D>
__host__ __device__ constexpr int tri(int a, int b) {
    return D == 3 ? (a == 0 ? b : (a == 1 ? 2 + b : 5)) : (a == 0 ? b : 2);
}

// lo + k h as an FP32 pair, |error| <= 2^-46 max(|lo|, |hi|) (k an integer below 2^24).
__device__ __forceinline__ void axis_point(const GridF &gf, int a, int k, float &ch, float &cl) {
    const float K = (float)k;
    const float p = __fmul_rn(K, gf.hh[a]);
    const float e = fmaf(K, gf.hl[a], fmaf(K, gf.hh[a], -p));
    const float s = __fadd_rn(gf.loh[a], p);
    const float bb = __fsub_rn(s, gf.loh[a]);
    float t = __fadd_rn(__fsub_rn(gf.loh[a], __fsub_rn(s, bb)), __fsub_rn(p, bb));
    t = __fadd_rn(t, __fadd_rn(gf.lol[a], e));
    ch = __fadd_rn(s, t);
    cl = __fsub_rn(t, __fsub_rn(ch, s));
}

template <int D>
__device__ __forceinline__ void local_terms(const SeedRec32 &r, const float (&ch)[3], const float (&cl)[3],
                                            const float (&off)[3], const float (&rr)[3], const GridF &gf,
                                            Local<D> &L) {
    float d[D], p[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        d[a] = ((ch[a] - r.xh[a]) + (cl[a] - r.xl[a])) + off[a];
        p[a] = fabsf(d[a]) + rr[a] + kEta * (fabsf(r.xh[a]) + gf.ymax[a]);
    }
    float q = 0.f, S = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        float t = 0.f, s = 0.f;
#pragma unroll
        for (int b = 0; b < D; ++b) {
            const float m = r.a[tri<D>(a < b ? a : b, a < b ? b : a)];
            t = fmaf(m, d[b], t);
            s = fmaf(fabsf(m), p[b], s);
        }
        L.h[a] = t;
        q = fmaf(d[a], t, q);
        S = fmaf(p[a], s, S);
    }
    L.q = q;
    L.S = S;
    L.wh = r.wh;
    L.wl = r.wl;
#pragma unroll
    for (int e = 0; e < Geom<D>::NP; ++e) L.a[e] = r.a[e];
}

// The polynomial C_i - C_a: value, gradient and (packed) matrix at the point, and E.
template <int D>
struct Diff {
    float d0, E;
    float g[D];
    float a[Geom<D>::NP];
};
template <int D>
__device__ __forceinline__ void difference(const Local<D> &L, const Local<D> &R, Diff<D> &F) {
    const float dw = (L.wh - R.wh) + (L.wl - R.wl);
    F.d0 = (L.q - R.q) - dw;
#pragma unroll
    for (int a = 0; a < D; ++a) F.g[a] = 2.f * (L.h[a] - R.h[a]);
#pragma unroll
    for (int e = 0; e < Geom<D>::NP; ++e) F.a[e] = L.a[e] - R.a[e];
    F.E = kCoef * (L.S + R.S + fabsf(dw) + kEta * (fabsf(L.wh) + fabsf(R.wh))) + 1e-37f;
}
// Whether seed i can cost as little as a somewhere in the box of half-widths rr.
template <int D>
__device__ __forceinline__ bool can_win(const Diff<D> &F, const float (&rr)[3]) {
    float lo = F.d0 - F.E;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        lo -= fabsf(F.g[a]) * rr[a];
        lo += fminf(F.a[tri<D>(a, a)], 0.f) * (rr[a] * rr[a]);
#pragma unroll
        for (int b = a + 1; b < D; ++b) lo -= 2.f * fabsf(F.a[tri<D>(a, b)]) * (rr[a] * rr[b]);
    }
    return !(lo > 0.f);  // a NaN keeps the seed
}

template <int D>
__device__ __forceinline__ void store_local(float4 (&s)[5], const Local<D> &L, int id) {
    if (D == 3) {
        s[0] = make_float4(L.q, L.S, L.wh, L.wl);
        s[1] = make_float4(L.h[0], L.h[1], L.h[D - 1], __int_as_float(id));
        s[2] = make_float4(L.a[0], L.a[1], L.a[2], L.a[Geom<D>::NP - 3]);
        s[3] = make_float4(L.a[Geom<D>::NP - 2], L.a[Geom<D>::NP - 1], 0.f, 0.f);
    } else {
        s[0] = make_float4(L.q, L.S, L.wh, L.wl);
        s[1] = make_float4(L.h[0], L.h[1], 0.f, __int_as_float(id));
        s[2] = make_float4(L.a[0], L.a[1], L.a[2], 0.f);
    }
}
template <int D>
__device__ __forceinline__ void load_local(const float4 (&s)[5], Local<D> &L, int &id) {
    const float4 v0 = s[0], v1 = s[1], v2 = s[2];
    L.q = v0.x;
    L.S = v0.y;
    L.wh = v0.z;
    L.wl = v0.w;
    L.h[0] = v1.x;
    L.h[1] = v1.y;
    id = __float_as_int(v1.w);
    L.a[0] = v2.x;
    L.a[1] = v2.y;
    L.a[2] = v2.z;
    if (D == 3) {
        const float4 v3 = s[3];
        L.h[D - 1] = v1.z;
        L.a[Geom<D>::NP - 3] = v2.w;
        L.a[Geom<D>::NP - 2] = v3.x;
        L.a[Geom<D>::NP - 1] = v3.y;
    }
}

__device__ __forceinline__ unsigned long long f2_bits(float2 v) {
    return (unsigned long long)__float_as_uint(v.x) | ((unsigned long long)__float_as_uint(v.y) << 32);
}
// packed FP32x2 fused multiply-add
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
    return make_float2(__uint_as_float((unsigned)(r & 0xffffffffu)), __uint_as_float((unsigned)(r >> 32)));
}

// Moment words of one cell's pixels in a box from sums of local coordinates x = k - kb:
// u = 2 k + 1 = 2 x + o, o = 2 kb + 1, so with n the count
//     sum u_a = 2 X_a + o_a n,   sum u_a u_b = 4 X_ab + 2 o_b X_a + 2 o_a X_b + o_a o_b n.
// Lane v < K forms word v: X_ab (or X_a, or n) times c, plus m1 X_a + m2 X_b + m3 n.
struct WordMap {
    unsigned c, fv, fa, fb;  // multiplier and the fields of X_v, X_a, X_b (word * 2 + half)
    int a, b;                // axes (a < 0: the count; b < 0: a linear word)
};
// Where the packed reductions keep word v of apd_cell_moments: half (v & 1) of word v / 2
// after this order: 3D (n, x), (y, z), (xx, yy), (zz, xy), (xz, yz); 2D (xx, n), (x, y),
// (xy, yy), the first with n in bits 20-31.
template <int D>
__device__ __forceinline__ unsigned field_of(int v) {
    if (D == 3) {
        const unsigned long long t = 0x0ull | (1ull << 4) | (2ull << 8) | (3ull << 12) | (4ull << 16) | (7ull << 20) |
                                     (8ull << 24) | (5ull << 28) | (9ull << 32) | (6ull << 36);
        return (unsigned)(t >> (4 * v)) & 15u;
    }
    const unsigned t = 1u | (2u << 4) | (3u << 8) | (0u << 12) | (4u << 16) | (5u << 20);
    return (t >> (4 * v)) & 15u;
}
template <int D>
__device__ __forceinline__ WordMap word_map() {
    constexpr int K = moment_width(D);
    const int v = min((int)(threadIdx.x & 31), K - 1);
    WordMap m;
    m.a = m.b = -1;
    if (v >= 1 && v <= D) m.a = v - 1;
    int e = 1 + D;
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = a; b < D; ++b) {
            if (v == e) {
                m.a = a;
                m.b = b;
            }
            ++e;
        }
    m.c = m.a < 0 ? 1u : (m.b < 0 ? 2u : 4u);
    m.fv = field_of<D>(v);
    m.fa = m.b >= 0 ? field_of<D>(1 + m.a) : 0u;
    m.fb = m.b >= 0 ? field_of<D>(1 + m.b) : 0u;
    return m;
}
// The factors of a tile or region that starts at pixel kb.
struct WordScale {
    unsigned m1, m2;
    unsigned long long m3;
};
__device__ __forceinline__ WordScale word_scale(const WordMap &m, const int (&kb)[3]) {
    const unsigned o0 = 2u * (unsigned)kb[0] + 1u, o1 = 2u * (unsigned)kb[1] + 1u, o2 = 2u * (unsigned)kb[2] + 1u;
    const unsigned oa = m.a == 0 ? o0 : (m.a == 1 ? o1 : o2), ob = m.b == 0 ? o0 : (m.b == 1 ? o1 : o2);
    WordScale s;
    s.m1 = m.b >= 0 ? 2u * ob : 0u;
    s.m2 = m.b >= 0 ? 2u * oa : 0u;
    s.m3 = m.a < 0 ? 0ull : (m.b < 0 ? (unsigned long long)oa : (unsigned long long)oa * ob);
    return s;
}
__device__ __forceinline__ unsigned long long word_of(const WordMap &m, const WordScale &s, unsigned xv, unsigned xa,
                                                      unsigned xb, unsigned n) {
    return (unsigned long long)m.c * xv + (unsigned long long)s.m1 * xa + (unsigned long long)s.m2 * xb + s.m3 * n;
}
// The warp's word from the packed reductions p.
template <int D>
__device__ __forceinline__ unsigned long long packed_word(const WordMap &m, const WordScale &s, const unsigned (&p)[5]) {
    auto field = [&](unsigned f) -> unsigned {
        const unsigned i = f >> 1;
        if (D == 3) {
            const unsigned w = i == 0u ? p[0] : (i == 1u ? p[1] : (i == 2u ? p[2] : (i == 3u ? p[3] : p[4])));
            return (f & 1u) ? w >> 16 : w & 0xffffu;
        }
        const unsigned w = i == 1u ? p[1] : p[2];
        const unsigned v = (f & 1u) ? w >> 16 : w & 0xffffu;
        return i == 0u ? ((f & 1u) ? p[0] >> 20 : p[0] & 0xfffffu) : v;
    };
    const unsigned n = D == 3 ? p[0] & 0xffffu : p[0] >> 20;
    return word_of(m, s, field(m.fv), field(m.fa), field(m.fb), n);
}
// The word of a full box of cnt[a] pixels per axis.
template <int D>
__device__ __forceinline__ unsigned long long box_word(const WordMap &m, const WordScale &s, const int (&cnt)[3]) {
    unsigned n = 1u;
    unsigned s1[3] = {0u, 0u, 0u}, s2[3] = {0u, 0u, 0u};
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const unsigned k = (unsigned)cnt[a];
        n *= k;
        s1[a] = k * (k - 1u) / 2u;
        s2[a] = k * (k - 1u) * (2u * k - 1u) / 6u;
    }
    auto pick = [](int a, const unsigned (&t)[3]) { return a == 0 ? t[0] : (a == 1 ? t[1] : t[2]); };
    const unsigned cu[3] = {(unsigned)cnt[0], (unsigned)cnt[1], (unsigned)cnt[2]};
    const unsigned na = n / max(pick(m.a, cu), 1u);
    const unsigned xa = m.a < 0 ? 0u : pick(m.a, s1) * na;
    if (m.a < 0) return n;
    if (m.b < 0) return word_of(m, s, xa, 0u, 0u, n);
    const unsigned nb = n / max(pick(m.b, cu), 1u);
    const unsigned xb = pick(m.b, s1) * nb;
    const unsigned xab = m.a == m.b ? pick(m.a, s2) * na : pick(m.a, s1) * pick(m.b, s1) * (na / max(pick(m.b, cu), 1u));
    return word_of(m, s, xab, xa, xb, n);
}

// Packed sums of a label's pixels over the warp: mask[r] the lane's row r (of eight
// pixels from x0), y0 / z0 its first row; rows r = 1 lie 4 planes (3D) or 8 rows (2D)
// further.  Every half stays below 2^16 (2D: sum x^2 < 2^18 beside the count).
template <int D>
__device__ __forceinline__ void packed_sums(const unsigned *lut, const unsigned (&mask)[2], unsigned x0, unsigned y0,
                                            unsigned z0, unsigned (&p)[5]) {
    const unsigned full = 0xffffffffu;
    unsigned c[2], sx[2], sxx[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const unsigned t = lut[mask[r]];
        c[r] = t & 0xffu;
        const unsigned x1 = (t >> 8) & 0xffu, x2 = t >> 16;
        if (D == 3) {
            sx[r] = x1;
            sxx[r] = x2;
        } else {
            sx[r] = x1 + x0 * c[r];
            sxx[r] = x2 + x0 * (2u * x1 + x0 * c[r]);
        }
    }
    const unsigned cc = c[0] + c[1], xx = sx[0] + sx[1], x2 = sxx[0] + sxx[1];
    if (D == 3) {
        const unsigned zb = z0 + 4u;
        const unsigned zc = z0 * c[0] + zb * c[1], zx = z0 * sx[0] + zb * sx[1];
        const unsigned zz = z0 * z0 * c[0] + zb * zb * c[1];
        p[0] = __reduce_add_sync(full, cc | (xx << 16));
        p[1] = __reduce_add_sync(full, (y0 * cc) | (zc << 16));
        p[2] = __reduce_add_sync(full, x2 | ((y0 * y0 * cc) << 16));
        p[3] = __reduce_add_sync(full, zz | ((y0 * xx) << 16));
        p[4] = __reduce_add_sync(full, zx | ((y0 * zc) << 16));
    } else {
        const unsigned yb = y0 + 8u;
        const unsigned yc = y0 * c[0] + yb * c[1], yx = y0 * sx[0] + yb * sx[1];
        const unsigned yy = y0 * y0 * c[0] + yb * yb * c[1];
        p[0] = __reduce_add_sync(full, x2 | (cc << 20));
        p[1] = __reduce_add_sync(full, xx | (yc << 16));
        p[2] = __reduce_add_sync(full, yx | (yy << 16));
        p[3] = p[4] = 0u;
    }
}

// Once per block: the row-mask table.  Followed by a barrier before the first tile.
template <int D>
__device__ __forceinline__ void init_shared(Shared<D> &sm) {
    for (int m = threadIdx.x; m < 256; m += blockDim.x) {
        unsigned c = 0u, x1 = 0u, x2 = 0u;
#pragma unroll
        for (int b = 0; b < 8; ++b)
            if ((m >> b) & 1) {
                c += 1u;
                x1 += (unsigned)b;
                x2 += (unsigned)(b * b);
            }
        sm.lut[m] = c | (x1 << 8) | (x2 << 16);
    }
}

// Lower bound of the costs of group gb's seeds (relative to w_ref) over an absolute
// box of pixel centres (outward slack and roundings).
template <int D>
__device__ __forceinline__ float group_lower(const GroupBound &gb, const float (&alo)[3], const float (&ahi)[3]) {
    float d2 = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const float slack = 1e-6f * (fabsf(alo[a]) + fabsf(ahi[a]) + fabsf(gb.lo[a]) + fabsf(gb.hi[a]));
        const float q = fmaxf(fmaxf(gb.lo[a] - ahi[a], alo[a] - gb.hi[a]) - slack, 0.f);
        d2 = __fmaf_rd(q, q, d2);
    }
    return __fadd_rd(__fmul_rd(__fmul_rd(gb.lam, d2), 1.f - 1e-5f), gb.wgap);
}

struct Box {
    float ch[3], cl[3], rr[3];
};

// Where the list is too short: the same test of every seed against the region's reference,
// a bit per seed.  Out of line, and its work done twice, since few regions come here.
template <int D>
__device__ __noinline__ void mask_groups(Shared<D> &sm, const Src &s, const Box b) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned full = 0xffffffffu;
    const float zero3[3] = {0.f, 0.f, 0.f};
    const unsigned k = lane < kWarps ? sm.key[lane] : 0xffffffffu;
    const unsigned km = __reduce_min_sync(full, k);
    Local<D> R;
    int a0;
    load_local<D>(sm.ref[__ffs(__ballot_sync(full, lane < kWarps && k == km)) - 1], R, a0);
    for (int grp = wid; grp < s.n_groups; grp += kWarps) {
        const int p = grp * 32 + lane;
        bool keep = false;
        if (p < s.n) {
            Local<D> L;
            Diff<D> F;
            local_terms<D>(s.recs[p], b.ch, b.cl, zero3, b.rr, s.gf, L);
            difference<D>(L, R, F);
            keep = p == a0 || can_win<D>(F, b.rr);
        }
        const unsigned bits = __ballot_sync(full, keep);
        if (lane == 0) sm.mask[grp] = bits;
    }
}

// The seeds that can be the argmin somewhere in the box of half-widths rr around ch + cl,
// listed in sm.list by the whole block (two barriers; none follows the last entry's
// write but the second).  Returns their number, which may exceed kListCap (the list is
// then incomplete); r0h + r0l is the reference seed's weight.
template <int D>
__device__ __forceinline__ unsigned region_list(Shared<D> &sm, const Src &s, const float (&ch)[3], const float (&cl)[3],
                                                const float (&rr)[3], float &r0h, float &r0l) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned full = 0xffffffffu;
    const float finf = __int_as_float(0x7f800000);
    const int n = s.n;
    float4(&ref)[5] = sm.ref[wid];
    const float zero3[3] = {0.f, 0.f, 0.f};
    const float wrh = s.sc->wref_h, wrl = s.sc->wref_l;

    // the groups' lower bounds: warp w takes the groups w, w + 8, ... (one per lane and
    // round, so that near groups, adjacent in scan order, go to different warps)
    float glb[2] = {finf, finf};
    {
        float alo[3] = {0.f, 0.f, 0.f}, ahi[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < D; ++a) {
            alo[a] = __fsub_rd(ch[a], __fadd_ru(rr[a], fabsf(cl[a])));
            ahi[a] = __fadd_ru(ch[a], __fadd_ru(rr[a], fabsf(cl[a])));
        }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            if (s.n_groups <= t * kThreads) break;
            const int grp = wid + kWarps * (lane + 32 * t);
            if (grp < s.n_groups) glb[t] = group_lower<D>(s.groups[grp], alo, ahi);
        }
    }
    // each warp's group of least bound, and in it the seed of least cost at the centre
    // with an upper bound U of its cost over the region (relative to w_ref)
    {
        const unsigned k0 = okey(fminf(glb[0], glb[1]));
        const unsigned kmin = __reduce_min_sync(full, k0);
        const int src = __ffs(__ballot_sync(full, k0 == kmin)) - 1;
        const int t = glb[0] <= glb[1] ? 0 : 1;
        const int grp = wid + kWarps * (src + 32 * __shfl_sync(full, t, src));
        unsigned ck = 0xffffffffu;
        const int p = grp * 32 + lane;
        Local<D> L;
        float wn = 0.f;
        const bool have = grp < s.n_groups && p < n;
        if (have) {
            local_terms<D>(s.recs[p], ch, cl, zero3, rr, s.gf, L);
            wn = -((L.wh - wrh) + (L.wl - wrl));
            ck = min(okey(L.q + wn), 0xfffffffeu);
        }
        const unsigned cm = __reduce_min_sync(full, ck);
        const int who = __ffs(__ballot_sync(full, ck == cm)) - 1;
        if (lane == who) {
            sm.key[wid] = cm;
            if (have) {
                float v = L.q + 1e-5f * (L.S + fabsf(wn)) + 1e-30f;
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    v += 2.f * fabsf(L.h[a]) * rr[a];
#pragma unroll
                    for (int b = 0; b < D; ++b) v += fabsf(L.a[tri<D>(a < b ? a : b, a < b ? b : a)]) * rr[a] * rr[b];
                }
                store_local<D>(ref, L, p);
                ref[4].x = v + wn + 1e-5f * (fabsf(v) + fabsf(wn)) + 1e-13f * fabsf(L.wh);
            }
        }
    }
    if (tid == 0) {
        sm.count = 0u;
    }
    __syncthreads();
    Local<D> R;
    int a0;
    float U;
    {
        const unsigned k = lane < kWarps ? sm.key[lane] : 0xffffffffu;
        const unsigned km = __reduce_min_sync(full, k);
        const int w = __ffs(__ballot_sync(full, lane < kWarps && k == km)) - 1;
        load_local<D>(sm.ref[w], R, a0);
        U = sm.ref[w][4].x;
    }
    r0h = R.wh;
    r0l = R.wl;
    // the seeds that can win somewhere in the region against a0
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        if (s.n_groups <= t * kThreads) break;
        unsigned m = __ballot_sync(full, !(glb[t] > U) && wid + kWarps * (lane + 32 * t) < s.n_groups);
        while (m) {
            const int gl = __ffs(m) - 1;
            m &= m - 1u;
            const int p = (wid + kWarps * (gl + 32 * t)) * 32 + lane;
            bool keep = false;
            if (p < n) {
                Local<D> L;
                Diff<D> F;
                local_terms<D>(s.recs[p], ch, cl, zero3, rr, s.gf, L);
                difference<D>(L, R, F);
                keep = p == a0 || can_win<D>(F, rr);
            }
            const unsigned km = __ballot_sync(full, keep);
            if (km) {
                unsigned at = 0u;
                if (lane == 0) at = atomicAdd(&sm.count, (unsigned)__popc(km));
                at = __shfl_sync(full, at, 0) + (unsigned)__popc(km & ((1u << lane) - 1u));
                if (keep && at < (unsigned)kListCap) sm.list[at] = (uint16_t)p;
            }
        }
    }
    __syncthreads();
    const unsigned total = sm.count;
    if (total > (unsigned)kListCap) {
        mask_groups<D>(sm, s, Box{{ch[0], ch[1], ch[2]}, {cl[0], cl[1], cl[2]}, {rr[0], rr[1], rr[2]}});
        __syncthreads();
    }
    return total;
}

// The seeds that region_list has listed, in chunks of a warp.
template <int D>
struct Listed {
    unsigned total;
    bool scan;  // too many for the list: chunk c is what is listed of group c
    int chunks;
    __device__ __forceinline__ Listed(const Src &s, unsigned total_)
        : total(total_), scan(total_ > (unsigned)kListCap), chunks(scan ? s.n_groups : (int)((total_ + 31u) / 32u)) {}
    __device__ __forceinline__ bool none(const Shared<D> &sm, int c) const { return scan && sm.mask[c] == 0u; }
    // scan position of this lane's candidate of chunk c (-1: none)
    __device__ __forceinline__ int at(const Shared<D> &sm, int c) const {
        const int lane = threadIdx.x & 31, e = c * 32 + lane;
        if (scan) return (sm.mask[c] >> lane) & 1u ? e : -1;
        return e < (int)total ? (int)sm.list[e] : -1;
    }
};

// The warp's tile's offset from the region's centre and half-widths (rounded up).
template <int D>
__device__ __forceinline__ void tile_box(const GridDev &g, const int (&tc)[3], float (&toff)[3], float (&tr)[3]) {
    using G = Geom<D>;
    const int tdim[3] = {G::TX, G::TY, G::TZ}, rdim[3] = {G::RX, G::RY, G::RZ};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        toff[a] = a < D ? (float)(tc[a] * tdim[a] + tdim[a] / 2 - rdim[a] / 2) * g.h32[a] : 0.f;
        tr[a] = a < D ? __fmul_ru(__fmul_ru(0.5f * (float)(tdim[a] - 1), g.h32[a]), 1.f + 0x1p-22f) : 0.f;
    }
}
template <int D>
__device__ __forceinline__ void warp_tile(int wid, int (&tc)[3]) {
    using G = Geom<D>;
    tc[0] = wid % (G::RX / G::TX);
    tc[1] = (wid / (G::RX / G::TX)) % (G::RY / G::TY);
    tc[2] = wid / ((G::RX / G::TX) * (G::RY / G::TY));
}

// The polynomial of seed p as entry `at` of the warp's buffer.
template <int D>
__device__ __forceinline__ void put_poly(float4 (*buf)[3], int at, const Src &s, int p, const Diff<D> &F) {
    constexpr int NP = Geom<D>::NP;
    const int id = s.perm ? s.perm[p] : p;
    buf[at][0] = make_float4(F.d0, F.g[0], F.g[1], D == 3 ? F.g[D - 1] : 0.f);
    if (D == 3) {
        buf[at][1] = make_float4(F.a[0], 2.f * F.a[1], 2.f * F.a[2], F.a[NP - 3]);
        buf[at][2] = make_float4(2.f * F.a[NP - 2], F.a[NP - 1], __int_as_float(id), 0.f);
    } else {
        buf[at][1] = make_float4(F.a[0], 2.f * F.a[1], F.a[2], __int_as_float(id));
    }
}

// A tile whose polynomials do not fit the warp's buffer: piece c of them formed again,
// from the tile's list where it is complete (`listed` seeds), else from the region's.
// Returns their number.
template <int D>
__device__ __forceinline__ int refill(Shared<D> &sm, const Src &s, const uint16_t *tile, const int bx, const int by,
                                   const int bz, const int c, const int listed, const int best_pos) {
    using G = Geom<D>;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int k[3] = {bx * G::RX + G::RX / 2, by * G::RY + G::RY / 2, bz * G::RZ + G::RZ / 2};
    float ch[3] = {0.f, 0.f, 0.f}, cl[3] = {0.f, 0.f, 0.f}, toff[3], tr[3];
#pragma unroll
    for (int a = 0; a < D; ++a) axis_point(s.gf, a, k[a], ch[a], cl[a]);
    int tc[3];
    warp_tile<D>(wid, tc);
    tile_box<D>(s.g, tc, toff, tr);
    Local<D> R, L;
    int id;
    load_local<D>(sm.ref[wid], R, id);
    const bool kept = listed <= s.tile_cap;
    int p;
    if (kept) p = 32 * c + lane < listed ? (int)tile[32 * c + lane] : -1;
    else p = Listed<D>(s, sm.count).at(sm, c);
    __syncwarp();
    bool keep = false;
    Diff<D> F;
    if (p >= 0 && p != best_pos) {
        local_terms<D>(s.recs[p], ch, cl, toff, tr, s.gf, L);
        difference<D>(L, R, F);
        keep = kept || can_win<D>(F, tr);
    }
    const unsigned km = __ballot_sync(0xffffffffu, keep);
    if (keep) put_poly<D>(sm.poly[wid], __popc(km & ((1u << lane) - 1u)), s, p, F);
    __syncwarp();
    return __popc(km);
}

// The warp's tile of region (bx, by, bz): its first pixel, the pixels of it that are scored.
template <int D>
struct TileWindow {
    int tc[3], kb[3], lo3[3], cnt[3];
    bool empty, whole;
    __device__ __forceinline__ TileWindow(const GridDev &g, const int bx, const int by, const int bz)
        : empty(false), whole(true) {
        using G = Geom<D>;
        const int tdim[3] = {G::TX, G::TY, G::TZ};
        const int rb[3] = {bx * G::RX, by * G::RY, bz * G::RZ};
        warp_tile<D>(threadIdx.x >> 5, tc);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            kb[a] = rb[a] + tc[a] * tdim[a];
            int lo = kb[a], hi = kb[a] + tdim[a];
            if (a < D) {
                hi = min(hi, a == D - 1 ? win_hi(g) : g.res[a]);
                if (a == D - 1) lo = max(lo, win_lo(g));
            }
            lo3[a] = lo;
            cnt[a] = hi - lo;
            empty = empty || cnt[a] <= 0;
            whole = whole && cnt[a] == tdim[a];
        }
    }
};

// A lane's two rows of eight pixels.
template <int D>
struct LaneRows {
    int x0, y0, z0, k0, kb1, kb2;  // first pixel and rows in the tile, in the grid
    unsigned wmask;
    __device__ __forceinline__ LaneRows(const GridDev &g, const int (&kb)[3]) {
        const int lane = threadIdx.x & 31;
        x0 = D == 3 ? 0 : 8 * (lane & 3);
        y0 = D == 3 ? (lane & 7) : (lane >> 2);
        z0 = D == 3 ? (lane >> 3) : 0;
        k0 = kb[0] + x0;
        kb1 = kb[1];
        kb2 = kb[2];
        const int w0 = min(8, g.res[0] - k0);
        wmask = w0 >= 8 ? 0xffu : (w0 > 0 ? (1u << w0) - 1u : 0u);
    }
    __device__ __forceinline__ int k1(int r) const { return kb1 + (D == 3 ? y0 : y0 + 8 * r); }
    __device__ __forceinline__ int k2(int r) const { return D == 3 ? kb2 + z0 + 4 * r : 0; }
    // row r: the pixels scored
    __device__ __forceinline__ unsigned valid(const GridDev &g, int r) const {
        const int kl = D == 3 ? k2(r) : k1(r);
        return k1(r) < g.res[1] && kl >= win_lo(g) && kl < win_hi(g) ? wmask : 0u;
    }
    __device__ __forceinline__ void put_labels(const Src &s, int r, unsigned vm, const unsigned (&lab)[8]) const {
        const GridDev &g = s.g;
        const long long plane = (long long)g.res[0] * (long long)g.res[1];
        int32_t *q = s.labels + ((long long)k0 + (long long)g.res[0] * k1(r) + plane * k2(r));
        if (vm == 0xffu && (reinterpret_cast<uintptr_t>(q) & 15) == 0) {
            reinterpret_cast<int4 *>(q)[0] = make_int4(lab[0], lab[1], lab[2], lab[3]);
            reinterpret_cast<int4 *>(q)[1] = make_int4(lab[4], lab[5], lab[6], lab[7]);
        } else {
#pragma unroll
            for (int p = 0; p < 8; ++p)
                if ((vm >> p) & 1u) q[p] = (int)lab[p];
        }
    }
};

// Labels and moments of the warp's tile from its polynomials less the reference's:
// each(f) calls f(k) for every one, in buffer entry k; m of them with `fast`, else any
// number.  Emax: the largest E of the list.
template <int D, bool MASKED, class Each>
__device__ __forceinline__ void score_pixels(Shared<D> &sm, const Src &s, const int (&kb)[3], const int (&cnt)[3],
                                             const bool whole, const unsigned (&marked)[2], const int ref_id,
                                             const float Emax, const bool fast, const int m, const Each each) {
    using G = Geom<D>;
    constexpr int K = moment_width(D);
    const GridDev &g = s.g;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned full = 0xffffffffu;
    const float finf = __int_as_float(0x7f800000);
    const int n = s.n;
    const LaneRows<D> rows(g, kb);
    const int x0 = rows.x0, y0 = rows.y0, z0 = rows.z0;
    const float4(*buf)[3] = sm.poly[wid];
    const WordMap wm = word_map<D>();
    auto row_mask = [&](int r) -> unsigned { return MASKED ? marked[r] : rows.valid(g, r); };
    // ---- pixels: lane owns two rows of eight ----
    float2 dx[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
        dx[q] = make_float2(((float)(x0 + 2 * q - G::TX / 2) + 0.5f) * g.h32[0],
                            ((float)(x0 + 2 * q + 1 - G::TX / 2) + 0.5f) * g.h32[0]);
    const float gap = 2.f * Emax;
    const WordScale ws = word_scale(wm, kb);
    // the costs of buffer entry k on the row (f1, f2), less the reference's; its seed
    auto row_values = [&](int k, float f1, float f2, float (&v)[8]) -> unsigned {
        const float4 v0 = buf[k][0], v1 = buf[k][1];
        float a, b;
        unsigned id;
        if (D == 3) {
            const float4 v2 = buf[k][2];
            b = fmaf(v1.z, f2, fmaf(v1.y, f1, v0.y));
            const float t1 = fmaf(v2.x, f2, fmaf(v1.w, f1, v0.z));
            const float t2 = fmaf(v2.y, f2, v0.w);
            a = fmaf(f2, t2, fmaf(f1, t1, v0.x));
            id = __float_as_uint(v2.z);
        } else {
            b = fmaf(v1.y, f1, v0.y);
            a = fmaf(f1, fmaf(v1.z, f1, v0.z), v0.x);
            id = __float_as_uint(v1.w);
        }
        const float2 q2 = make_float2(v1.x, v1.x), bb = make_float2(b, b), aa = make_float2(a, a);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 t = ffma2(ffma2(q2, dx[q], bb), dx[q], aa);
            v[2 * q] = t.x;
            v[2 * q + 1] = t.y;
        }
        return id;
    };
    auto row_offsets = [&](int r, float &f1, float &f2) {
        f1 = ((float)((D == 3 ? y0 : y0 + 8 * r) - G::TY / 2) + 0.5f) * g.h32[1];
        f2 = D == 3 ? ((float)(z0 + 4 * r - G::TZ / 2) + 0.5f) * g.h32[2] : 0.f;
    };
    unsigned nq = 0u;  // near ties of the tile, in the warp's queue
    auto enqueue = [&](int r, unsigned qm) {
        if (!__any_sync(full, qm != 0u)) return;
        const int c = __popc(qm);
        int sum = c;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int t = __shfl_up_sync(full, sum, off);
            if (lane >= off) sum += t;
        }
        int at = (int)nq + sum - c;
        const int first = x0 + G::TX * (D == 3 ? y0 + G::TY * (z0 + 4 * r) : y0 + 8 * r);
        for (unsigned q = qm; q; q &= q - 1u) sm.queue[wid][at++] = (uint16_t)(first + __ffs(q) - 1);
        nq += (unsigned)__shfl_sync(full, sum, 31);
    };
    unsigned pk[5];
    if (fast) {
        // byte k (of two words) of mk[r]: the pixels of row r that entry k holds
        unsigned mlo[2], mhi[2], okm[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float f1, f2, b1[8], b2[8];
            row_offsets(r, f1, f2);
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                b1[p] = 0.f;
                b2[p] = finf;
            }
            unsigned lo = 0u, hi = 0u;
            for (int k = 0; k < m; ++k) {
                float v[8];
                row_values(k, f1, f2, v);
                unsigned nm = 0u;
#pragma unroll
                for (int p = 0; p < 8; ++p) {
                    if (v[p] < b1[p]) nm |= 1u << p;
                    b2[p] = fminf(b2[p], fmaxf(b1[p], v[p]));
                    b1[p] = fminf(b1[p], v[p]);
                }
                const unsigned rep = ~(nm * 0x01010101u);
                const unsigned own = nm << (8 * (k & 3));
                lo = (lo & rep) | (k < 4 ? own : 0u);
                hi = (hi & rep) | (k < 4 ? 0u : own);
            }
            unsigned qm = 0u;
#pragma unroll
            for (int p = 0; p < 8; ++p)
                if (!(b2[p] - b1[p] > gap)) qm |= 1u << p;
            const unsigned vm = row_mask(r);
            qm &= vm;
            if (s.labels && vm) {
                unsigned lab[8];
#pragma unroll
                for (int p = 0; p < 8; ++p) lab[p] = (unsigned)ref_id;
                for (int k = 0; k < m; ++k) {
                    const unsigned id = __float_as_uint(D == 3 ? buf[k][2].z : buf[k][1].w);
                    const unsigned mk = ((k < 4 ? lo : hi) >> (8 * (k & 3)));
#pragma unroll
                    for (int p = 0; p < 8; ++p) lab[p] = (mk >> p) & 1u ? id : lab[p];
                }
                rows.put_labels(s, r, vm, lab);
            }
            enqueue(r, qm);
            const unsigned ok = vm & ~qm;
            okm[r] = ok;
            mlo[r] = lo & (ok * 0x01010101u);
            mhi[r] = hi & (ok * 0x01010101u);
        }
        unsigned long long others = 0ull;
        for (int k = 0; k < m; ++k) {
            const unsigned sh = 8 * (k & 3);
            const unsigned mask[2] = {((k < 4 ? mlo[0] : mhi[0]) >> sh) & 0xffu, ((k < 4 ? mlo[1] : mhi[1]) >> sh) & 0xffu};
            okm[0] &= ~mask[0];
            okm[1] &= ~mask[1];
            if (!__any_sync(full, (mask[0] | mask[1]) != 0u)) continue;
            const int id = __float_as_int(D == 3 ? buf[k][2].z : buf[k][1].w);
            packed_sums<D>(sm.lut, mask, (unsigned)x0, (unsigned)y0, (unsigned)z0, pk);
            const unsigned long long word = packed_word<D>(wm, ws, pk);
            others += word;
            if (lane < K) atomicAdd(&s.gmom[(size_t)id * K + lane], word);
        }
        // the reference's pixels: the rest of a whole tile without near ties
        unsigned long long word = 0ull;
        if (whole && nq == 0u) {
            word = box_word<D>(wm, ws, cnt) - others;
        } else if (__any_sync(full, (okm[0] | okm[1]) != 0u)) {
            packed_sums<D>(sm.lut, okm, (unsigned)x0, (unsigned)y0, (unsigned)z0, pk);
            word = packed_word<D>(wm, ws, pk);
        }
        if (lane < K && word) atomicAdd(&s.gmom[(size_t)ref_id * K + lane], word);
    } else {
        unsigned lab[2][8];  // seed index; 0xffffffff: outside the grid or a near tie
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float f1, f2, b1[8], b2[8];
            row_offsets(r, f1, f2);
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                b1[p] = 0.f;
                b2[p] = finf;
                lab[r][p] = (unsigned)ref_id;
            }
            each([&](int k) {
                float v[8];
                const unsigned id = row_values(k, f1, f2, v);
#pragma unroll
                for (int p = 0; p < 8; ++p) {
                    b2[p] = fminf(b2[p], fmaxf(b1[p], v[p]));
                    lab[r][p] = v[p] < b1[p] ? id : lab[r][p];
                    b1[p] = fminf(b1[p], v[p]);
                }
            });
            unsigned qm = 0u;
#pragma unroll
            for (int p = 0; p < 8; ++p)
                if (!(b2[p] - b1[p] > gap)) qm |= 1u << p;
            const unsigned vm = row_mask(r);
            qm &= vm;
            if (s.labels && vm) rows.put_labels(s, r, vm, lab[r]);
            enqueue(r, qm);
            const unsigned ok = vm & ~qm;
#pragma unroll
            for (int p = 0; p < 8; ++p)
                if (!((ok >> p) & 1u)) lab[r][p] = 0xffffffffu;
        }
        while (true) {  // label by label in increasing order
            unsigned mn = 0xffffffffu;
#pragma unroll
            for (int p = 0; p < 8; ++p) mn = min(mn, min(lab[0][p], lab[1][p]));
            mn = __reduce_min_sync(full, mn);
            if (mn >= (unsigned)n) break;
            unsigned mask[2] = {0u, 0u};
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int p = 0; p < 8; ++p)
                    if (lab[r][p] == mn) {
                        mask[r] |= 1u << p;
                        lab[r][p] = 0xffffffffu;
                    }
            packed_sums<D>(sm.lut, mask, (unsigned)x0, (unsigned)y0, (unsigned)z0, pk);
            const unsigned long long word = packed_word<D>(wm, ws, pk);
            if (lane < K) atomicAdd(&s.gmom[(size_t)mn * K + lane], word);
        }
    }

    // ---- near ties, a lane per pixel: every seed within the gap of the least value is
    // a candidate (any other costs more); the candidates' FP64 costs in the reference
    // arithmetic decide, the lowest index on ties ----
    if (nq == 0u) return;
    if (lane == 0) atomicAdd(&sm.queued, nq);
    __syncwarp();
    for (unsigned base = 0; base < nq; base += 32u) {
        const bool act = base + (unsigned)lane < nq;
        const int px = act ? (int)sm.queue[wid][base + lane] : 0;
        const int xl = px % G::TX, yl = (px / G::TX) % G::TY, zl = px / (G::TX * G::TY);
        const float f0 = ((float)(xl - G::TX / 2) + 0.5f) * g.h32[0];
        const float f1 = ((float)(yl - G::TY / 2) + 0.5f) * g.h32[1];
        const float f2 = D == 3 ? ((float)(zl - G::TZ / 2) + 0.5f) * g.h32[2] : 0.f;
        auto value = [&](int k, int &id) -> float {
            const float4 v0 = buf[k][0], v1 = buf[k][1];
            if (D == 3) {
                const float4 v2 = buf[k][2];
                const float b = fmaf(v1.z, f2, fmaf(v1.y, f1, v0.y));
                const float t1 = fmaf(v2.x, f2, fmaf(v1.w, f1, v0.z));
                const float t2 = fmaf(v2.y, f2, v0.w);
                id = __float_as_int(v2.z);
                return fmaf(fmaf(v1.x, f0, b), f0, fmaf(f2, t2, fmaf(f1, t1, v0.x)));
            }
            id = __float_as_int(v1.w);
            return fmaf(fmaf(v1.x, f0, fmaf(v1.y, f1, v0.y)), f0, fmaf(f1, fmaf(v1.z, f1, v0.z), v0.x));
        };
        float v1 = 0.f, v2 = finf, v3 = finf;  // the three least values, the seeds of two
        int i1 = ref_id, i2 = -1;
        each([&](int k) {
            int id;
            const float v = value(k, id);
            const bool lt1 = v < v1, lt2 = v < v2;
            v3 = lt2 ? v2 : fminf(v3, v);
            v2 = lt1 ? v1 : (lt2 ? v : v2);
            i2 = lt1 ? i1 : (lt2 ? id : i2);
            v1 = lt1 ? v : v1;
            i1 = lt1 ? id : i1;
        });
        const float thr = v1 + gap;
        const int kp[3] = {kb[0] + xl, kb[1] + yl, kb[2] + zl};
        double y[D];
#pragma unroll
        for (int a = 0; a < D; ++a) y[a] = __dadd_rn(g.lo[a], __dmul_rn((double)kp[a] + 0.5, g.h[a]));
        double cb = __longlong_as_double(0x7ff0000000000000ll);
        int ib = 0x7fffffff;
        auto settle = [&](int id) {
            const double c = cost64<D>(y, s.x + (size_t)id * D, s.A + (size_t)id * D * D, s.w[id]);
            if (c < cb || (c == cb && id < ib)) {
                cb = c;
                ib = id;
            }
        };
        if (act) settle(i1);
        if (act && i2 >= 0 && !(v2 > thr)) settle(i2);
        const bool more = act && !(v3 > thr);
        if (__any_sync(full, more)) {  // three candidates or more
            if (more && i1 != ref_id && i2 != ref_id && !(0.f > thr)) settle(ref_id);
            each([&](int k) {
                int id;
                const float v = value(k, id);
                if (more && !(v > thr) && id != i1 && id != i2) settle(id);
            });
        }
        if (act) {
            if (ib < 0 || ib >= n) {
                atomicOr(&s.sc->status, ST_BAD_LABEL);
            } else {
                if (s.labels)
                    s.labels[(long long)kp[0] + (long long)g.res[0] * kp[1] + (D == 3 ? (long long)g.res[0] * (long long)g.res[1] * kp[2] : 0ll)] = ib;
                unsigned long long u[3], *o = s.gmom + (size_t)ib * K;
#pragma unroll
                for (int a = 0; a < D; ++a) u[a] = 2ull * (unsigned long long)kp[a] + 1ull;
                atomicAdd(&o[0], 1ull);
#pragma unroll
                for (int a = 0; a < D; ++a) atomicAdd(&o[1 + a], u[a]);
                int e = 1 + D;
#pragma unroll
                for (int a = 0; a < D; ++a)
#pragma unroll
                    for (int b = a; b < D; ++b) atomicAdd(&o[e++], u[a] * u[b]);
            }
        }
    }
}

// A tile whose polynomials do not fit the warp's buffer: they are formed again for every
// pass over them (refill).  Out of line, with what it needs formed again too: beside the
// other tiles' code the passes cost those registers and a tenth of their instructions (a
// batch of 48 2D diagrams: 71.3 M warp instructions an evaluation, so 65.8 M; spills 512 /
// 1108 bytes, so 144 / 352 in 3D).
template <int D, bool MASKED>
__device__ __noinline__ void score_pixels_refilled(Shared<D> &sm, const Src &s, const uint16_t *tile, const int bx,
                                                   const int by, const int bz, const unsigned marked0,
                                                   const unsigned marked1, const int listed, const int best_pos,
                                                   const float Emax) {
    const unsigned full = 0xffffffffu;
    const TileWindow<D> t(s.g, bx, by, bz);
    const unsigned marked[2] = {marked0, marked1};
    const bool whole = MASKED ? __all_sync(full, marked0 == 0xffu && marked1 == 0xffu) : t.whole;
    const int ref_id = __float_as_int(sm.ref[threadIdx.x >> 5][1].w);  // see store_local
    const int pieces = listed <= s.tile_cap ? (listed + 31) / 32 : Listed<D>(s, sm.count).chunks;
    score_pixels<D, MASKED>(sm, s, t.kb, t.cnt, whole, marked, ref_id, Emax, false, 0, [&](auto f) {
        for (int c = 0; c < pieces; ++c) {
            const int m = refill<D>(sm, s, tile, bx, by, bz, c, listed, best_pos);
            for (int k = 0; k < m; ++k) f(k);
        }
    });
}

// Scores region (bx, by, bz); `s` is the same in every thread; `tiles`: kWarps lists of
// tile_cap positions in shared memory.  The caller puts a barrier between the previous
// region and the next.
template <int D, bool MASKED = false>
__device__ __forceinline__ void score_region(Shared<D> &sm, uint16_t *tiles, const Src &s, const int bx, const int by,
                                             const int bz) {
    using G = Geom<D>;
    constexpr int K = moment_width(D);
    const GridDev &g = s.g;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned full = 0xffffffffu;
    const int rdim[3] = {G::RX, G::RY, G::RZ};
    const int rb[3] = {bx * G::RX, by * G::RY, bz * G::RZ};
    float4(&ref)[5] = sm.ref[wid];

    const TileWindow<D> win(g, bx, by, bz);
    const int (&kb)[3] = win.kb;
    float toff[3], tr[3];
    tile_box<D>(g, win.tc, toff, tr);
    bool empty = win.empty, whole = win.whole;
    const LaneRows<D> rows(g, kb);
    unsigned marked[2] = {0u, 0u};
    if constexpr (MASKED) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const unsigned vm = rows.valid(g, r);
            if (!vm) continue;
            const int k0 = rows.k0, k1 = rows.k1(r), k2 = rows.k2(r);
            const uint8_t *row = s.mask + (size_t)s.cres[0] * ((size_t)(k1 / s.r) + (size_t)s.cres[1] * (size_t)(k2 / s.r));
            int kx = k0 / s.r, next = (kx + 1) * s.r;
            bool on = row[kx] != 0;
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                if (!((vm >> p) & 1u)) continue;
                if (k0 + p == next) {
                    on = row[++kx] != 0;
                    next += s.r;
                }
                marked[r] |= on ? 1u << p : 0u;
            }
        }
        whole = __all_sync(full, marked[0] == 0xffu && marked[1] == 0xffu);
        empty = !__any_sync(full, (marked[0] | marked[1]) != 0u);
        if (!__syncthreads_or(!empty)) return;  // no marked pixel in the region
    }

    // region centre (lane a: axis a) as an FP32 pair, half-widths rounded up
    float ch[3] = {0.f, 0.f, 0.f}, cl[3] = {0.f, 0.f, 0.f};
    {
        float h = 0.f, l = 0.f;
        if (lane < D) {
            const int k = lane == 0 ? rb[0] + G::RX / 2 : (lane == 1 ? rb[1] + G::RY / 2 : rb[2] + G::RZ / 2);
            axis_point(s.gf, lane, k, h, l);
        }
#pragma unroll
        for (int a = 0; a < D; ++a) {
            ch[a] = __shfl_sync(full, h, a);
            cl[a] = __shfl_sync(full, l, a);
        }
    }
    float rr[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < D; ++a)
        rr[a] = __fmul_ru(__fmul_ru(0.5f * (float)(rdim[a] - 1), g.h32[a]), 1.f + 0x1p-22f);
    if (tid == 0) {
        sm.pairs = 0u;
        sm.queued = 0u;
    }
    float r0h, r0l;
    const unsigned total = region_list<D>(sm, s, ch, cl, rr, r0h, r0l);
    const Listed<D> src(s, total);
    const int n_src = src.chunks;

    if (empty) return;

    // the listed seed of least cost at the tile's centre
    unsigned best = 0xffffffffu;
    int best_pos = 0x7fffffff;
    Local<D> L;  // of the last chunk (the only one of most lists)
    int pos = -1;
    for (int c = 0; c < n_src; ++c) {
        if (src.none(sm, c)) continue;
        pos = src.at(sm, c);
        unsigned ck = 0xffffffffu;
        if (pos >= 0) {
            local_terms<D>(s.recs[pos], ch, cl, toff, tr, s.gf, L);
            ck = min(okey(L.q - ((L.wh - r0h) + (L.wl - r0l))), 0xfffffffeu);
        }
        const unsigned cm = __reduce_min_sync(full, ck);
        const int who = (int)__reduce_min_sync(full, ck == cm && pos >= 0 ? (unsigned)pos : 0x7fffffffu);
        if (cm < best || (cm == best && who < best_pos)) {
            best = cm;
            best_pos = who;
            if (pos == who && pos >= 0) store_local<D>(ref, L, s.perm ? s.perm[pos] : pos);
        }
    }
    if (best == 0xffffffffu) {  // cannot happen: the region lists a0
        if (lane == 0) atomicOr(&s.sc->status, ST_BAD_LABEL);
        return;
    }
    __syncwarp();
    Local<D> R;
    int ref_id;
    load_local<D>(ref, R, ref_id);

    // polynomials of the seeds that can win somewhere in the tile, compacted
    float Emax = 0.f;
    int m = 0;          // in the buffer
    int listed = 0;     // in all chunks
    float4(*buf)[3] = sm.poly[wid];
    uint16_t *const tile = tiles + wid * s.tile_cap;
    bool one = true;  // every polynomial is in the buffer
    for (int c = 0; c < n_src; ++c) {
        if (src.none(sm, c)) continue;
        const int p = n_src == 1 ? pos : src.at(sm, c);
        bool keep = false;
        Diff<D> F;
        if (p >= 0 && p != best_pos) {
            if (n_src > 1) local_terms<D>(s.recs[p], ch, cl, toff, tr, s.gf, L);
            difference<D>(L, R, F);
            keep = can_win<D>(F, tr);
        }
        const unsigned km = __ballot_sync(full, keep);
        const int before = __popc(km & ((1u << lane) - 1u));
        const int add = __popc(km);
        one = one && m + add <= kBuf;
        if (keep) {
            Emax = fmaxf(Emax, F.E);
            if (one) put_poly<D>(buf, m + before, s, p, F);
            if (total > (unsigned)kBuf && listed + before < s.tile_cap) tile[listed + before] = (uint16_t)p;
        }
        if (one) m += add;
        listed += add;
    }
    Emax = __uint_as_float(__reduce_max_sync(full, __float_as_uint(Emax)));
    __syncwarp();
    if (lane == 0) atomicAdd(&sm.pairs, (unsigned)(listed + 1));
    if (listed == 0) {  // one cell
        const WordMap wm = word_map<D>();
        unsigned long long word;
        if (MASKED && !whole) {
            unsigned pk[5];
            packed_sums<D>(sm.lut, marked, (unsigned)rows.x0, (unsigned)rows.y0, (unsigned)rows.z0, pk);
            word = packed_word<D>(wm, word_scale(wm, kb), pk);
        } else {
            word = box_word<D>(wm, word_scale(wm, win.lo3), win.cnt);
        }
        if (lane < K) atomicAdd(&s.gmom[(size_t)ref_id * K + lane], word);
        if (s.labels) {
            const unsigned id = (unsigned)ref_id;
            const unsigned lab[8] = {id, id, id, id, id, id, id, id};
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (const unsigned vm = MASKED ? marked[r] : rows.valid(g, r)) rows.put_labels(s, r, vm, lab);
        }
        return;
    }

    if (!one) {
        score_pixels_refilled<D, MASKED>(sm, s, tile, bx, by, bz, marked[0], marked[1], listed, best_pos, Emax);
        return;
    }
    score_pixels<D, MASKED>(sm, s, kb, win.cnt, whole, marked, ref_id, Emax, m <= kFast, m, [&](auto f) {
        for (int k = 0; k < m; ++k) f(k);
    });
}

}  // namespace region
}  // namespace apd
