// The pruned scorer of the one-instance calls: one block per grid region
// (apd_region.cuh).
#include "apd_region.cuh"

namespace apd {

namespace {

using namespace region;

// Block b is region b of the scoring window: nx x ny (x nz) regions, the last axis
// starting at region index `toff`.
// Four blocks per SM (64 registers, some spills) were a little faster than three, and those
// than two without spills (256^3, 1000 seeds: the whole call 195, 197 and 207 us with the
// preparation it had then): the lists' two barriers and the dependent loads want more warps
// more than they want registers.  The kernel itself takes 99 us there.
template <int D>
__global__ void __launch_bounds__(kThreads, 4)
    assign_region_kernel(const __grid_constant__ Src src, const int nx, const int ny, const int toff) {
    __shared__ Shared<D> sm;
    extern __shared__ uint16_t tiles[];
    init_shared<D>(sm);
    const int b = (int)blockIdx.x;
    const int bx = b % nx, r = b / nx;
    const int by = D == 3 ? r % ny : r + toff, bz = D == 3 ? r / ny + toff : 0;
    score_region<D>(sm, tiles, src, bx, by, bz);
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(src.pairs_scored, (unsigned long long)sm.pairs * (unsigned long long)kTilePix);
        if (sm.queued) atomicAdd(&src.sc->flag_count, sm.queued);
    }
}

// Masked form: a persistent grid over the listed regions.
template <int D>
__global__ void __launch_bounds__(kThreads, 4)
    masked_region_kernel(const __grid_constant__ Src src, const int nx, const int ny, const int32_t *__restrict__ list) {
    __shared__ Shared<D> sm;
    extern __shared__ uint16_t tiles[];
    init_shared<D>(sm);
    const int count = (int)src.sc->mask_regions;
    unsigned queued = 0u;
    for (int i = (int)blockIdx.x; i < count; i += (int)gridDim.x) {
        if (threadIdx.x == 0) sm.queued = 0u;
        const int b = list[i];
        const int r = b / nx;
        score_region<D, true>(sm, tiles, src, b % nx, D == 3 ? r % ny : r, D == 3 ? r / ny : 0);
        __syncthreads();
        if (threadIdx.x == 0) queued += sm.queued;
    }
    if (threadIdx.x == 0 && queued) atomicAdd(&src.sc->flag_count, queued);
}

template <int D>
Src make_src(const GridDev &g, int n, const double *x, const double *A, const double *w, Workspace &ws,
             int32_t *labels, unsigned long long *gmom) {
    Src src{};
    src.g = g;
    src.gf = make_gridf(g);
    src.n = n;
    src.n_groups = (n + kGroup - 1) / kGroup;
    src.recs = ws.sorted ? ws.recs32s : ws.recs32;
    src.perm = ws.sorted ? ws.perm : nullptr;
    src.groups = ws.groups;
    src.x = x;
    src.A = A;
    src.w = w;
    src.gmom = gmom;
    src.labels = labels;
    src.sc = ws.sc;
    src.pairs_scored = ws.pairs_scored;
    return src;
}

// The long tile lists take a block past the shared memory a kernel gets unasked.
template <class F>
cudaError_t allow_tiles(F *kernel, int cap, unsigned bit, Workspace &ws) {
    if (cap <= kTileCap || (ws.attr_done & bit)) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)tile_bytes(kTileCapMax));
    if (e == cudaSuccess) ws.attr_done |= bit;
    return e;
}

template <int D>
cudaError_t launch_t(const GridDev &g, int n, const double *x, const double *A, const double *w, Workspace &ws,
                     int32_t *labels, unsigned long long *gmom, cudaStream_t st) {
    using G = Geom<D>;
    Src src = make_src<D>(g, n, x, A, w, ws, labels, gmom);
    constexpr int RL = D == 3 ? G::RZ : G::RY;
    const int toff = win_lo(g) / RL;
    const int tcount = (win_hi(g) - 1) / RL - toff + 1;
    const int nx = (g.res[0] + G::RX - 1) / G::RX;
    const int ny = D == 3 ? (g.res[1] + G::RY - 1) / G::RY : tcount;
    const long long blocks = (long long)nx * ny * (D == 3 ? tcount : 1);
    src.tile_cap = tile_cap(blocks, win_pixels(g), n, ws.sms);
    cudaError_t e = allow_tiles(assign_region_kernel<D>, src.tile_cap, D == 3 ? kAttrRegion3 : kAttrRegion2, ws);
    if (e != cudaSuccess) return e;
    e = record_scoring_start(ws, st);
    if (e != cudaSuccess) return e;
    assign_region_kernel<D><<<(unsigned)blocks, kThreads, tile_bytes(src.tile_cap), st>>>(src, nx, ny, toff);
    return cudaGetLastError();
}

}  // namespace

// Needs the groups' bounds, at most two groups per lane of a region's block (the
// Morton-sorted counts; beyond them the FP32 kernel streams the seeds) and axes
// whose indices are exact in FP32.
bool region_lists(const GridDev &g, int n, const Workspace &ws) {
    return ws.groups && (n + kGroup - 1) / kGroup <= kMaxGroups && g.res[0] < (1 << 23) && g.res[1] < (1 << 23) &&
           g.res[2] < (1 << 23);
}
// Thousands of seeds on grids of hardly more pixels than seeds go to the group-pruned FP32
// kernel (or the tensor-core lists): a tile's list is then longer than its pixels.
// MEASURED, us per call, regions / FP32 kernel: 2D n = 5000 on 100^2 1469 / 1335, n = 12000
// on 128^2 2148 / 1650; 3D n = 8300 on 20 x 17 x 16 3363 / 2324, n = 9000 on 28^3 1741 / 1434;
// and above the line 3D n = 5000 on 32^3 933 / 1056, n = 16000 on 48^3 1442 / 1892, with fewer
// seeds 2D n = 3000 on 80^2 768 / 1301.
bool region_form(const GridDev &g, int n, const Workspace &ws) {
    const bool crowded = n > 4096 && 2 * g.J < 5ll * n;
    return ws.prune && !crowded && region_lists(g, n, ws);
}

void region_dims(int dim, int (&r)[3]) {
    r[0] = dim == 3 ? Geom<3>::RX : Geom<2>::RX;
    r[1] = dim == 3 ? Geom<3>::RY : Geom<2>::RY;
    r[2] = dim == 3 ? Geom<3>::RZ : 1;
}

cudaError_t launch_assign_region(const GridDev &g, int n, const double *x, const double *A, const double *w,
                                 Workspace &ws, int32_t *labels, unsigned long long *moments, cudaStream_t st) {
    return g.dim == 3 ? launch_t<3>(g, n, x, A, w, ws, labels, moments, st)
                      : launch_t<2>(g, n, x, A, w, ws, labels, moments, st);
}

template <int D>
static cudaError_t masked_t(const GridDev &gc, const GridDev &gf, int r, int n, const double *x, const double *A,
                            const double *w, const uint8_t *mask, const int32_t *list, Workspace &ws,
                            unsigned long long *moments, cudaStream_t st) {
    using G = Geom<D>;
    Src src = make_src<D>(gf, n, x, A, w, ws, nullptr, moments);
    src.mask = mask;
    src.r = r;
    for (int a = 0; a < 3; ++a) src.cres[a] = gc.res[a];
    const int nx = (gf.res[0] + G::RX - 1) / G::RX, ny = (gf.res[1] + G::RY - 1) / G::RY;
    const long long all = (long long)nx * ny * (D == 3 ? (gf.res[2] + G::RZ - 1) / G::RZ : 1);
    src.tile_cap = tile_cap(all, gf.J, n, ws.sms);
    const long long resident = (long long)blocks_per_sm(src.tile_cap) * ws.sms;
    const int blocks = (int)(all < resident ? all : resident);
    const cudaError_t e = allow_tiles(masked_region_kernel<D>, src.tile_cap, D == 3 ? kAttrMasked3 : kAttrMasked2, ws);
    if (e != cudaSuccess) return e;
    masked_region_kernel<D><<<blocks, kThreads, tile_bytes(src.tile_cap), st>>>(src, nx, ny, list);
    return cudaGetLastError();
}

cudaError_t launch_masked_region(const GridDev &gc, const GridDev &gf, int r, int n, const double *x, const double *A,
                                 const double *w, const uint8_t *mask, const int32_t *list, Workspace &ws,
                                 unsigned long long *moments, cudaStream_t st) {
    return gf.dim == 3 ? masked_t<3>(gc, gf, r, n, x, A, w, mask, list, ws, moments, st)
                       : masked_t<2>(gc, gf, r, n, x, A, w, mask, list, ws, moments, st);
}

}  // namespace apd
