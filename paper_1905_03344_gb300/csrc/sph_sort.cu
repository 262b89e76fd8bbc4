// sph_sort.cu -- neighbour discovery, first half (Table 1 "Neighbour
// Discovery"; the paper's tree walk is replaced by a Morton-ordered cell
// grid): per-patch bounding box and largest h (FP64, ordered-integer
// atomics), grid parameters, Morton cell keys, a stable LSD radix sort of
// (key, slot), and the gather of every particle field into the sorted order,
// which also writes the cell table and the FP32 cell-relative records.
// Also the device-wide exclusive scan used by the CSR.
#include "sph_internal.cuh"

namespace sphg {

static inline int blocks_for(int64_t work, int threads, int sms, int per_sm)
{
    int64_t b = (work + threads - 1) / threads;
    int64_t cap = (int64_t)sms * per_sm;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

__device__ __forceinline__ unsigned long long umin64(unsigned long long a, unsigned long long b)
{
    return a < b ? a : b;
}
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b)
{
    return a > b ? a : b;
}

// ---------------------------------------------------------------------------
// A1a: per-patch min/max of x, y and max of h; one block per work item (a
// chunk of one patch), one atomic per block and value.  Min/max are exact,
// so the result does not depend on the order of the atomics.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_reduce_bbox(State s, const WorkItem* items, int nitems,
                                                     PatchRed* red)
{
    wait_before();
    __shared__ unsigned long long sh[5][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const WorkItem w = items[it];
        unsigned long long v[5] = {~0ull, ~0ull, 0ull, 0ull, 0ull};
#pragma unroll 4
        for (int64_t i = w.begin + threadIdx.x; i < w.end; i += blockDim.x) {
            unsigned long long a = ord_f64(s.x[i]), b = ord_f64(s.y[i]), c = ord_f64(s.h[i]);
            v[0] = umin64(v[0], a);
            v[1] = umin64(v[1], b);
            v[2] = umax64(v[2], a);
            v[3] = umax64(v[3], b);
            v[4] = umax64(v[4], c);
        }
        for (int o = 16; o > 0; o >>= 1) {
            v[0] = umin64(v[0], __shfl_xor_sync(0xffffffffu, v[0], o));
            v[1] = umin64(v[1], __shfl_xor_sync(0xffffffffu, v[1], o));
            v[2] = umax64(v[2], __shfl_xor_sync(0xffffffffu, v[2], o));
            v[3] = umax64(v[3], __shfl_xor_sync(0xffffffffu, v[3], o));
            v[4] = umax64(v[4], __shfl_xor_sync(0xffffffffu, v[4], o));
        }
        if (lane == 0)
            for (int q = 0; q < 5; q++) sh[q][warp] = v[q];
        __syncthreads();
        if (threadIdx.x == 0) {
            const int nw = blockDim.x >> 5;
            for (int ww = 1; ww < nw; ww++) {
                v[0] = umin64(v[0], sh[0][ww]);
                v[1] = umin64(v[1], sh[1][ww]);
                v[2] = umax64(v[2], sh[2][ww]);
                v[3] = umax64(v[3], sh[3][ww]);
                v[4] = umax64(v[4], sh[4][ww]);
            }
            PatchRed* r = red + w.patch;
            atomicMin(&r->xmin, v[0]);
            atomicMin(&r->ymin, v[1]);
            atomicMax(&r->xmax, v[2]);
            atomicMax(&r->ymax, v[3]);
            atomicMax(&r->hmax, v[4]);
        }
        __syncthreads();
    }
}

int launch_reduce_bbox(const Launch& L, const State& s, const WorkItem* items, int nitems,
                       PatchRed* red)
{
    if (nitems <= 0) return 0;
    int grid = nitems < L.sms * 8 ? nitems : L.sms * 8;
    launch_next(k_reduce_bbox, grid, 256, 0, L.stream, s, items, nitems, red);
    return 1;
}

// What a sort starts from: cleared reductions, radix counters and cell table,
// and an empty list pool for the search after it.  (Three memsets between the
// kernels, each as long as a small kernel, are gone with it: ten steps of 33^3
// mixed 2435 -> 2349 us, of 20^3 in FP64 3082 -> 3002 us.)
__global__ void __launch_bounds__(256) k_reset_red(int npatch, PatchRed* red, SortClear c)
{
    wait_before();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gs = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = p; k < c.words; k += gs) c.work[k] = 0u;
    for (int64_t k = p; k < c.cells; k += gs) c.cell[k] = make_uint4(0u, 0u, 0u, 0u);
    if (p < 2) c.pool_used[p] = 0ull;
    if (p < npatch) {
        red[p].xmin = ~0ull;
        red[p].ymin = ~0ull;
        red[p].xmax = 0ull;
        red[p].ymax = 0ull;
        red[p].hmax = 0ull;
        red[p].hcmin = ~0ull;
        for (int b = 0; b < kHBins; b++) red[p].hist[b] = 0u;
    }
}

// ---------------------------------------------------------------------------
// A1a': per patch, a histogram of h / h_max in kHBins bins (integer counts,
// so independent of the order of the atomics); it sets the class threshold.
// One atomic on shared memory per particle, one on the patch's bin per block.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_h_hist(State s, const WorkItem* items, int nitems, PatchRed* red)
{
    wait_before();
    __shared__ uint32_t hist[kHBins];
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const WorkItem w = items[it];
        for (int b = threadIdx.x; b < kHBins; b += blockDim.x) hist[b] = 0u;
        __syncthreads();
        const double hmax = unord_f64(red[w.patch].hmax);
        const double scale = hmax > 0.0 ? (double)kHBins / hmax : 0.0;
        const float scale_f = (float)scale;
        for (int64_t i0 = w.begin; i0 < w.end; i0 += blockDim.x) {
            const int64_t i = i0 + threadIdx.x;
            int b;
            if (i < w.end) {
                // the bin in FP32 where it is clear of the bins' edges (h is
                // at most h_max, so past the last edge it is the last bin)
                const double h = s.h[i];
                const float tf = f64_to_f32(h) * scale_f;
                b = (int)tf;
                const float fr = tf - (float)b;
                if (b >= kHBins - 1 && fr > 1e-4f) {
                    b = kHBins - 1;
                } else if (b > kHBins - 1) {
                    b = kHBins - 1;
                } else if (!(fr > 1e-4f && fr < 1.0f - 1e-4f)) {
                    const double t = h * scale;
                    b = t >= 0.0 && t < (double)kHBins ? (int)t : kHBins - 1;
                }
                atomicAdd(&hist[b], 1u);
            }
        }
        __syncthreads();
        for (int b = threadIdx.x; b < kHBins; b += blockDim.x)
            if (hist[b]) atomicAdd(&red[w.patch].hist[b], hist[b]);
        __syncthreads();
    }
}

int launch_h_hist(const Launch& L, const State& s, const WorkItem* items, int nitems, PatchRed* red)
{
    if (nitems <= 0) return 0;
    int grid = nitems < L.sms * 8 ? nitems : L.sms * 8;
    launch_next(k_h_hist, grid, 256, 0, L.stream, s, items, nitems, red);
    return 1;
}

int launch_reset_red(const Launch& L, int npatch, PatchRed* red, const SortClear& c)
{
    const int64_t most = c.words > c.cells ? c.words : c.cells;
    launch_next(k_reset_red, blocks_for(most > npatch ? most : npatch, 256, L.sms, 8), 256, 0, L.stream, npatch, red, c);
    return 1;
}

// ---------------------------------------------------------------------------
// A1b: grid of each patch.  Class threshold h_s: the upper edge of the
// lowest histogram bin above which at most 1/kBigShare of the patch lies (h_s
// = h_max, no big particles, when that edge is above 0.8 h_max).  Fine cell
// edge s = 2 h_s cell_factor (with margin), stencil half-extent K = 1 for
// cell_factor >= 1, 2 for >= 1/2, else 3, so K s >= 2 h_s; with K = 3 the
// edge is also at least min(h_s, kCellMed h_median).  Coarse cells are aligned blocks
// of 2^kc fine cells with 2^kc s >= 2 h_max, so the 3 x 3 x 3 coarse block
// around a particle holds every big particle that can reach it.  At most 128
// cells per axis and cell_cap fine + coarse cells per patch (s grows if not).
// Along z: ncz = floor(lz / s) cells of edge lz / ncz; when fewer than 2K+1,
// every z cell is visited once and the minimum image is taken in FP32.
// ---------------------------------------------------------------------------
__global__ void k_grid_params(int npatch, const PatchRed* red, PatchDev* pd, double cell_factor,
                              int* status, unsigned long long* vote)
{
    wait_before();
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < 2) vote[p] = 0ull;          // counted afresh by k_cell_hnb
    if (p >= npatch) return;
    PatchDev P = pd[p];
    const int K = stencil_k(cell_factor);
    double xmin = 0, ymin = 0, xmax = 0, ymax = 0, hmax = 0;
    const int64_t np = P.end - P.begin;
    if (np > 0) {
        xmin = unord_f64(red[p].xmin);
        ymin = unord_f64(red[p].ymin);
        xmax = unord_f64(red[p].xmax);
        ymax = unord_f64(red[p].ymax);
        hmax = unord_f64(red[p].hmax);
    }
    double ex = xmax - xmin, ey = ymax - ymin;
    if (!isfinite(ex) || !isfinite(ey) || !isfinite(hmax) || !isfinite(xmin) || !isfinite(ymin)) {
        // non-finite positions: flag, and keep a one-cell grid so that every
        // index computed from it stays inside the cell table
        atomicOr(status, kStNonFinite);
        xmin = ymin = 0.0;
        ex = ey = 0.0;
        hmax = 0.0;
    }
    // class threshold from the histogram of h / h_max
    double hs = hmax;
    {
        const int64_t allow = np / kBigShare;
        int64_t above = 0;
        int b = kHBins - 1;
        while (b > 0 && above + (int64_t)red[p].hist[b] <= allow) {
            above += red[p].hist[b];
            b--;
        }
        const double edge = hmax * (double)(b + 1) / (double)kHBins;
        if (edge < 0.8 * hmax) hs = edge;
    }
    double s = 2.0 * hs * cell_factor * kCellMargin;
    // the median of h, from the histogram, to a bin
    double hmed = hmax;
    {
        int64_t acc = 0;
        for (int b = 0; b < kHBins; b++) {
            acc += red[p].hist[b];
            if (2 * acc >= np) {
                hmed = hmax * ((double)b + 0.5) / (double)kHBins;
                break;
            }
        }
    }
    if (K == 3) {
        // the stencil reaches 3 cells, so cells may be finer than h_s: as
        // fine as 2 h_s cell_factor, but not below min(h_s, kCellMed h_med),
        // the edge that served the interior particles best.  With a narrow
        // spread of h this is the h_s-sized cell of cell_factor 1/2.
        const double sm = fmin(hs, kCellMed * hmed) * kCellMargin;
        if (s < sm) s = sm;
    }
    const double sext = fmax(ex, ey) / (double)(kMaxCellsAxis - 1) * kCellMargin;
    if (s < sext) s = sext;
    if (!(s > 0.0)) s = P.lz > 0.0 ? P.lz : 1.0;
    int64_t ncx = 1, ncy = 1, ncz = 1, ncxc = 1, ncyc = 1, nczc = 1;
    int kc = 0;
    bool fits = false;
    for (int iter = 0; iter < 200 && !fits; iter++) {
        ncx = (int64_t)floor(ex / s) + 1;
        ncy = (int64_t)floor(ey / s) + 1;
        ncz = (int64_t)floor(P.lz / s);
        if (ncz < 1) ncz = 1;
        if (ncz > kMaxCellsAxis) ncz = kMaxCellsAxis;
        kc = 0;
        if (hs < hmax) {
            while (kc < kMortonBits && (double)(1 << kc) * s < 2.0 * hmax * kCellMargin) kc++;
            // whole coarse cells along the period (a partial one would let a big
            // particle two coarse cells away across the wrap reach the block)
            if (ncz >= (1 << kc)) ncz = (ncz >> kc) << kc;
        } else {
            kc = kMortonBits;   // no big particles: one (empty) coarse cell
        }
        ncxc = (ncx + (1 << kc) - 1) >> kc;
        ncyc = (ncy + (1 << kc) - 1) >> kc;
        nczc = (ncz + (1 << kc) - 1) >> kc;
        fits = ncx <= kMaxCellsAxis && ncy <= kMaxCellsAxis && ncx * ncy * ncz + ncxc * ncyc * nczc <= P.cell_cap;
        if (!fits) s *= 1.25;
    }
    if (!fits || ncx < 1 || ncy < 1) {
        atomicOr(status, kStNonFinite);
        ncx = ncy = ncz = ncxc = ncyc = nczc = 1;
        kc = 0;
    }
    P.xmin = xmin;
    P.ymin = ymin;
    P.hmax = hmax;
    P.s = s;
    P.sz = P.lz / (double)ncz;
    P.ncx = (int)ncx;
    P.ncy = (int)ncy;
    P.ncz = (int)ncz;
    P.K = K;
    P.zmode = ncz >= 2 * K + 1 ? 0 : 1;
    P.s_f = (float)s;
    P.sz_f = (float)P.sz;
    P.lz_f = (float)P.lz;
    P.inv_s_f = (float)(1.0 / s);
    P.inv_sz_f = (float)(1.0 / P.sz);
    P.hmax_f = (float)hmax;
    P.hlz = 0.5 * P.lz;
    P.hsz = 0.5 * P.sz;
    P.hs = hs;
    P.hs_f = (float)hs;
    P.hmed = hmed;
    P.nbig = 0;
    P.row_fill = 0;
    P.row_inset = 0;
    P.h_spread = 0;
    P.kc = kc;
    P.ncxc = (int)ncxc;
    P.ncyc = (int)ncyc;
    P.nczc = (int)nczc;
    P.zmode_c = nczc >= 3 ? 0 : 1;
    P.coarse_base = P.cell_base + ncx * ncy * ncz;
    pd[p] = P;
}

int launch_grid_params(const Launch& L, int npatch, const PatchRed* red, PatchDev* pd,
                       double cell_factor, int* status, unsigned long long* vote)
{
    launch_next(k_grid_params, (npatch + 127) / 128, 128, 0, L.stream, npatch, red, pd, cell_factor, status, vote);
    return 1;
}

// ---------------------------------------------------------------------------
// A1c: key = patch << 22 | big << 21 | Morton(cx, cy, cz), big = (h > h_s),
// cell coordinates in FP32 from the FP64 offset to the grid origin (error <
// 1e-4 cell, inside the margin).  Counts the big particles of each patch.
// ---------------------------------------------------------------------------
// Also counts the digits of every pass of the radix sort (hist, kRsMaxPasses
// x 256).
__device__ __forceinline__ void count_digits(uint32_t key, int passes, uint32_t (*sh)[256])
{
    for (int p = 0; p < passes; p++) atomicAdd(&sh[p][(key >> (8 * p)) & 255u], 1u);
}

__device__ __forceinline__ void add_digits(int passes, const uint32_t (*sh)[256], uint32_t* hist)
{
    for (int k = threadIdx.x; k < passes * 256; k += blockDim.x) {
        const uint32_t c = (&sh[0][0])[k];
        if (c) atomicAdd(&hist[k], c);
    }
}

__global__ void __launch_bounds__(256) k_keys(int64_t n, State s, const uint16_t* patch_of,
                                              PatchDev* pd, uint32_t* keys, uint32_t* vals, int passes, uint32_t* hist)
{
    wait_before();
    __shared__ uint32_t sh[kRsMaxPasses][256];
    for (int k = threadIdx.x; k < kRsMaxPasses * 256; k += blockDim.x) (&sh[0][0])[k] = 0u;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int p = patch_of[i];
        PatchDev* P = pd + p;
        const bool big = above(s.h[i], P->hs);
        // one atomic per warp and patch: the lanes of a warp that share the
        // patch add their big particles together
        const unsigned act = __activemask();
        const unsigned peers = __match_any_sync(act, p);
        const unsigned bigs = __ballot_sync(act, big) & peers;
        if (bigs && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&P->nbig, __popc(bigs));
        const float tx = f64_to_f32(s.x[i] - P->xmin) * P->inv_s_f;
        const float ty = f64_to_f32(s.y[i] - P->ymin) * P->inv_s_f;
        const float tz = f64_to_f32(s.z[i] + P->hlz) * P->inv_sz_f;
        int cx = (int)floorf(tx), cy = (int)floorf(ty), cz = (int)floorf(tz);
        cx = min(max(cx, 0), P->ncx - 1);
        cy = min(max(cy, 0), P->ncy - 1);
        cz = min(max(cz, 0), P->ncz - 1);
        const uint32_t key = ((uint32_t)p << kPatchShift) | ((uint32_t)big << kClassShift) | part1by2((uint32_t)cx) |
                             (part1by2((uint32_t)cy) << 1) | (part1by2((uint32_t)cz) << 2);
        keys[i] = key;
        vals[i] = (uint32_t)i;
        count_digits(key, passes, sh);
    }
    __syncthreads();
    add_digits(passes, sh, hist);
}

int launch_keys(const Launch& L, int64_t n, const State& s, const uint16_t* patch_of,
                PatchDev* pd, const RadixSort& rs, int passes)
{
    if (n <= 0) return 0;
    uint32_t *k, *v;
    rs.input(passes, k, v);
    launch_next(k_keys, blocks_for(n, 256, L.sms, 8), 256, 0, L.stream, n, s, patch_of, pd, k, v, passes, rs.work);
    return 1;
}

// ---------------------------------------------------------------------------
// Block-wide exclusive scan helpers (blockDim.x a multiple of 32, <= 1024).
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v)
{
    const int lane = threadIdx.x & 31;
    for (int o = 1; o < 32; o <<= 1) {
        T t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// returns the exclusive prefix of v over the block; *total receives the sum
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T* total, T* sh /* >= 33 */)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T inc = warp_incl_scan(v);
    if (lane == 31) sh[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nw ? sh[lane] : T(0);
        T wi = warp_incl_scan(w);
        if (lane < nw) sh[lane] = wi - w;
        if (lane == 31) sh[32] = wi;
    }
    __syncthreads();
    T res = inc - v + sh[warp];
    *total = sh[32];
    __syncthreads();
    return res;
}

// ---------------------------------------------------------------------------
// Device-wide exclusive scan, reduce-then-scan in three launches.
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

template <typename Tin, typename Tout>
__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const Tin* in, int64_t n, Tout* part)
{
    __shared__ Tout sh[33];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    Tout v = 0;
    for (int k = 0; k < kScanItems; k++) {
        int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
        if (i < n) v += (Tout)in[i];
    }
    Tout tot;
    block_excl_scan<Tout>(v, &tot, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

template <typename Tout>
__global__ void __launch_bounds__(1024) k_scan_spine(Tout* part, int64_t nb)
{
    __shared__ Tout sh[33];
    Tout carry = 0;
    for (int64_t base = 0; base < nb; base += blockDim.x) {
        int64_t i = base + threadIdx.x;
        Tout v = i < nb ? part[i] : Tout(0);
        Tout tot;
        Tout ex = block_excl_scan<Tout>(v, &tot, sh);
        if (i < nb) part[i] = ex + carry;
        carry += tot;
    }
}

template <typename Tin, typename Tout>
__global__ void __launch_bounds__(kScanThreads) k_scan_down(const Tin* in, int64_t n, const Tout* part,
                                                           Tout* out, int write_total)
{
    __shared__ Tout sh[33];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    Tout loc[kScanItems];
    Tout sum = 0;
    for (int k = 0; k < kScanItems; k++) {
        int64_t i = base + k;
        Tout v = i < n ? (Tout)in[i] : Tout(0);
        loc[k] = sum;
        sum += v;
    }
    Tout tot;
    Tout ex = block_excl_scan<Tout>(sum, &tot, sh) + part[blockIdx.x];
    for (int k = 0; k < kScanItems; k++) {
        int64_t i = base + k;
        if (i < n) out[i] = ex + loc[k];
    }
    if (write_total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = part[blockIdx.x] + tot;
}

int64_t scan_tmp_words(int64_t n) { return (n + kScanTile - 1) / kScanTile + 1; }

int launch_scan_u32_to_u64(const Launch& L, int64_t n, const uint32_t* in, uint64_t* out, uint64_t* tmp)
{
    if (n <= 0) {
        cudaMemsetAsync(out, 0, sizeof(uint64_t), L.stream);
        return 0;
    }
    const int64_t nb = (n + kScanTile - 1) / kScanTile;
    k_scan_reduce<uint32_t, uint64_t><<<(unsigned)nb, kScanThreads, 0, L.stream>>>(in, n, tmp);
    k_scan_spine<uint64_t><<<1, 1024, 0, L.stream>>>(tmp, nb);
    k_scan_down<uint32_t, uint64_t><<<(unsigned)nb, kScanThreads, 0, L.stream>>>(in, n, tmp, out, 1);
    return 3;
}

// ---------------------------------------------------------------------------
// Stable LSD radix sort, 8-bit digits, one kernel per pass, after Adinets and
// Merrill, "Onesweep: a faster least significant digit radix sort for GPUs",
// 2022, with the decoupled look-back of Merrill and Garland, "Single-pass
// parallel prefix scan with decoupled look-back", 2016.  The digits of all
// passes are counted while the keys are made.  A block takes the next
// tile (in the order of a ticket), ranks its keys stably (warp match +
// per-warp counters, warps in tile order), publishes the tile's digit counts
// and looks back over the tiles before it for their sum, each of which is
// published as its own counts first and as the sum up to it once that is
// known; then it stages the tile in shared memory in digit order and writes
// each digit run contiguously.  A tile only waits for tiles with earlier
// tickets, which never wait for it.  The wait is bounded all the same; a
// block whose wait runs out flags it and writes nothing out of range.
//
// A pass is bound by the latency of a tile's chain (load, rank, look back,
// stage, write), so by how many tiles are resident: five blocks on an SM with
// 12 keys a thread, 48 registers and 35 KB; 16 keys at 128 registers, two
// blocks, took 100 us a pass at 8 M where this takes 72, votes per digit bit
// in place of the match 75, 8 keys 73.  Up to 622,592 keys (four tiles on each
// of 152 SMs) the tiles have 1024 keys, which keeps more SMs busy.  The pass per digit of
// a histogram, a three-kernel scan and a scatter (with a copy back after an
// odd number of passes) that this replaces took 15 launches where this takes
// 3: 460 -> 216 us at 8 M, 126 -> 51 us at 1 M, 102 -> 21 us at 8000.
// ---------------------------------------------------------------------------
constexpr int kRsThreads = 256;
constexpr int kRsWarps = kRsThreads / 32;
constexpr uint32_t kRsAggregate = 1u << 30, kRsPrefix = 2u << 30, kRsValue = kRsAggregate - 1u;
constexpr int kRsSpins = 1 << 22;
constexpr int kRsItems = 12;            // keys a thread takes in the larger tiles

template <int ITEMS>
__global__ void __launch_bounds__(kRsThreads, ITEMS == 4 ? 6 : 5) k_rs_pass(const uint32_t* kin,
        const uint32_t* vin, int64_t n, int shift, const uint32_t* ghist, uint32_t* ticket,
        volatile uint32_t* state, uint32_t* kout, uint32_t* vout, int* status)
{
    wait_before();
    constexpr int kTile = kRsThreads * ITEMS;
    __shared__ uint32_t s_keys[kTile];
    __shared__ uint32_t s_vals[kTile];
    __shared__ uint32_t s_wcnt[kRsWarps][256];
    __shared__ uint32_t s_dstart[256];
    __shared__ uint32_t s_goff[256];
    __shared__ uint32_t s_scan[33];
    __shared__ uint32_t s_tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
    for (int k = threadIdx.x; k < kRsWarps * 256; k += kRsThreads) (&s_wcnt[0][0])[k] = 0;
    __syncthreads();
    const int64_t tile = s_tile;
    const int64_t wbase = tile * kTile + (int64_t)warp * 32 * ITEMS;
    uint32_t kr[ITEMS], vr[ITEMS];
    uint16_t pr[ITEMS];
#pragma unroll
    for (int t = 0; t < ITEMS; t++) {
        const int64_t i = wbase + t * 32 + lane;
        kr[t] = i < n ? kin[i] : 0xffffffffu;
        vr[t] = i < n ? vin[i] : 0u;
    }
#pragma unroll
    for (int t = 0; t < ITEMS; t++) {
        const bool valid = wbase + t * 32 + lane < n;
        const uint32_t d = valid ? ((kr[t] >> shift) & 255u) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        uint32_t before = 0;
        if (valid) before = s_wcnt[warp][d];
        __syncwarp();
        if (valid && rank == 0) s_wcnt[warp][d] = before + (uint32_t)__popc(peers);
        __syncwarp();
        pr[t] = (uint16_t)(before + rank);
    }
    __syncthreads();
    {   // per digit: exclusive offsets of the warps, digit starts in the tile and in the output
        const int d = threadIdx.x;
        uint32_t cnt = 0;
        for (int w = 0; w < kRsWarps; w++) {
            const uint32_t c = s_wcnt[w][d];
            s_wcnt[w][d] = cnt;
            cnt += c;
        }
        volatile uint32_t* mine = state + tile * 256 + d;
        *mine = cnt | (tile == 0 ? kRsPrefix : kRsAggregate);
        uint32_t tot;
        const uint32_t start = block_excl_scan<uint32_t>(cnt, &tot, s_scan);
        const uint32_t first = block_excl_scan<uint32_t>(ghist[d], &tot, s_scan);
        // eight tiles back at a time (their loads are in flight together)
        uint32_t before = 0;
        int spins = 0;
        for (int64_t q = tile - 1; q >= 0;) {
            uint32_t v[8];
#pragma unroll
            for (int e = 0; e < 8; e++) v[e] = q - e >= 0 ? state[(q - e) * 256 + d] : 0u + kRsPrefix;
            int used = 0;
#pragma unroll
            for (int e = 0; e < 8; e++)
                if (used == e && v[e] >= kRsAggregate) {
                    before += v[e] & kRsValue;
                    used = v[e] >= kRsPrefix ? 64 : e + 1;
                }
            if (used >= 64) break;
            q -= used;
            if (used == 0 && ++spins > kRsSpins) {
                atomicOr(status, kStTimeout);
                break;
            }
        }
        if (tile > 0) *mine = (before + cnt) | kRsPrefix;
        s_dstart[d] = start;
        s_goff[d] = first + before - start;
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < ITEMS; t++) {
        if (wbase + t * 32 + lane < n) {
            const uint32_t d = (kr[t] >> shift) & 255u;
            const uint32_t lp = s_dstart[d] + s_wcnt[warp][d] + pr[t];
            s_keys[lp] = kr[t];
            s_vals[lp] = vr[t];
        }
    }
    __syncthreads();
    const int64_t rem = n - tile * kTile;
    const int tn = rem < kTile ? (int)rem : kTile;
    for (int k = threadIdx.x; k < tn; k += kRsThreads) {
        const uint32_t key = s_keys[k];
        const uint32_t g = s_goff[(key >> shift) & 255u] + (uint32_t)k;
        if (g < (uint32_t)n) {
            kout[g] = key;
            vout[g] = s_vals[k];
        }
    }
}

static int rs_items(int64_t n) { return n <= 608 * 1024 ? 4 : kRsItems; }
static int64_t rs_tiles(int64_t n) { return (n + rs_items(n) * kRsThreads - 1) / (rs_items(n) * kRsThreads); }

size_t radix_work_words(int64_t n) { return (size_t)kRsMaxPasses * (256 + 16 + 256 * (size_t)rs_tiles(n < 1 ? 1 : n)); }

size_t radix_work_capacity(int64_t cap)
{
    const size_t a = radix_work_words(cap), b = radix_work_words(cap < 608 * 1024 ? cap : 608 * 1024);
    return a > b ? a : b;
}

int launch_radix_sort(const Launch& L, int64_t n, int passes, const RadixSort& rs, int* status)
{
    if (n <= 0) return 0;
    uint32_t *ki, *vi;
    rs.input(passes, ki, vi);
    const int64_t tiles = rs_tiles(n);
    // the default split of the L1 would keep fewer blocks on an SM
    cudaFuncSetAttribute(k_rs_pass<4>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    cudaFuncSetAttribute(k_rs_pass<kRsItems>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    for (int ps = 0; ps < passes; ps++) {
        uint32_t* ko = ki == rs.keys ? rs.keys_alt : rs.keys;
        uint32_t* vo = vi == rs.vals ? rs.vals_alt : rs.vals;
        uint32_t* tickets = rs.work + kRsMaxPasses * 256;
        uint32_t* state = tickets + kRsMaxPasses * 16 + (int64_t)ps * 256 * tiles;
        const auto kern = rs_items(n) == 4 ? k_rs_pass<4> : k_rs_pass<kRsItems>;
        launch_next(kern, (unsigned)tiles, kRsThreads, 0, L.stream, ki, vi, n, 8 * ps, rs.work + 256 * ps, tickets + 16 * ps,
                    state, ko, vo, status);
        ki = ko;
        vi = vo;
    }
    return passes;
}

// ---------------------------------------------------------------------------
// Row-length bins of the pair sums: key = octave of |N(i)|, sorted stably by
// one radix pass; the bin starts are the scanned digit counts.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_octave_keys(int64_t n, const uint32_t* cnt, uint32_t* keys, uint32_t* vals, uint32_t* hist)
{
    __shared__ uint32_t sh[1][256];
    sh[0][threadIdx.x] = 0u;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t c = cnt[i];
        // 0 for an empty row, else 1 + ceil(log2 c) (32 - clz(c - 1) = ceil(log2 c))
        const int o = c == 0u ? 0 : 33 - __clz(c - 1u);
        const uint32_t key = (uint32_t)min(o, kPairOctaves - 1);
        keys[i] = key;
        vals[i] = (uint32_t)i;
        count_digits(key, 1, sh);
    }
    __syncthreads();
    add_digits(1, sh, hist);
}

__global__ void k_octave_bounds(const uint32_t* hist, int64_t n, uint32_t* bounds)
{
    const int o = threadIdx.x;
    const uint32_t c = o < kPairOctaves ? hist[o] : 0u;
    const uint32_t inc = warp_incl_scan(c);
    if (o <= kPairOctaves) bounds[o] = o < kPairOctaves ? inc - c : (uint32_t)n;
}

int launch_pair_bins(const Launch& L, int64_t n, const uint32_t* cnt, const RadixSort& rs, uint32_t* bounds, int* status)
{
    if (n <= 0) return 0;
    cudaMemsetAsync(rs.work, 0, radix_work_words(n) * sizeof(uint32_t), L.stream);
    uint32_t *k, *v;
    rs.input(1, k, v);
    k_octave_keys<<<blocks_for(n, 256, L.sms, 8), 256, 0, L.stream>>>(n, cnt, k, v, rs.work);
    const int launches = 1 + launch_radix_sort(L, n, 1, rs, status);
    k_octave_bounds<<<1, 32, 0, L.stream>>>(rs.work, n, bounds);
    return launches + 1;
}

// ---------------------------------------------------------------------------
// Gather every field into sorted order, write the permutation, the
// cell table (start/end by key boundaries, largest h per cell) and the FP32
// records with positions relative to the particle's cell origin.  Also forms
// the time-centred velocity v_{n-1/2} + a_{n-1} dt_{n-1}/2 used by the
// viscosity and the energy equation.
// ---------------------------------------------------------------------------
// the FP32 records of sorted slot k in cell (cx, cy, cz) of patch P: offsets
// from the cell origin, 4 hq^2 (hq: the h of the search), and for
// the pair sums the mass, the time-centred velocity v + a_{n-1} dt_{n-1}/2
// and 1/(2h) (mixed), or the same in FP64.  The z offset is taken from the
// image of z nearest the cell's centre: a particle that has left its cell
// since the sort (reused lists) may have crossed the periodic z boundary, and
// the pair separation, which wraps at most once, needs every offset within
// about a cell of its cell.  A particle inside its cell is its own nearest
// image, so this changes nothing right after a sort.
__device__ __forceinline__ void write_records(int64_t k, const PatchDev* P, uint32_t cx, uint32_t cy, uint32_t cz,
                                              double x, double y, double z, double vx, double vy, double vz,
                                              double m, double h, double u, double axp, double ayp, double azp,
                                              float hq, Recs& r, Fp64& f, int mixed, int kernel)
{
    const float ox = f64_to_f32(x - fma(small_to_f64(cx), P->s, P->xmin));
    const float oy = f64_to_f32(y - fma(small_to_f64(cy), P->s, P->ymin));
    double ozd = z - fma(small_to_f64(cz), P->sz, -P->hlz);
    const double oc = ozd - P->hsz;
    if (above(oc, P->hlz)) ozd -= P->lz;
    else if (below_neg(oc, P->hlz)) ozd += P->lz;
    const float oz = f64_to_f32(ozd);
    const float hf = f64_to_f32(h);
    r.r4[k] = make_float4(ox, oy, oz, 4.0f * hq * hq);
    const double half = P->step > 0 ? 0.5 * P->dt_prev : 0.0;
    const double vhx = vx + axp * half, vhy = vy + ayp * half, vhz = vz + azp * half;
    if (mixed) {
        r.r5[k] = make_float4(ox, oy, oz, f64_to_f32(m));
        r.rv[k] = make_float4(f64_to_f32(vhx), f64_to_f32(vhy), f64_to_f32(vhz), 0.5f / hf);
        r.uf[k] = f64_to_f32(u);
    } else {
        f.vhx[k] = vhx;
        f.vhy[k] = vhy;
        f.vhz[k] = vhz;
        const double w = 0.5 / h;
        const double w5 = w * w * w * w * w;
        f.w[k] = w;
        if (kernel == SPH_KERNEL_WENDLAND) {
            const double g0 = cbrt(w5);
            f.g0[k] = g0;
            f.g1[k] = g0 * w;
        } else {
            f.g0[k] = w5;
            f.g1[k] = w;
        }
    }
}

__global__ void __launch_bounds__(256) k_gather(int64_t n, const uint32_t* skeys, const uint32_t* svals,
                                                State src, State dst, const uint32_t* perm_src,
                                                uint32_t* perm_dst, const PatchDev* pd, Grid g,
                                                Recs r, Fp64 f, int mixed, int kernel, RowHint hint,
                                                const double* hsearch, double* hsearch_out, const int* status)
{
    wait_before();
    const bool have_hint = *hint.valid != 0;
    // a sort whose wait ran out: the particles keep their order, and the step
    // ends with its status
    if (*status & kStTimeout) {
        const double* from[13] = {src.x, src.y, src.z, src.vx, src.vy, src.vz, src.m, src.h, src.u, src.du_prev, src.axp, src.ayp, src.azp};
        double* to[13] = {dst.x, dst.y, dst.z, dst.vx, dst.vy, dst.vz, dst.m, dst.h, dst.u, dst.du_prev, dst.axp, dst.ayp, dst.azp};
        for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
            for (int q = 0; q < 13; q++) to[q][k] = from[q][k];
            perm_dst[k] = perm_src[k];
        }
        return;
    }
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t key = skeys[k];
        const uint32_t si = svals[k];
        const PatchDev* P = pd + (key >> kPatchShift);
        const double x = src.x[si], y = src.y[si], z = src.z[si];
        const double vx = src.vx[si], vy = src.vy[si], vz = src.vz[si];
        const double m = src.m[si], h = src.h[si];
        const double axp = src.axp[si], ayp = src.ayp[si], azp = src.azp[si];
        dst.x[k] = x; dst.y[k] = y; dst.z[k] = z;
        dst.vx[k] = vx; dst.vy[k] = vy; dst.vz[k] = vz;
        dst.m[k] = m; dst.h[k] = h;
        dst.u[k] = src.u[si];
        dst.du_prev[k] = src.du_prev[si];
        dst.axp[k] = axp; dst.ayp[k] = ayp; dst.azp[k] = azp;
        perm_dst[k] = perm_src[si];
        hint.rowcap[k] = have_hint ? hint.cnt_prev[si] : kNoHint;

        const uint32_t mort = key & kMortonMask;
        const bool big = (key >> kClassShift) & 1u;
        const uint32_t cx = compact1by2(mort), cy = compact1by2(mort >> 1), cz = compact1by2(mort >> 2);
        g.cellxyz[k] = cx | (cy << 8) | (cz << 16);
        // h of the search
        const float hf = f64_to_f32(hsearch ? hsearch[si] : h);
        if (hsearch_out) hsearch_out[k] = hsearch[si];
        write_records(k, P, cx, cy, cz, x, y, z, vx, vy, vz, m, h, dst.u[k], axp, ayp, azp, hf, r, f, mixed, kernel);
        if (!big) {
            // fine cell of small particles: bounded by a change of key
            const int64_t lin = P->cell_base + ((int64_t)cz * P->ncy + cy) * P->ncx + cx;
            if (k == P->begin || skeys[k - 1] != key) g.cell[lin].x = (uint32_t)k;
            if (k + 1 == P->end || skeys[k + 1] != key) g.cell[lin].y = (uint32_t)(k + 1);
            atomicMax(&g.cell[lin].z, __float_as_uint(hf));
        } else {
            // coarse cell of big particles: an aligned block of 2^kc fine cells,
            // contiguous in Morton order, bounded by a change of key >> 3 kc
            const int kc = P->kc;
            const int64_t lin = P->coarse_base +
                                ((int64_t)(cz >> kc) * P->ncyc + (cy >> kc)) * P->ncxc + (cx >> kc);
            const uint32_t pre = key >> (3 * kc);
            if (k == P->begin || (skeys[k - 1] >> (3 * kc)) != pre) g.cell[lin].x = (uint32_t)k;
            if (k + 1 == P->end || (skeys[k + 1] >> (3 * kc)) != pre) g.cell[lin].y = (uint32_t)(k + 1);
            atomicMax(&g.cell[lin].z, __float_as_uint(hf));
        }
    }
}

int launch_gather(const Launch& L, int64_t n, const uint32_t* skeys, const uint32_t* svals,
                  const State& src, const State& dst, const uint32_t* perm_src, uint32_t* perm_dst,
                  const PatchDev* pd, const Grid& g, const Recs& r, const Fp64& f, int mixed, int kernel,
                  const RowHint& hint, const int* status, const double* hsearch, double* hsearch_out)
{
    if (n <= 0) return 0;
    launch_next(k_gather, blocks_for(n, 256, L.sms, 16), 256, 0, L.stream, n, skeys, svals, src, dst, perm_src, perm_dst,
                pd, g, r, f, mixed, kernel, hint, hsearch, hsearch_out, status);
    return 1;
}

// records of the current state without a sort (between rebuilds of a reused
// candidate superset): the grid and cells of the last sort, the current
// positions, h and time state
__global__ void __launch_bounds__(256) k_refresh_records(int64_t n, State s, const uint16_t* patch_of,
                                                         const PatchDev* pd, const uint32_t* cellxyz, Recs r,
                                                         Fp64 f, int mixed, int kernel)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const PatchDev* P = pd + patch_of[k];
        const uint32_t c = cellxyz[k];
        const double h = s.h[k];
        write_records(k, P, c & 255u, (c >> 8) & 255u, c >> 16, s.x[k], s.y[k], s.z[k], s.vx[k], s.vy[k], s.vz[k],
                      s.m[k], h, s.u[k], s.axp[k], s.ayp[k], s.azp[k], (float)h, r, f, mixed, kernel);
    }
}

int launch_refresh_records(const Launch& L, int64_t n, const State& s, const uint16_t* patch_of,
                           const PatchDev* pd, const uint32_t* cellxyz, const Recs& r, const Fp64& f, int mixed, int kernel)
{
    if (n <= 0) return 0;
    k_refresh_records<<<blocks_for(n, 256, L.sms, 16), 256, 0, L.stream>>>(n, s, patch_of, pd, cellxyz, r, f,
                                                                          mixed, kernel);
    return 1;
}

// ---------------------------------------------------------------------------
// The row copy of the small particles' search records (see Grid): one warp
// per row of fine cells, which reserves the row's slots (where in the copy a
// row lies depends on scheduling, its contents do not), scans the cells'
// counts and copies their particles: 36 bytes a particle, 0.15 ms at 8 M
// (0.13 without the boxes).  The warp also leaves, over K cells to each side of
// every cell, the row's largest h in hnb_x and where its particles lie in y and
// z in row_box, and each cell's tight box in its record.  blockIdx.y is the
// patch.
// ---------------------------------------------------------------------------
// a distance from a face of the cell, in 1/255 of the edge, as an inset of a
// cell's box, rounded down
__device__ __forceinline__ uint32_t box_inset(float d255)
{
    return min(__float2uint_rd(fmaxf(d255, 0.0f) * ((float)kBoxQ / 255.0f)), (uint32_t)kBoxQ - 1u);
}

__global__ void __launch_bounds__(256) k_cell_rows(PatchDev* pd, Grid g, const float4* r4, int K, float* hnb_x)
{
    wait_before();
    constexpr int kPad = 4;             // at least K
    __shared__ float sh[8][kMaxCellsAxis + 2 * kPad];
    __shared__ uint32_t box[8][kMaxCellsAxis + 2 * kPad];
    PatchDev* P = pd + blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ncx = P->ncx, nrows = P->ncy * P->ncz;
    const float s_f = P->s_f, qy = 255.0f * P->inv_s_f, qz = 255.0f * P->inv_sz_f;
    const uint32_t first = (uint32_t)P->begin;
    for (int r = (int)blockIdx.x * 8 + warp; r < nrows; r += (int)gridDim.x * 8) {
        const int64_t lin = P->cell_base + (int64_t)r * ncx;
        // at most kMaxCellsAxis cells: four per lane, 32 apart
        uint32_t beg[4], off[4], cnt[4], tot = 0;
        if (lane < kPad) {
            sh[warp][lane] = sh[warp][kPad + ncx + lane] = 0.0f;
            box[warp][lane] = box[warp][kPad + ncx + lane] = ~0u;
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int x = k * 32 + lane;
            beg[k] = cnt[k] = off[k] = 0;
            if (k * 32 < ncx) {
                if (x < ncx) {
                    const uint4 c = g.cell[lin + x];
                    beg[k] = c.x;
                    cnt[k] = c.y - c.x;
                    sh[warp][kPad + x] = __uint_as_float(c.z);
                }
                uint32_t inc = cnt[k];
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += t;
                }
                off[k] = tot + inc - cnt[k];
                tot += __shfl_sync(0xffffffffu, inc, 31);
            }
        }
        uint32_t base = 0;
        if (lane == 0 && tot) base = first + atomicAdd(&P->row_fill, tot);
        base = __shfl_sync(0xffffffffu, base, 0);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int x = k * 32 + lane;
            if (x >= ncx) continue;
            const uint32_t b = base + off[k];
            g.row[lin + x] = make_uint2(b, b + cnt[k]);
            float m = 0.0f;
            for (int d = -K; d <= K; d++) m = fmaxf(m, sh[warp][kPad + x + d]);
            hnb_x[lin + x] = m;
            float xlo = 255.0f, xhi = 0.0f, ylo = 255.0f, yhi = 0.0f, zlo = 255.0f, zhi = 0.0f;
            for (uint32_t u = 0; u < cnt[k]; u++) {
                const uint32_t j = beg[k] + u;
                const float4 q = r4[j];
                xlo = fminf(xlo, q.x * qy);
                xhi = fmaxf(xhi, q.x * qy);
                ylo = fminf(ylo, q.y * qy);
                yhi = fmaxf(yhi, q.y * qy);
                zlo = fminf(zlo, q.z * qz);
                zhi = fmaxf(zhi, q.z * qz);
                g.row_rec[b + u] = make_float4(fmaf((float)x, s_f, q.x), q.y, q.z, q.w);
                g.row_id[b + u] = j | ((uint32_t)x << kColBits);
            }
            if (cnt[k])
                g.cell[lin + x].w = box_inset(xlo) | box_inset(255.0f - xhi) << 5 | box_inset(ylo) << 10 |
                                    box_inset(255.0f - yhi) << 15 | box_inset(zlo) << 20 | box_inset(255.0f - zhi) << 25;
            // rounded outwards (no particle: all ones, which any other undercuts)
            box[warp][kPad + x] = cnt[k] == 0 ? ~0u
                : __float2uint_rd(fmaxf(ylo, 0.0f)) | __float2uint_rd(fmaxf(255.0f - yhi, 0.0f)) << 8 |
                  __float2uint_rd(fmaxf(zlo, 0.0f)) << 16 | __float2uint_rd(fmaxf(255.0f - zhi, 0.0f)) << 24;
        }
        __syncwarp();
        uint32_t inset = 0, nbox = 0;
        for (int x = lane; x < ncx; x += 32) {
            uint32_t m = ~0u;
            for (int d = -K; d <= K; d++) m = __vminu4(m, box[warp][kPad + x + d]);
            g.row_box[lin + x] = m;
            if (m != ~0u) {
                inset += __dp4a(m, 0x01010101u, 0u);
                nbox++;
            }
        }
        inset = __reduce_add_sync(0xffffffffu, inset);
        nbox = __reduce_add_sync(0xffffffffu, nbox);
        if (lane == 0 && nbox) atomicAdd(&P->row_inset, (unsigned long long)inset << 32 | nbox);
        __syncwarp();
    }
}

// The largest h within K fine cells of each fine cell along each axis, from
// the maxima along x: over 2K+1 rows in y (in range) and 2K+1 z planes
// (periodic; with fewer z cells than that, every plane).  A small particle's
// search from this cell reaches no farther than 2 max(h_i, hnb).
//
// And the vote of the cell grid for the next sort: the fine cells that hold
// particles, and among them, in a patch whose spread of h is wide (h_s >
// 1.4 h_median), those whose particles' neighbourhoods have no h above 0.8
// h_s.  Many such cells (h wide but smooth in space, as behind the free
// surface of a patch) favour a 3-cell stencil over median-sized cells; few
// (h varying from particle to particle) favour cells of edge h_s.
//
// And how far hnb is above each cell's own largest h, which decides between
// the walk over rows and the one over cells (use_cells).
__global__ void __launch_bounds__(256) k_cell_hnb(PatchDev* pd, Grid g, int K, const float* hnb_x, unsigned long long* vote)
{
    wait_before();
    PatchDev* P = pd + blockIdx.y;
    const int ncx = P->ncx, ncy = P->ncy, ncz = P->ncz;
    const int64_t nxy = (int64_t)ncx * ncy;
    const int64_t nfine = nxy * ncz;
    const bool wide = P->hs > 1.4 * P->hmed;
    const float lim = 0.8f * P->hs_f;
    // every z plane when they are fewer than 2K+1
    const int kz = 2 * K + 1 > ncz ? (ncz - 1) / 2 + 1 : K;
    uint32_t ne = 0, nn = 0, over = 0;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nfine; c += (int64_t)gridDim.x * blockDim.x) {
        const int z = (int)(c / nxy), y = (int)(c - z * nxy) / ncx;
        const int ylo = max(-K, -y), yhi = min(K, ncy - 1 - y);
        float m = 0.0f;
        for (int dz = -kz; dz <= kz; dz++) {
            int q = z + dz;
            while (q < 0) q += ncz;
            while (q >= ncz) q -= ncz;
            const float* p = hnb_x + P->cell_base + c + (int64_t)(q - z) * nxy;
            for (int dy = ylo; dy <= yhi; dy++) m = fmaxf(m, p[(int64_t)dy * ncx]);
        }
        g.hnb[P->cell_base + c] = m;
        const uint4 cr = g.cell[P->cell_base + c];
        if (cr.x < cr.y) {
            ne++;
            nn += (uint32_t)(wide && m < lim);
            over += (uint32_t)fminf(fmaf(__fdividef(m, __uint_as_float(cr.z)), 256.0f, -256.0f), 1024.0f);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        ne += __shfl_xor_sync(0xffffffffu, ne, o);
        nn += __shfl_xor_sync(0xffffffffu, nn, o);
        over += __shfl_xor_sync(0xffffffffu, over, o);
    }
    if ((threadIdx.x & 31) == 0 && ne) {
        atomicAdd(&P->h_spread, (unsigned long long)over << 32 | ne);
        atomicAdd(&vote[0], (unsigned long long)ne);
        atomicAdd(&vote[1], (unsigned long long)nn);
    }
}

int launch_cell_tables(const Launch& L, int npatch, PatchDev* pd, const Grid& g, const float4* r4, int K, float* tmp,
                       unsigned long long* vote)
{
    if (npatch <= 0) return 0;
    const int rows_x = npatch > 8 ? 64 : (L.sms * 8 + npatch - 1) / npatch;
    const int cells_x = npatch > 8 ? 16 : (L.sms * 8 + npatch - 1) / npatch;
    launch_next(k_cell_rows, dim3((unsigned)rows_x, (unsigned)npatch), 256, 0, L.stream, pd, g, r4, K, tmp);
    launch_next(k_cell_hnb, dim3((unsigned)cells_x, (unsigned)npatch), 256, 0, L.stream, pd, g, K, tmp, vote);
    return 2;
}

}  // namespace sphg
