// sph_internal.cuh -- device data layout and launch declarations shared by
// the CUDA translation units of libsph_gb300.so.  Not part of the C ABI.
//
// Particles live in HBM as structure-of-arrays, sorted by (patch, class,
// Morton cell).  Per patch, the particles with h <= h_s are "small" and the
// few above are "big" (h_s: a high quantile of h, so that about 1/64 of the
// patch is big).  A uniform grid of cells with edge s >= 2 h_s cell_factor
// covers the bounding box in x, y and the period lz in z; a small particle
// searches the (2K+1)^3 cells around its own (K = 1 for cell_factor >= 1,
// 2 for >= 1/2, 3 below) for small neighbours, row by row, pruned by the
// largest h around its cell, or cell by cell, pruned by each cell's own.  Big
// particles are indexed separately by coarse cells (aligned blocks of 2^kc
// fine cells with edge >= 2 h_max), which every particle searches for big
// neighbours; a big particle searches the fine grid as far as its own 2 h.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "../../include/sph.h"

namespace sphg {

constexpr int kMortonBits = 7;                 // per axis: at most 128 cells
constexpr int kMaxCellsAxis = 1 << kMortonBits;
constexpr int kClassShift = 3 * kMortonBits;   // key = patch << 22 | big << 21 | morton
constexpr int kPatchShift = kClassShift + 1;
constexpr uint32_t kMortonMask = (1u << kClassShift) - 1u;
constexpr int kColBits = 25;                   // packed column: j | stencil << 25
constexpr uint32_t kColMask = (1u << kColBits) - 1u;
constexpr int64_t kMaxParticles = int64_t(1) << kColBits;
constexpr int kMaxPatches = 256;
// Particles per work item (a chunk of one patch that one block of 256 threads
// takes): eight items for every SM where there are few particles (two blocks
// for all of 8000 left the step's passes at 40 us each), else rounds of eight
// of at most 4096 particles each (a shorter item spends the FP64 pipe on its
// block sum: 1024 took 0.74 ms in k_update at 8 M, 4096 0.63).
inline int item_chunk(int64_t n, int sms)
{
    const int64_t slots = (int64_t)sms * 8;
    const int64_t rounds = (n + slots * 4096 - 1) / (slots * 4096);
    const int64_t per = slots * (rounds < 1 ? 1 : rounds);
    const int64_t c = ((n + per - 1) / per + 255) / 256 * 256;
    return (int)(c < 256 ? 256 : c);
}
constexpr uint32_t kFarCode = 127;             // column stencil code: offset from the cell coordinates
#ifndef SPH_BIG_SHARE
#define SPH_BIG_SHARE 64
#endif
constexpr int kBigShare = SPH_BIG_SHARE;       // about 1/kBigShare of a patch is big
constexpr int kHFacN = 4096;                   // entries of the h-adaptation factor table

// status word bits (device, sticky until the host clears it)
constexpr int kStOverflow = 1;
constexpr int kStNonFinite = 2;
constexpr int kStTimeout = 4;
constexpr int kStBad = kStOverflow | kStNonFinite | kStTimeout;  // later phases skip

// Guard band of the FP32 neighbour pre-filter: a candidate is decided in FP32
// only when r^2 is outside [T (1 - tol), T (1 + tol)], T the FP64 threshold;
// otherwise the exact FP64 predicate decides.  tol = 2^-13 + 2^-16 s/h_i
// bounds the FP32 rounding of r^2 computed from cell-relative coordinates
// shifted by at most 3 cells (error below 60 * 2^-24 s/h relative to T) with
// a margin of more than 4x.
constexpr float kTolBase = 1.0f / 8192.0f;
constexpr float kTolCell = 1.0f / 65536.0f;
// stencil half-extent for a cell factor: K s >= 2 h_s needs K cell_factor >= 1
__host__ __device__ __forceinline__ int stencil_k(double cell_factor)
{
    return cell_factor >= 1.0 ? 1 : (cell_factor >= 0.5 ? 2 : 3);
}
// Cell edges carry a relative margin so that FP32 cell assignment can never
// separate two particles closer than 2 h_max by more than K cells.
constexpr double kCellMargin = 1.0 + 1.0 / 1024.0;
// with a 3-cell stencil, cells no finer than min(h_s, kCellMed h_median)
constexpr double kCellMed = 1.3;

struct PatchDev {
    int64_t begin, end;          // sorted slot range (fixed after set_patches)
    int64_t cell_base, cell_cap; // slice of the cell tables
    int32_t item_begin, item_end;  // work items of this patch
    double xmin, ymin, s, sz, hmax, lz;
    float s_f, sz_f, lz_f, inv_s_f, inv_sz_f, hmax_f;
    int32_t ncx, ncy, ncz, K;
    int32_t zmode;               // 0: 2K+1 distinct z cells; 1: all z cells + float wrap
    int32_t nbig;                // big particles (h > hs), counted by the key kernel
    uint32_t row_fill;           // slots of the row copy handed out so far
    double hs;                   // class threshold: small iff h <= hs
    double hlz, hsz;             // lz / 2, sz / 2
    float hs_f;
    double hmed;                 // median of h (histogram bin centre)
    int32_t kc;                  // coarse cell = 2^kc fine cells per axis
    int32_t ncxc, ncyc, nczc;    // coarse grid
    int32_t zmode_c;             // 0: 3 distinct coarse z cells; 1: all of them
    int64_t coarse_base;         // first coarse cell in the cell tables
    // of the row boxes (Grid::row_box): the sum of the four insets over the
    // fine cells that have one, << 32, and the count of these
    unsigned long long row_inset;
    // ... of hnb / (the cell's largest h) - 1 in 1/256, over the fine cells that
    // hold particles
    unsigned long long h_spread;
    // time state
    double dt, dt_prev;
    int64_t step;
};

// Per-patch reduction slots, ordered-integer encoded doubles.
constexpr int kHBins = 64;       // histogram of h / h_max for the class threshold
struct PatchRed {
    unsigned long long xmin, ymin, xmax, ymax, hmax, hcmin;
    uint32_t hist[kHBins];
};

struct WorkItem {
    int64_t begin, end;
    int32_t patch, pad;
};

// Device views handed to the kernels.
struct State {
    double *x, *y, *z, *vx, *vy, *vz, *m, *h, *u, *du_prev, *axp, *ayp, *azp;
};

// Cell record, 16 bytes: particles [x, y) of the sorted order (x = y: empty;
// fine cells hold small particles, coarse cells big ones), z = the largest h
// in the cell (FP32 bits), w = for fine cells the tight box of the cell's
// particles, as insets from the cell faces in 1/kBoxQ of the cell edge:
// bits 0-4 low x, 5-9 high x, 10-14 low y, 15-19 high y, 20-24 low z,
// 25-29 high z (rounded outwards up to the FP32 rounding of the offsets).
//
// The search reads its small candidates from a second copy of the records, in
// which the particles of a row of fine cells (all x at one y, z) are
// contiguous and ordered by cell: row[fine cell] = {first, end} slot of the
// cell in that copy, row_rec = {x from the grid's origin, oy, oz, 4 h^2} and
// row_id = sorted slot | x cell << kColBits.  A row of the search sphere is
// then one run of slots, where the Morton order holds one run per cell.
constexpr int kBoxQ = 32;
struct Grid {
    uint4* cell;         // [cell] record above
    uint2* row;          // [fine cell]
    float4* row_rec;     // [slot], padded past the end (read in groups)
    uint32_t* row_id;    // [slot], padded likewise
    uint32_t* row_box;   // [fine cell] where in y and z the particles of the
                         // row lie, K cells to each side of this one: insets
                         // from the cell's low and high y, low and high z
                         // face, a byte each, in 1/255 of the edge
    uint32_t* cellxyz;   // [particle] cx | cy << 8 | cz << 16
    const uint16_t* patch_of;  // [particle] patch index
    float* hnb;          // [fine cell] the largest h of the fine cells within
                         // K cells along each axis (z periodic): no small
                         // particle searching from this cell meets a larger one
};

struct Recs {             // FP32 records (written by gather / density)
    float4* r4;          // {ox, oy, oz, 4 h^2}  neighbour pre-filter
    float4* r5;          // {ox, oy, oz, m}      pair sums (mixed)
    float4* rv;          // {vhx, vhy, vhz, 1/(2h)} time-centred velocity (mixed)
    float4* rt;          // {rho, P/rho^2, c, h} thermodynamics (mixed)
    float* hc;           // h/c (mixed)
    float* pf;           // P (mixed)
    float* uf;           // u, staged by the gather (mixed)
    float4* acc;         // {ax, ay, az, du} (mixed)
};

struct Fp64 {             // FP64-path fields
    double *vhx, *vhy, *vhz;   // time-centred velocity
    double *rho, *P, *c, *A, *hc;
    double *w;                 // 1/(2h)
    double *g0, *g1;           // of the kernel gradient's factor: w^(5/3) and
                               // w^(8/3) (Wendland), w^5 and w (Sinc)
    double *ha, *ca;           // of the viscosity, from the density sum:
                               // h sqrt(eps) / 2 and c alpha / sqrt(eps)
    double *ax, *ay, *az, *du;
};

// ---- small device helpers ------------------------------------------------
__device__ __forceinline__ unsigned long long ord_f64(double d)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(d);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__host__ __device__ __forceinline__ double unord_f64(unsigned long long u)
{
    unsigned long long b = (u >> 63) ? (u & 0x7fffffffffffffffull) : ~u;
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double d;
    memcpy(&d, &b, sizeof(d));
    return d;
#endif
}
// FP64 conversions, sign tests and comparisons in integer arithmetic.  An SM
// retires two FP64 operations a clock, and a conversion or a comparison takes
// as much of that pipe as a multiply-add: with them the passes over the
// particles (keys, gather, update) were bound by it, not by memory.
//
// the nearest float, ties to even, as (float)d
__device__ __forceinline__ float f64_to_f32(double d)
{
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const uint32_t e = (hi >> 20) & 0x7ffu;
    if (e - 897u > 253u) return (hi << 1 | lo) == 0u ? __uint_as_float(hi) : (float)d;   // 0; outside the normal floats
    const uint32_t m = __funnelshift_l(lo, hi & 0x000fffffu, 3);      // 23 bits
    const uint32_t rest = lo << 3;
    const uint32_t up = rest > 0x80000000u || (rest == 0x80000000u && (m & 1u)) ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | (((e - 896u) << 23) + m + up));
}
// (double)f
__device__ __forceinline__ double f32_to_f64(float f)
{
    const uint32_t u = __float_as_uint(f), t = u & 0x7fffffffu;
    if (t - 0x00800000u >= 0x7f000000u) return t == 0u ? __hiloint2double((int)u, 0) : (double)f;   // 0; subnormal, infinite, NaN
    return __hiloint2double((int)((u & 0x80000000u) | ((t >> 3) + 0x38000000u)), (int)(u << 29));
}
// (double)v for 0 <= v < 2^20
__device__ __forceinline__ double small_to_f64(uint32_t v)
{
    if (v == 0u) return 0.0;
    const int k = 31 - __clz(v);
    return __hiloint2double((int)(((1023u + (uint32_t)k) << 20) | ((v << (20 - k)) & 0x000fffffu)), 0);
}
// a > b and a < -b for b > 0 and a no NaN
__device__ __forceinline__ bool above(double a, double b) { return __double_as_longlong(a) > __double_as_longlong(b); }
__device__ __forceinline__ bool below_neg(double a, double b)
{
    return (unsigned long long)__double_as_longlong(a) > ((unsigned long long)__double_as_longlong(b) | 0x8000000000000000ull);
}

__host__ __device__ __forceinline__ uint32_t part1by2(uint32_t v)
{
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}
__host__ __device__ __forceinline__ uint32_t compact1by2(uint32_t v)
{
    v &= 0x09249249u;
    v = (v | (v >> 2)) & 0x030C30C3u;
    v = (v | (v >> 4)) & 0x0300F00Fu;
    v = (v | (v >> 8)) & 0x030000FFu;
    v = (v | (v >> 16)) & 0x000003FFu;
    return v;
}

#ifdef __CUDACC__
// Sums of 7 per-thread values over a block of 256 threads, in a fixed order;
// thread q < 7 returns sum q.  The lanes of a warp halve the values they hold
// while they add (four, two and one of eight, then two plain steps): 9
// additions on the FP64 pipe where a butterfly per value takes 35.
__device__ __forceinline__ double block_sum7(const double (&v)[7], double (*sh)[8])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
    double a[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const double hi = k < 3 ? v[k + 4] : 0.0;
        a[k] = (h16 ? hi : v[k]) + __shfl_xor_sync(0xffffffffu, h16 ? v[k] : hi, 16);
    }
    double b[2];
#pragma unroll
    for (int k = 0; k < 2; k++) b[k] = (h8 ? a[k + 2] : a[k]) + __shfl_xor_sync(0xffffffffu, h8 ? a[k] : a[k + 2], 8);
    double c = (h4 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h4 ? b[0] : b[1], 4);
    c += __shfl_xor_sync(0xffffffffu, c, 2);
    c += __shfl_xor_sync(0xffffffffu, c, 1);
    const int q = (h16 ? 4 : 0) + (h8 ? 2 : 0) + (h4 ? 1 : 0);
    if ((lane & 3) == 0 && q < 7) sh[q][warp] = c;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < 7)
        for (int w = 0; w < 8; w++) s += sh[threadIdx.x][w];
    __syncthreads();
    return s;
}

// one particle's share of the conserved sums, accumulated with FMAs: M, P,
// L_z = m (x v_y - y v_x), twice E_kin (to be halved), E_int
__device__ __forceinline__ void cons_accum(double x, double y, double vx, double vy, double vz, double m,
                                           double u, double (&acc)[7])
{
    acc[0] += m;
    acc[1] = fma(m, vx, acc[1]);
    acc[2] = fma(m, vy, acc[2]);
    acc[3] = fma(m, vz, acc[3]);
    acc[4] = fma(m, fma(x, vy, -y * vx), acc[4]);
    acc[5] = fma(m, fma(vx, vx, fma(vy, vy, vz * vz)), acc[5]);
    acc[6] = fma(m, u, acc[6]);
}

// s + c: a compensated sum (Neumaier)
__device__ __forceinline__ void neumaier_add(double& s, double& c, double v)
{
    const double t = s + v;
    if (fabs(s) >= fabs(v)) c += (s - t) + v;
    else c += (v - t) + s;
    s = t;
}

// Compensated sum of part[0], part[stride], ... part[(n - 1) stride] by a
// block of 256 threads: thread t takes the terms t, t + 256, ... in order,
// lane l of the first warp adds the sums of threads l, l + 32, ..., and lane 0
// the 32 lane sums in lane order.  The order is fixed, so the result is
// reproducible; thread 0 returns it.  Bound by the chain of dependent
// additions and loads: one warp for the partials of 8 M particles took 32 us,
// one thread for those of 2 M 150.
__device__ __forceinline__ double block_neumaier(const double* part, int n, int stride, double* sh_s, double* sh_c)
{
    double s = 0.0, c = 0.0;
    for (int k = threadIdx.x; k < n; k += 256) neumaier_add(s, c, part[(int64_t)k * stride]);
    if (n > 32) {                       // (no term beyond the first warp otherwise)
        sh_s[threadIdx.x] = s;
        sh_c[threadIdx.x] = c;
        __syncthreads();
    }
    if (threadIdx.x >= 32) return 0.0;
    for (int k = threadIdx.x + 32; k < 256 && k < n; k += 32) {
        neumaier_add(s, c, sh_s[k]);
        c += sh_c[k];
    }
    double S = 0.0, C = 0.0;
    for (int l = 0; l < 32 && l < n; l++) {
        const double sl = __shfl_sync(0xffffffffu, s, l);
        const double cl = __shfl_sync(0xffffffffu, c, l);
        neumaier_add(S, C, sl);
        C += cl;
    }
    return S + C;
}
#endif

#ifdef __CUDACC__
// The kernels of a step follow one another on one stream, and for a few
// thousand particles most of them run for less time than the next one's launch
// takes.  So they are launched with programmatic stream serialization: the
// next kernel's launch is under way while the one before it ends, and its
// threads begin with wait_before(), which holds them until that kernel is
// complete and its writes are visible.  Every kernel launched by launch_next()
// begins with it, so each is complete before a later one reads or writes; none
// of them reads through the non-coherent path, whose loads could move above
// it.  Ten steps of 20^3 particles in FP64 3467 -> 3092 us, of 33^3 mixed
// 2773 -> 2439 us, sort and lists of 45^3 326 -> 302 us; 64 patches and 100^3
// as before.
__device__ __forceinline__ void wait_before() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
inline void launch_next(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, P(args)...);
}
#endif

// ---- launch wrappers (each returns the number of kernels launched) --------
struct Launch {
    cudaStream_t stream;
    int sms;
};

int launch_reduce_bbox(const Launch& L, const State& s, const WorkItem* items, int nitems,
                       PatchRed* red);
int launch_h_hist(const Launch& L, const State& s, const WorkItem* items, int nitems, PatchRed* red);
int launch_grid_params(const Launch& L, int npatch, const PatchRed* red, PatchDev* pd,
                       double cell_factor, int* status, unsigned long long* vote);
// the buffers of the radix sort: the sorted pairs end up in (keys, vals); work
// holds the digit counts of every pass, the passes' tickets and the tiles'
// look-back words, all cleared before the keys are made
constexpr int kRsMaxPasses = 4;
struct RadixSort {
    uint32_t *keys, *vals, *keys_alt, *vals_alt, *work;
    // where the unsorted pairs go, for an odd or even number of passes
    void input(int passes, uint32_t*& k, uint32_t*& v) const
    {
        k = passes & 1 ? keys_alt : keys;
        v = passes & 1 ? vals_alt : vals;
    }
};
size_t radix_work_words(int64_t n);       // words of work a sort of n uses
size_t radix_work_capacity(int64_t cap);  // ... of at most cap
int launch_keys(const Launch& L, int64_t n, const State& s, const uint16_t* patch_of, PatchDev* pd, const RadixSort& rs, int passes);
// LSD radix sort of 8 * passes key bits
int launch_radix_sort(const Launch& L, int64_t n, int passes, const RadixSort& rs, int* status);
// Row-length hints for the list pool: the previous lists' row lengths,
// carried into the new sorted order by the gather.  Only a hint: the list
// kernel reserves from it and repairs rows that outgrow their reservation.
constexpr uint32_t kNoHint = 0xffffffffu;
struct RowHint {
    const uint32_t* cnt_prev;    // row lengths in the previous sorted order
    const int* valid;            // nonzero: cnt_prev belongs to the order being gathered from
    uint32_t* rowcap;            // out: hint per new sorted slot, kNoHint if none
};
// hsearch (optional, the order gathered from): the h of the search when it
// is not the particles' h (the candidate superset of reused lists), gathered
// into hsearch_out and used for the search records and cell maxima
int launch_gather(const Launch& L, int64_t n, const uint32_t* skeys, const uint32_t* svals,
                  const State& src, const State& dst, const uint32_t* perm_src,
                  uint32_t* perm_dst, const PatchDev* pd, const Grid& g, const Recs& r,
                  const Fp64& f, int mixed, int kernel, const RowHint& hint, const int* status, const double* hsearch = nullptr,
                  double* hsearch_out = nullptr);
// the FP32 records of the current state in the current sorted order, on the
// grid of the last sort (what the gather writes, with the unscaled h)
int launch_refresh_records(const Launch& L, int64_t n, const State& s, const uint16_t* patch_of,
                           const PatchDev* pd, const uint32_t* cellxyz, const Recs& r, const Fp64& f, int mixed, int kernel);
// after the gather: the row copy of the small particles' search records,
// g.hnb for stencil half-extent K (tmp: one float per cell) and the state's
// vote for the grid of the next sort (vote[0]: non-empty fine cells, vote[1]:
// those whose hnb is below 0.8 h_s in a patch with h_s above 1.4 h_median;
// cleared by launch_grid_params)
int launch_cell_tables(const Launch& L, int npatch, PatchDev* pd, const Grid& g, const float4* r4, int K, float* tmp,
                       unsigned long long* vote);
// temporary words of the device-wide exclusive scan over n values
int64_t scan_tmp_words(int64_t n);

struct NbArgs {
    int64_t n;
    int K;                               // stencil half-extent of every patch
    int npatch;
    const PatchDev* pd;
    Grid g;
    const float4* r4;
    const double *x, *y, *z, *h;
    const WorkItem* units;               // 32 consecutive particles of one patch each
    int64_t nunits;
    uint32_t* cnt;                       // |N(i)|
    uint32_t* nown;                      // n_i
    unsigned long long* rowstart;        // first pool entry of row i
    uint32_t* col;                       // the list pool
    const uint32_t* rowcap;              // row-length hints (kNoHint: none)
    unsigned long long* pool_used;       // [0] entries reserved, [1] entries listed (nnz)
    int* hint_ok;                        // set: the row lengths belong to the current order
    int64_t max_pairs;                   // bound on nnz
    int64_t pool_cap;                    // entries the pool holds (max_pairs + slack)
    int* status;
};
// exact = 1: the neighbour lists and n_i; exact = 0: the candidate superset
// of reused lists (every candidate within the grid's scaled search radius)
int launch_nb_lists(const Launch& L, const NbArgs& a, int exact);
// exact lists (a.col, a.cnt, a.nown; rows at a.rowstart) from the superset
// rows col_s / cnt_s at the same offsets, on the current records and state
int launch_nb_filter(const Launch& L, const NbArgs& a, const uint32_t* col_s, const uint32_t* cnt_s);
int launch_canonical_rows(const Launch& L, int64_t n, const unsigned long long* rowstart,
                          const uint32_t* cnt, const uint64_t* off, const uint32_t* col, uint32_t* out);
// exclusive scan of n u32 values into u64 out[0..n], out[n] = total
int launch_scan_u32_to_u64(const Launch& L, int64_t n, const uint32_t* in, uint64_t* out, uint64_t* tmp);

struct PairArgs {
    int64_t n;
    const PatchDev* pd;
    const uint16_t* patch_of;
    const unsigned long long* rowstart;  // row i is col[rowstart[i] .. + cnt[i])
    const uint32_t* cnt;
    const uint32_t* col;
    const uint32_t* cellxyz;             // [particle] cell, for kFarCode columns
    State s;
    Recs r;
    Fp64 f;
    double gamma, alpha, beta, eps;
    double vh, vc, vb;                   // sqrt(eps) / 2, alpha / sqrt(eps), 2 beta / eps
    int kernel, kernel_n;                // SPH_KERNEL_*; n of the Sinc kernel
    int grad_h;                          // 1: grad-h form (density stores A/Omega)
    double kb;                           // sigma_W (Wendland) or B_n (Sinc)
    int* status;
    // row-length bins (nullptr order: every particle, in sorted order): the
    // launch takes positions bounds[bin_lo] .. bounds[bin_hi + 1] of order,
    // the particles whose rows fall in those octaves
    const uint32_t* order;
    const uint32_t* bounds;
    int bin_lo, bin_hi;
};
int launch_density(const Launch& L, const PairArgs& a, int tpp, int mixed);
int launch_momentum(const Launch& L, const PairArgs& a, int tpp, int mixed);
// Row-length bins: octave 0 holds the empty rows, octave o >= 1 the rows with
// |N(i)| in (2^(o-2), 2^(o-1)], o < kPairOctaves (the last octave takes every
// longer row).  With a target of 2^w list words per lane, octave o gets
// clamp(2^(o-1-w), 1, 32) lanes per particle -- the smallest power of two
// that keeps a lane at 2^w words or fewer -- and the rows of one launch's
// warps differ by less than 2x.
constexpr int kPairOctaves = 16;
__host__ __device__ __forceinline__ int octave_tpp(int o, int w)
{
    const int e = o - 1 - w;
    return e <= 0 ? 1 : (e >= 5 ? 32 : 1 << e);
}
// order = the particles stably sorted by octave (sorted order kept inside
// each octave), bounds[o] = first position of octave o, bounds[kPairOctaves] = n
// (rs.vals is the order)
int launch_pair_bins(const Launch& L, int64_t n, const uint32_t* cnt, const RadixSort& rs, uint32_t* bounds, int* status);
// the sums over row-length bins with 2^w words per lane (one launch per
// distinct lanes-per-particle value)
int launch_density_binned(const Launch& L, PairArgs a, int w, int mixed);
int launch_momentum_binned(const Launch& L, PairArgs a, int w, int mixed);
// list-free pair sums over the search of the current grid; the density pass also writes |N(i)| and n_i and adds the
// pairs to pool_used[1]
int launch_fused_density(const Launch& L, const NbArgs& a, const PairArgs& pa, int mixed);
int launch_fused_momentum(const Launch& L, const NbArgs& a, const PairArgs& pa, int mixed);

struct StepArgs {
    int64_t n;
    PatchDev* pd;
    int npatch;
    const WorkItem* items;
    int nitems;
    PatchRed* red;
    State s;
    Recs r;
    Fp64 f;
    const uint32_t* nown;
    double courant, dt_growth, dt_fixed, n_target;
    int adapt_h, mixed;
    const double* hfac;  // [n] 0.5 (1 + cbrt(n_target / n)) for 0 < n < kHFacN, host-computed

    double* partials;    // [nitems][7]
    double* cons;        // [npatch][7]
    int* status;
    const unsigned long long* listed;  // entries of this step's lists
    unsigned long long* pair_acc;      // ... summed over the steps
    unsigned* dt_ticket;               // blocks of k_dt that are done (0 between steps)
};
// the time-step of every patch from its smallest h/c, and the step's pairs
// added to pair_acc
int launch_dt(const Launch& L, const StepArgs& a);
int launch_update(const Launch& L, const StepArgs& a);
// reused candidate supersets: the state the superset was built on (sorted
// order), and the check that it still holds every neighbour pair
struct SkinRef {
    double *x0, *y0, *z0;  // positions the superset was built on
    double* h0;            // its search h (the superset lists r < 2 max(h0_i, h0_j))
};
int launch_skin_snapshot(const Launch& L, int64_t n, const State& s, const SkinRef& ref);
// the superset's search h per particle (current order): h (1 + skin + 3 (f - 1)+),
// f the h-adaptation factor of the last step (from n_i; 1 when nown is NULL)
int launch_skin_radius(const Launch& L, int64_t n, const State& s, const uint32_t* nown, const double* hfac,
                       double n_target, double skin, double* hsearch);
// flag (device) = 1 while max |x - x0| <= min (h0 - h), h0 = the superset's search h
int launch_skin_check(const Launch& L, int64_t n, const State& s, const uint16_t* patch_of, const PatchDev* pd,
                      const SkinRef& ref, unsigned long long* red, int* flag);
int launch_conserved_items(const Launch& L, const StepArgs& a);
int launch_conserved_finalize(const Launch& L, const StepArgs& a);
int launch_step_finalize(const Launch& L, const StepArgs& a);
int launch_unpermute_f64(const Launch& L, int64_t n, const double* src, const uint32_t* perm,
                         double* dst);
int launch_unpermute_f32(const Launch& L, int64_t n, const float* src, int stride,
                         const uint32_t* perm, double* dst);
int launch_unpermute_u32(const Launch& L, int64_t n, const uint32_t* src, const uint32_t* perm,
                         double* dst);
// new particles: src (x y z vx vy vz m h u; may be s's own arrays) into s, the
// time fields cleared, perm the identity; status: kStNonFinite for bad values
int launch_load(const Launch& L, int64_t n, const double* const src[9], const State& s, uint32_t* perm, int* status);
// what k_reset_red clears besides the reductions
struct SortClear {
    uint32_t* work;                // radix sort's histograms, tickets and tile states
    int64_t words;
    uint4* cell;                   // cell table
    int64_t cells;
    unsigned long long* pool_used;
};
int launch_reset_red(const Launch& L, int npatch, PatchRed* red, const SortClear& c);

}  // namespace sphg
