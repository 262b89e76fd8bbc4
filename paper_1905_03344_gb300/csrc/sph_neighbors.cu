// sph_neighbors.cu -- neighbour discovery, second half: the symmetric
// neighbour lists, one row per particle from the search in sph_walk.cuh.
//
// Rows go straight to the pool.  Each lane reserves its row before the walk,
// from the row-length hint c (the particle's row length in the previous
// lists) as c + c/3 + 8 entries -- on a lattice a small change of h adds a
// whole shell of neighbours at once, up to about a third of the row -- or,
// without a hint, from a first walk that only counts.  Reservations are
// rounded up to a multiple of 8 entries, so every row starts on a 32-byte
// boundary.  Hits collect in a 16-slot ring in shared memory and leave it as
// whole 32-byte sectors.  A row that outgrows its reservation is walked again
// into a fresh reservation of its exact (rounded) length.  Shared memory per
// warp is 2 KB, which leaves the SM's L1 to the candidate gathers.  Row
// contents are fixed by the inputs; only the place of a row in the pool
// depends on scheduling, and every consumer reads a row through its start
// and length, so all results are bitwise reproducible.  The canonical CSR
// with prefix offsets is built from the pool on demand (sph_get_neighbors).
#include "sph_pairmath.cuh"
#include "sph_walk.cuh"

namespace sphg {

// counting walk (col = nullptr) and repair walk (straight to the pool): one
// out-of-line copy serves both
template <bool EXACT, int K>
__device__ __noinline__ RowSink<kWalkFlat, EXACT> walk_all_flat(const NbArgs& a, const PatchDev* P, int64_t i,
                                                             bool big, RowSink<kWalkFlat, EXACT> row)
{
    walk_all<RowSink<kWalkFlat, EXACT>, K>(a, P, i, big, row);
    return row;
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, int lane)
{
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// EXACT = false: the candidate superset (every candidate within the scaled
// search radius in FP32, no n_i).  K = 0: the patches searched by rows; else
// those searched by cells, with stencils of K.  Two kernels, since one that
// branches between the two walks, at the 64 registers of eight blocks an SM,
// took 3 % longer in either (200^3 8.85 -> 9.1 ms, 64 patches 5.97 -> 6.17); a
// launch that finds no patch of its kind is done in 2 us.
template <bool EXACT, int K>
__global__ void __launch_bounds__(32 * kNbtWarps, SPH_NB_MINB) k_nb_thread(NbArgs a)
{
    wait_before();
    extern __shared__ __align__(16) uint32_t nb_ring[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* ring = nb_ring + warp * (32 * (kRing + kPend)) + lane;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.hint_ok = 1;
    if (*a.status & kStBad) return;
    const unsigned long long pool_cap = (unsigned long long)a.pool_cap;
    if (a.npatch == 1 && use_cells(a.pd) != (K > 0)) return;
    for (int64_t q = (int64_t)blockIdx.x * kNbtWarps + warp; q < a.nunits; q += (int64_t)gridDim.x * kNbtWarps) {
        const WorkItem U = a.units[q];
        const PatchDev* P = a.pd + U.patch;
        if (use_cells(P) != (K > 0)) continue;
        const int64_t i = U.begin + lane;
        const bool act = i < U.end;
        // big particles sit at the end of their patch
        const bool big = act && i >= P->end - (int64_t)P->nbig;
        // reservation: the hint plus a margin, or the counted length
        uint32_t res = 0;
        if (act) {
            const uint32_t hint = a.rowcap[i];
            if (hint == kNoHint) {
                const RowSink<kWalkFlat, EXACT> rc =
                    walk_all_flat<EXACT, K>(a, P, i, big, RowSink<kWalkFlat, EXACT>{nullptr, nullptr, 0u, 0u, 0u, 0u});
                res = round8(rc.cnt);
            } else {
                const uint32_t c = min(hint, (uint32_t)a.n);
                res = round8(c + c / 3u + kHintMargin);
            }
        }
        const uint32_t inc = warp_incl_scan(res, lane);
        const uint32_t tot = __shfl_sync(0xffffffffu, inc, 31);
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(&a.pool_used[0], (unsigned long long)tot);
        base = __shfl_sync(0xffffffffu, base, 0);
        const bool ok = base + tot <= pool_cap;
        if (!ok && lane == 0) atomicOr(a.status, kStOverflow);
        unsigned long long r0 = base + (inc - res);
        RowSink<kWalkRing, EXACT> row = {a.col + r0, ring, ok ? res : 0u, 0u, 0u, 0u};
        if (act) {
            walk_all<RowSink<kWalkRing, EXACT>, K>(a, P, i, big, row);
            row.finish();
            // only a row that is in the pool (within the sink's reservation,
            // which is 0 for a warp whose reservation did not fit)
            if (row.npend > 0 && row.npend <= (uint32_t)kPend && row.cnt <= row.res) row.resolve_band(a, P, i);
        }
        if (act && ok && (row.cnt > res || row.npend > (uint32_t)kPend)) {
            // outgrew the reservation, or deferred more guard-band words than
            // it notes: walk again, deciding in place, into an exact reservation
            const uint32_t need = round8(row.cnt);
            r0 = atomicAdd(&a.pool_used[0], (unsigned long long)need);
            if (r0 + need <= pool_cap) {
                const RowSink<kWalkFlat, EXACT> rr = walk_all_flat<EXACT, K>(
                    a, P, i, big, RowSink<kWalkFlat, EXACT>{a.col + r0, nullptr, need, 0u, 0u, 0u});
                row.cnt = rr.cnt;
                row.own = rr.own;
            } else {
                atomicOr(a.status, kStOverflow);
            }
        }
        if (act) {
            a.rowstart[i] = r0;
            a.cnt[i] = row.cnt;
            if (EXACT) a.nown[i] = row.own;
        }
        const uint32_t listed = __shfl_sync(0xffffffffu, warp_incl_scan(act ? row.cnt : 0u, lane), 31);
        if (lane == 0) {
            const unsigned long long before = atomicAdd(&a.pool_used[1], (unsigned long long)listed);
            if (before + listed > (unsigned long long)a.max_pairs) atomicOr(a.status, kStOverflow);
        }
    }
}

template <bool EXACT, int K>
void launch_nb_thread(const Launch& L, const NbArgs& a)
{
    const size_t smem = sizeof(uint32_t) * 32 * (kRing + kPend) * kNbtWarps;
    static int per_sm = 0;
    if (!per_sm) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_nb_thread<EXACT, K>, 32 * kNbtWarps, smem);
        if (per_sm < 1) per_sm = 1;
        // shared memory only for the rings of the resident CTAs: the rest is L1
        int smem_max = 0, dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
        if (smem_max > 0) {
            const size_t need = (size_t)per_sm * (smem + 1024);
            int pct = (int)((need * 100 + (size_t)smem_max - 1) / (size_t)smem_max);
            pct = pct < 1 ? 1 : (pct > 100 ? 100 : pct);
            cudaFuncSetAttribute(k_nb_thread<EXACT, K>, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
        }
    }
    launch_next(k_nb_thread<EXACT, K>, L.sms * per_sm, 32 * kNbtWarps, smem, L.stream, a);
}

// ---- a team of lanes per particle ------------------------------------------
// For few particles: one thread per particle leaves the SMs with a warp or two
// each (8000 particles are 1.6 warps per SM), and a search lasts as long as
// one thread's chain of loads and tests.  Here eight lanes share a particle.
// They first write down its runs of candidates (a row each, the empty ones
// left out) in shared memory, then test the runs eight candidates at a time,
// one per lane: neighbouring lanes load neighbouring records, a vote gives
// each hit its place in the row, and the row is the one that a single thread
// would write.
//
// Bound by instruction issue: about 1600 warp instructions a particle against
// 870 of the thread walk, so the line lies where 152 SMs fill up; on the
// irregular patch, whose threads wait for the longest row of their warp, that
// is past 91,000 particles.  Search in us, thread / team: lattice 20^3 95 / 28,
// 33^3 100 / 70, 45^3 139 / 168; h raised behind the surface 20^3 143 / 53,
// 33^3 171 / 136, 45^3 200 / 298; irregular 20^3 182 / 66, 33^3 408 / 152, 45^3
// 473 / 421.  A team whose lanes take whole rows instead (hits collected in
// shared memory) took 33 us at 20^3, 101 at 33^3 and 424 on the irregular 33^3.
constexpr int kTeam = 8;
constexpr int kTeams = 32 / kTeam;      // particles a warp searches for at a time
constexpr int kTeamRuns = 32;           // runs written down at a time
constexpr int64_t kTeamMost = 50000;    // particles up to which teams search

struct TeamShared {
    uint4 run[kTeams][kTeamRuns];       // first candidate, end, column word bits (low bit: no code), z shift (coarse)
    float2 off[kTeams][kTeamRuns];      // the particle's y and z in the row's frame
};

// one particle's search, as the lanes of its team hold it
struct TeamCtx {
    float xi, yi, zi, Ti, eps;
    uint32_t i, cc;
    uint32_t cnt, own, lim;
    uint32_t* col;
};

enum TeamKind { kTeamRow = 0, kTeamRowWrap = 1, kTeamCoarse = 2 };

// the candidates of nr runs of each team; flag: every candidate has a stencil
// code (coarse cells: distinct coarse z cells)
template <int KIND, bool EXACT>
__device__ __forceinline__ void team_tests(const NbArgs& a, const PatchDev* P, const uint4* run, const float2* off, int nr, int lane,
                                           bool flag, TeamCtx& C)
{
    const uint32_t tl = lane & (kTeam - 1), tsh = lane & ~(kTeam - 1), lt = (1u << tl) - 1u;
    const float lz_f = P->lz_f, inv_lz = 1.0f / lz_f, s_f = P->s_f, sz_f = P->sz_f;
    const bool wrap = KIND == kTeamRowWrap || (KIND == kTeamCoarse && !flag);
    const int nmax = __reduce_max_sync(0xffffffffu, nr);
#pragma unroll 1
    for (int e = 0; e < nmax; e++) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        float2 f = make_float2(0.0f, 0.0f);
        if (e < nr) {
            v = run[e];
            if (KIND != kTeamCoarse) f = off[e];
        }
#pragma unroll 1
        for (uint32_t k = v.x + tl; __any_sync(0xffffffffu, k < v.y); k += kTeam) {
            const bool in_run = k < v.y;
            const uint32_t kk = in_run ? k : (v.y ? v.y - 1u : 0u);
            float4 q;
            uint32_t w, j;
            float dx, dy, dz;
            if (KIND == kTeamCoarse) {
                j = kk;
                q = a.r4[j];
                const uint32_t cj = a.g.cellxyz[j];
                const int dcx = (int)(cj & 255u) - (int)(C.cc & 255u), dcy = (int)((cj >> 8) & 255u) - (int)((C.cc >> 8) & 255u);
                const int dcz = (int)(cj >> 16) + (int)v.w - (int)(C.cc >> 16);
                w = j | (stencil_code(P, dcx, dcy, dcz, flag) << kColBits);
                dx = C.xi - fmaf((float)(cj & 255u), s_f, q.x);
                dy = (C.yi - (float)dcy * s_f) - q.y;
                dz = (C.zi - (float)dcz * sz_f) - q.z;
            } else {
                q = a.g.row_rec[kk];
                const uint32_t id = a.g.row_id[kk];
                j = id & kColMask;
                w = id + v.z;
                if (!flag && ((v.z & 1u) || (id >> kColBits) - ((C.cc & 255u) - 2u) > 4u)) w = j | (kFarCode << kColBits);
                dx = C.xi - q.x;
                dy = f.x - q.y;
                dz = f.y - q.z;
            }
            if (wrap) dz = fmaf(-lz_f, rintf(dz * inv_lz), dz);
            // (masked by a predicate: no value of r2 is beyond every threshold,
            // which are in the caller's units)
            const bool valid = in_run && j != C.i;
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            float d = r2 - fmaxf(C.Ti, q.w), o = r2 - C.Ti;
            if (EXACT) {
                // the guard band: decided exactly
                const float eps = C.eps * fmaxf(C.Ti, q.w);
                if (valid && fminf(fabsf(d), fabsf(o)) <= eps) {
                    const int x = exact_pair_at(a, (int64_t)C.i, j, P->lz);
                    d = x & 1 ? -1.0f : 1.0f;
                    o = x & 2 ? -1.0f : 1.0f;
                }
                C.own += (uint32_t)(valid && o < 0.0f);
            } else {
                d -= C.eps * fmaxf(C.Ti, q.w);
            }
            const bool in = valid && d < 0.0f;
            const uint32_t m = (__ballot_sync(0xffffffffu, in) >> tsh) & ((1u << kTeam) - 1u);
            const uint32_t p = C.cnt + (uint32_t)__popc(m & lt);
            if (in && p < C.lim) __stcs(C.col + p, w);
            C.cnt += (uint32_t)__popc(m);
        }
    }
}

// the whole search of the teams' particles (act: the team has one)
template <bool EXACT>
__device__ __forceinline__ void team_search(const NbArgs& a, const PatchDev* P, TeamShared& sh, int lane, bool act, const RowReach& R,
                                            float hf, TeamCtx& C)
{
    const int tl = lane & (kTeam - 1), team = lane / kTeam;
    const uint32_t tsh = lane & ~(kTeam - 1), lt = (1u << tl) - 1u;
    uint4* run = sh.run[team];
    float2* off = sh.off[team];
    const float s_f = P->s_f, sz_f = P->sz_f, inv_s = P->inv_s_f;
    const int ncx = P->ncx, ncy = P->ncy, ncz = P->ncz;
    const uint32_t cbase = (uint32_t)P->cell_base;
    const int cx = C.cc & 255, cy = (C.cc >> 8) & 255, cz = C.cc >> 16;
    const float xs = C.xi * inv_s;
    const int xlo = max(cx - R.kx, 0), xhi = min(cx + R.kx, ncx - 1);
    const int ylo = max(-R.kx, -cy), ny = min(R.kx, ncy - 1 - cy) - ylo + 1;
    const bool coded = R.kx <= 2 && (R.zw ? P->zmode && ncz <= 5 : R.kz <= 2);
    C.eps = row_tol(s_f / hf, R.zw ? max(R.kx, ncz) : max(R.kx, R.kz));
    // (teams whose walk wraps z, by a large radius or a small patch, after the others)
#pragma unroll 1
    for (int zw = 0; zw < 2; zw++) {
        const int nrow = act && (int)R.zw == zw ? ny * (zw ? ncz : 2 * R.kz + 1) : 0;
        const int most = __reduce_max_sync(0xffffffffu, nrow);
        const bool all_coded = __all_sync(0xffffffffu, coded || nrow == 0);
#pragma unroll 1
        for (int r0 = 0; r0 < most; r0 += kTeamRuns) {
            int nr = 0;
#pragma unroll 1
            for (int r = r0 + tl; __any_sync(0xffffffffu, r - tl < min(nrow, r0 + kTeamRuns)); r += kTeam) {
                uint32_t k = 0, ke = 0, add = 1u;
                float2 f = make_float2(0.0f, 0.0f);
                if (r < min(nrow, r0 + kTeamRuns)) {
                    const int iz = r / ny, dcy = ylo + r - iz * ny;
                    const int dcz = zw ? iz : iz - R.kz;
                    int czj = cz + dcz;
                    if (czj < 0) czj += ncz;
                    else if (czj >= ncz) czj -= ncz;
                    const uint32_t lrow = cbase + ((uint32_t)czj * (uint32_t)ncy + (uint32_t)(cy + dcy)) * (uint32_t)ncx;
                    const uint32_t box = R.kx <= P->K && use_boxes(P) ? a.g.row_box[lrow + (uint32_t)cx] : 0u;
                    f = make_float2(C.yi - (float)dcy * s_f, C.zi - (float)dcz * sz_f);
                    const float rem2 = R.Rg2 - (zw ? row_gap2<false>(box, f.x, f.y, s_f, sz_f) : row_gap2<true>(box, f.x, f.y, s_f, sz_f));
                    if (rem2 > 0.0f) {
                        // the chord, in cells (Rg's margins cover the rounding
                        // and the FP32 cell assignment)
                        const float half = __fsqrt_rn(rem2) * inv_s;
                        const int x0 = max((int)floorf(xs - half), xlo), x1 = min((int)floorf(xs + half), xhi);
                        if (x0 <= x1) {
                            k = a.g.row[lrow + (uint32_t)x0].x;
                            ke = a.g.row[lrow + (uint32_t)x1].y;
                            const int zd = zw ? (P->zmode ? iz : 5) : dcz + 2;
                            if ((uint32_t)(dcy + 2) <= 4u && (uint32_t)zd <= 4u)
                                add = (uint32_t)(2 + 5 * (dcy + 2) + 25 * zd - cx) << kColBits;
                        }
                    }
                }
                const uint32_t m = (__ballot_sync(0xffffffffu, k < ke) >> tsh) & ((1u << kTeam) - 1u);
                if (k < ke) {
                    const int at = nr + __popc(m & lt);
                    run[at] = make_uint4(k, ke, add, 0u);
                    off[at] = f;
                }
                nr += __popc(m);
            }
            __syncwarp();
            if (zw) team_tests<kTeamRowWrap, EXACT>(a, P, run, off, nr, lane, all_coded, C);
            else team_tests<kTeamRow, EXACT>(a, P, run, off, nr, lane, all_coded, C);
            __syncwarp();
        }
    }
    if (P->nbig <= 0) return;
    // the coarse cells
    const bool zwc = P->zmode_c != 0;
    const int kc = P->kc, Cc = 1 << kc;
    const int ncell = act ? 9 * (zwc ? P->nczc : 3) : 0;
    const int most = __reduce_max_sync(0xffffffffu, ncell);
    C.eps = row_tol(s_f / hf, 2 * Cc);
#pragma unroll 1
    for (int r0 = 0; r0 < most; r0 += kTeamRuns) {
        int nr = 0;
#pragma unroll 1
        for (int r = r0 + tl; r - tl < min(most, r0 + kTeamRuns); r += kTeam) {
            uint32_t k = 0, ke = 0;
            int zs = 0;
            if (r < min(ncell, r0 + kTeamRuns)) {
                const int iz = r / 9, t = r - iz * 9, dy = t / 3 - 1, dx = t - (dy + 1) * 3 - 1;
                const int X = (cx >> kc) + dx, Y = (cy >> kc) + dy;
                int Z = iz;
                if (!zwc) {
                    Z = (cz >> kc) + iz - 1;
                    if (Z < 0) { Z += P->nczc; zs = -ncz; }
                    else if (Z >= P->nczc) { Z -= P->nczc; zs = ncz; }
                }
                if ((unsigned)X < (unsigned)P->ncxc && (unsigned)Y < (unsigned)P->ncyc) {
                    const uint4 cr = a.g.cell[P->coarse_base + ((int64_t)Z * P->ncyc + Y) * P->ncxc + X];
                    if (cr.x < cr.y) {
                        const float ylow = (float)(Y * Cc - cy) * s_f, yhigh = (float)(min(Y * Cc + Cc, ncy) - cy) * s_f;
                        const float gx = fmaxf(fmaxf((float)(X * Cc) * s_f - C.xi, C.xi - (float)min(X * Cc + Cc, ncx) * s_f), 0.0f);
                        const float gy = fmaxf(fmaxf(ylow - C.yi, C.yi - yhigh), 0.0f);
                        float gz = 0.0f;
                        if (!zwc)
                            gz = fmaxf(fmaxf((float)(Z * Cc + zs - cz) * sz_f - C.zi,
                                             C.zi - (float)(min(Z * Cc + Cc, ncz) + zs - cz) * sz_f), 0.0f);
                        const float Rr = fmaxf(hf, __uint_as_float(cr.z)) * (2.0f * (1.0f + 1.0f / 512.0f)) + s_f * (1.0f / 4096.0f);
                        if (fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < Rr * Rr) {
                            k = cr.x;
                            ke = cr.y;
                        }
                    }
                }
            }
            const uint32_t m = (__ballot_sync(0xffffffffu, k < ke) >> tsh) & ((1u << kTeam) - 1u);
            if (k < ke) run[nr + __popc(m & lt)] = make_uint4(k, ke, 0u, (uint32_t)zs);
            nr += __popc(m);
        }
        __syncwarp();
        team_tests<kTeamCoarse, EXACT>(a, P, run, off, nr, lane, !zwc, C);
        __syncwarp();
    }
}

// A warp takes a unit of 32 consecutive particles of one patch, or 32 >>
// sub_log of them, four at a time.
template <bool EXACT>
__global__ void __launch_bounds__(32 * kNbtWarps, 5) k_nb_team(const __grid_constant__ NbArgs a, int sub_log)
{
    wait_before();
    __shared__ TeamShared shared[kNbtWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    TeamShared& sh = shared[warp];
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.hint_ok = 1;
    if (*a.status & kStBad) return;
    const int width = 32 >> sub_log;
    const int64_t nparts = a.nunits << sub_log;
    for (int64_t q = (int64_t)blockIdx.x * kNbtWarps + warp; q < nparts; q += (int64_t)gridDim.x * kNbtWarps) {
        // the big particles at the end of a patch have the longest searches: begin with them
        const int64_t part = nparts - 1 - q;
        const WorkItem U = a.units[part >> sub_log];
        const PatchDev* P = a.pd + U.patch;
        const int64_t begin = U.begin + (part & ((1 << sub_log) - 1)) * width;
        const int n = (int)min((int64_t)width, U.end - begin);
        if (n <= 0) continue;
        // lane l holds particle begin + l's row: words reserved, words and n_i
        // found
        const bool act = lane < n;
        const uint32_t hint = act ? a.rowcap[begin + lane] : 0u;
        uint32_t res = 0, cnt = 0, own = 0;
        unsigned long long r0 = 0;
        bool ok = true;
        // pass 0 counts the rows (without hints), 1 writes them, 2 writes the
        // rows that outgrew their reservation again
        int pass = __any_sync(0xffffffffu, act && hint == kNoHint) ? 0 : 1;
        uint32_t todo = 0xffffffffu >> (32 - n);
#pragma unroll 1
        for (;;) {
            if (pass == 1) {
                if (act) {
                    const uint32_t c = min(hint, (uint32_t)a.n);
                    res = hint == kNoHint ? round8(cnt) : round8(c + c / 3u + kHintMargin);
                }
                const uint32_t inc = warp_incl_scan(res, lane);
                const uint32_t tot = __shfl_sync(0xffffffffu, inc, 31);
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(&a.pool_used[0], (unsigned long long)tot);
                base = __shfl_sync(0xffffffffu, base, 0);
                ok = base + tot <= (unsigned long long)a.pool_cap;
                if (!ok && lane == 0) atomicOr(a.status, kStOverflow);
                r0 = base + (inc - res);
            }
#pragma unroll 1
            for (int g = 0; g < n; g += kTeams) {
                if (!(todo >> g & ((1u << kTeams) - 1u))) continue;
                const int p = g + lane / kTeam;
                const bool on = p < n && (todo >> p & 1u);
                const int64_t i = begin + (p < n ? p : 0);
                TeamCtx C;
                C.i = (uint32_t)i;
                C.cc = a.g.cellxyz[i];
                const float4 ri = a.r4[i];
                const float hf = (float)a.h[i];
                C.xi = fmaf((float)(C.cc & 255u), P->s_f, ri.x);   // as in the row copy
                C.yi = ri.y;
                C.zi = ri.z;
                C.Ti = ri.w;
                C.cnt = C.own = 0u;
                const uint32_t room = __shfl_sync(0xffffffffu, res, p & 31);
                const unsigned long long at = __shfl_sync(0xffffffffu, r0, p & 31);
                C.lim = on && pass != 0 && ok ? room : 0u;
                C.col = a.col + at;
                const RowReach R = row_reach(a, P, C.cc, hf, i >= P->end - (int64_t)P->nbig);
                team_search<EXACT>(a, P, sh, lane, on, R, hf, C);
#pragma unroll
                for (int o = kTeam / 2; o > 0; o >>= 1) C.own += __shfl_xor_sync(0xffffffffu, C.own, o);
                // to the lane that holds the particle
                const int src = ((lane - g) & (kTeams - 1)) * kTeam;
                const uint32_t c = __shfl_sync(0xffffffffu, C.cnt, src), w = __shfl_sync(0xffffffffu, C.own, src);
                if (lane >= g && lane < g + kTeams && (todo >> lane & 1u)) {
                    cnt = c;
                    own = w;
                }
            }
            if (pass == 0) {
                pass = 1;
                continue;
            }
            if (pass == 2 || !ok) break;
            // outgrew the reservation: again, into an exact one
            const bool more = act && cnt > res;
            todo = __ballot_sync(0xffffffffu, more);
            if (!todo) break;
            if (more) {
                res = round8(cnt);
                r0 = atomicAdd(&a.pool_used[0], (unsigned long long)res);
                if (r0 + res > (unsigned long long)a.pool_cap) {
                    atomicOr(a.status, kStOverflow);
                    res = 0u;
                    r0 = 0ull;
                }
            }
            pass = 2;
        }
        if (act) {
            a.rowstart[begin + lane] = r0;
            a.cnt[begin + lane] = cnt;
            if (EXACT) a.nown[begin + lane] = own;
        }
        const uint32_t listed = __reduce_add_sync(0xffffffffu, act ? cnt : 0u);
        if (lane == 0) {
            const unsigned long long before = atomicAdd(&a.pool_used[1], (unsigned long long)listed);
            if (before + listed > (unsigned long long)a.max_pairs) atomicOr(a.status, kStOverflow);
        }
    }
}

template <bool EXACT>
static void launch_nb_team(const Launch& L, const NbArgs& a)
{
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_nb_team<EXACT>, 32 * kNbtWarps, 0);
    if (per_sm < 1) per_sm = 1;
    // smaller parts while there would be fewer than two for every resident warp
    const int64_t resident = (int64_t)L.sms * per_sm * kNbtWarps;
    int sub_log = 0;
    while (sub_log < 3 && (a.nunits << sub_log) < 2 * resident) sub_log++;
    const int64_t need = ((a.nunits << sub_log) + kNbtWarps - 1) / kNbtWarps, cap = (int64_t)L.sms * per_sm;
    launch_next(k_nb_team<EXACT>, (unsigned)(need < cap ? need : cap), 32 * kNbtWarps, 0, L.stream, a, sub_log);
}

template <bool EXACT>
static int launch_nb(const Launch& L, const NbArgs& a)
{
    if (a.n <= kTeamMost) {
        launch_nb_team<EXACT>(L, a);
        return 1;
    }
    if (a.K == 1) {
        launch_nb_thread<EXACT, 1>(L, a);
        return 1;
    }
    launch_nb_thread<EXACT, 0>(L, a);
    if (a.K == 2) launch_nb_thread<EXACT, 2>(L, a);
    else launch_nb_thread<EXACT, 3>(L, a);
    return 2;
}

int launch_nb_lists(const Launch& L, const NbArgs& a, int exact)
{
    if (a.n <= 0 || a.nunits <= 0) return 0;
    return exact ? launch_nb<true>(L, a) : launch_nb<false>(L, a);
}

// ---- exact lists from a reused candidate superset -------------------------
// Row i of the superset (col_s from rowstart[i], cnt_s[i] words, built on an
// earlier state with the search radius scaled by 1 + skin) is decided again
// on the current state: the FP32 test on the records refreshed for the
// current positions and h, and the exact FP64 predicate inside the guard
// band, as in the search.  The accepted words keep their order and go to
// the exact pool at the same offset.  A group of TPP lanes per row: each
// lane decides one word per round; the group ballots and writes the accepted
// words contiguously.  Groups of a warp run their rounds together (a shorter
// row idles through the longer one's last rounds), so TPP = 32: one row per
// warp in lockstep.
template <int TPP>
__global__ void __launch_bounds__(256) k_nb_filter(NbArgs a, const uint32_t* col_s, const uint32_t* cnt_s)
{
    if (*a.status & kStBad) return;
    const int lane = threadIdx.x & 31;
    const int gl = lane & (TPP - 1);
    const unsigned gmask = TPP == 32 ? 0xffffffffu : (((1u << TPP) - 1u) << (lane & ~(TPP - 1)));
    const unsigned below = (1u << lane) - 1u;    // lanes before this one
    const int64_t gs = ((int64_t)gridDim.x * blockDim.x) / TPP;
    unsigned long long listed = 0;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / TPP; i < a.n; i += gs) {
        const PatchDev* P = a.pd + a.g.patch_of[i];
        const float s_f = P->s_f, sz_f = P->sz_f, lz_f = P->lz_f;
        const int zmode = P->zmode, Dcode = zmode ? max(2, P->ncz) : 2;
        const float4 ri = a.r4[i];
        const uint32_t ci = a.g.cellxyz[i];
        const float Ti = ri.w;
        const float sh = s_f / (float)a.h[i];
        const unsigned long long rs = a.rowstart[i];
        const uint32_t len = cnt_s[i];
        uint32_t out = 0, own = 0;
        for (uint32_t k0 = 0; k0 < len; k0 += TPP) {
            const uint32_t k = k0 + (uint32_t)gl;
            bool in = false, io = false;
            uint32_t w = 0;
            if (k < len) {
                w = col_s[rs + k];
                const uint32_t j = w & kColMask;
                const float4 q = a.r4[j];
                const uint32_t code = w >> kColBits;
                float dx, dy, dz;
                int D;
                if (code != kFarCode) {
                    const float4 e = stencil_offset(code);
                    if (zmode) rel_dx<1>(e, s_f, sz_f, lz_f, (float)P->ncz, ri.x, ri.y, ri.z, q, dx, dy, dz);
                    else rel_dx<0>(e, s_f, sz_f, lz_f, (float)P->ncz, ri.x, ri.y, ri.z, q, dx, dy, dz);
                    D = Dcode;
                } else {
                    const uint32_t cj = a.g.cellxyz[j];
                    rel_dx_far(ci, cj, s_f, sz_f, lz_f, ri.x, ri.y, ri.z, q, dx, dy, dz);
                    const int ax = abs((int)(cj & 255u) - (int)(ci & 255u));
                    const int ay = abs((int)((cj >> 8) & 255u) - (int)((ci >> 8) & 255u));
                    const int az = abs((int)(cj >> 16) - (int)(ci >> 16));
                    D = max(ax, max(ay, az));
                }
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                const float T = fmaxf(Ti, q.w);
                const float tol = guard_tol(sh, D);
                const float fhi = 1.0f + tol;
                if (r2 <= T * fhi) {
                    const int d = pair_decision(a, P, i, j, r2, Ti, T, 1.0f - tol, fhi);
                    in = d & 1;
                    io = (d >> 1) & 1;
                }
            }
            const unsigned bin = __ballot_sync(gmask, in) & gmask;
            const unsigned bio = __ballot_sync(gmask, io) & gmask;
            if (in) a.col[rs + out + (uint32_t)__popc(bin & below)] = w;
            out += (uint32_t)__popc(bin);
            own += (uint32_t)__popc(bio);
        }
        if (gl == 0) {
            a.cnt[i] = out;
            a.nown[i] = own;
            listed += out;
        }
    }
    for (int o = 16; o > 0; o >>= 1) listed += __shfl_xor_sync(0xffffffffu, listed, o);
    if (lane == 0 && listed) {
        const unsigned long long before = atomicAdd(&a.pool_used[1], listed);
        if (before + listed > (unsigned long long)a.max_pairs) atomicOr(a.status, kStOverflow);
    }
}

int launch_nb_filter(const Launch& L, const NbArgs& a, const uint32_t* col_s, const uint32_t* cnt_s)
{
    if (a.n <= 0) return 0;
    constexpr int TPP = 32;
    int64_t blocks = (a.n * TPP + 255) / 256;
    if (blocks > (int64_t)L.sms * 8) blocks = (int64_t)L.sms * 8;
    k_nb_filter<TPP><<<(unsigned)blocks, 256, 0, L.stream>>>(a, col_s, cnt_s);
    return 1;
}

// canonical CSR: row i of the pool, columns without the stencil bits, to
// out[off[i] ..]; one warp per row
__global__ void k_canonical_rows(int64_t n, const unsigned long long* rowstart, const uint32_t* cnt,
                                 const uint64_t* off, const uint32_t* col, uint32_t* out)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += nw) {
        const unsigned long long r0 = rowstart[i];
        const uint64_t o = off[i];
        for (uint32_t k = lane; k < cnt[i]; k += 32) out[o + k] = col[r0 + k] & kColMask;
    }
}

int launch_canonical_rows(const Launch& L, int64_t n, const unsigned long long* rowstart,
                          const uint32_t* cnt, const uint64_t* off, const uint32_t* col, uint32_t* out)
{
    if (n <= 0) return 0;
    int64_t blocks = (n * 32 + 255) / 256;
    if (blocks > (int64_t)L.sms * 16) blocks = (int64_t)L.sms * 16;
    k_canonical_rows<<<(unsigned)blocks, 256, 0, L.stream>>>(n, rowstart, cnt, off, col, out);
    return 1;
}

}  // namespace sphg
