// sph_pairs.cu -- the SPH pair sums over the CSR neighbour lists (Sec. 3):
//   density  rho_i = m_i W(0, h_i) + sum_j m_j W(r_ij, h_i)        (R1, Eq. 2)
//   EOS      P = (gamma - 1) rho u,  c = sqrt(gamma P / rho)        (R9)
//   momentum a_i  = -sum_j m_j (A_i + A_j + Pi_ij) grad_i Wbar_ij   (R4)
//   energy   du_i =  sum_j m_j (A_i + Pi_ij / 2) v_ij . grad_i Wbar_ij (R6)
// with A = P / rho^2, Wbar_ij = (W(r,h_i) + W(r,h_j)) / 2 and the Monaghan
// viscosity Pi_ij = (-alpha cbar mu + beta mu^2) / rhobar for approaching
// pairs, mu = hbar v_ij . x_ij / (r^2 + eps hbar^2) (R5).
//
// Wendland kernel (Eq. 2, 1/h^3 restored): with w = 1/(2h) and
// q = 1 - r w = 1 - v/2,
//   W(r, h)         = sigma/h^3 q^4 (5 - 4 q)          (2v + 1 = 5 - 4q)
//   grad_i W(r, h)  = -160 sigma w^5 q^3 (x_i - x_j)   (5 sigma / h^5 = 160 sigma w^5)
// so grad_i Wbar_ij = -80 sigma (w_i^5 q_i^3 + w_j^5 q_j^3) (x_i - x_j), and the
// factor 80 sigma = 105/pi is applied once per particle.
//
// One group of TPP lanes per particle strides over the particle's row; the
// group reduces its partial sums with shuffles.  Mixed precision: positions
// are FP32 offsets from the particle's cell origin, the column word carries
// the stencil cell so x_i - x_j = (o_i - o_j) - dc s exactly up to FP32
// rounding of o (a neighbour beyond the 5 x 5 x 5 stencil, kFarCode, takes dc
// from both particles' cell coordinates); sums are Kahan-compensated FP32.
// FP64 path: every pair operation in double.
#include "sph_pairmath.cuh"

namespace sphg {


#ifndef SPH_ROW_PREFETCH
#define SPH_ROW_PREFETCH 1              // L2 prefetch of the next particle's row
#endif

// The list words stream from HBM (the pool is far larger than L2) and are
// read with the streaming hint (evict first), which leaves L2 to the
// neighbour records every row gathers.  Each
// group asks L2 for the row of the particle it takes next -- the group's lanes
// cover it in 128-byte lines -- while it works on the current one; the start
// of that row was read one particle earlier, so the request does not wait.
struct RowAhead {
    unsigned long long start;
    uint32_t len;
};

__device__ __forceinline__ RowAhead row_ahead_read(const PairArgs& a, int64_t i)
{
    RowAhead r = {0ull, 0u};
    if (i < a.n) {
        r.start = a.rowstart[i];
        r.len = a.cnt[i];
    }
    return r;
}

// the positions [kb, ke) a launch covers: every particle, or a range of
// row-length bins of the order
__device__ __forceinline__ void pair_range(const PairArgs& a, int64_t& kb, int64_t& ke)
{
    if (a.order) {
        kb = a.bounds[a.bin_lo];
        ke = a.bounds[a.bin_hi + 1];
    } else {
        kb = 0;
        ke = a.n;
    }
}

// the particle at position k (a.n past the range: no particle)
__device__ __forceinline__ int64_t pair_at(const PairArgs& a, int64_t k, int64_t ke)
{
    if (k >= ke) return a.n;
    return a.order ? (int64_t)a.order[k] : k;
}

template <int TPP>
__device__ __forceinline__ void row_ahead_prefetch(const PairArgs& a, const RowAhead& r, int gl)
{
#if SPH_ROW_PREFETCH
    for (uint32_t o = (uint32_t)gl * 32u; o < r.len; o += TPP * 32u)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.col + r.start + o));
#endif
}

// The four words a lane takes at a time from word k on: consecutive ones (one
// 16-byte load; rows start on 32-byte boundaries and are reserved in multiples
// of 8 words, so it never leaves the reservation), or every STEP-th, so that
// the lanes of a group take consecutive words, which are mostly consecutive
// neighbours in the records.  The momentum sum, with three gathers a word,
// gains by that from four lanes on (1 M irregular particles at 4 / 8 / 16
// lanes: 920 / 914 / 1020 -> 889 / 851 / 931 us; two lanes lose 4 %); the
// density sum, with one, does not.
template <int STEP>
__device__ __forceinline__ uint4 row_words(const uint32_t* row, uint32_t len, uint32_t k)
{
    if (STEP == 1) return k < len ? __ldcs(reinterpret_cast<const uint4*>(row + k)) : make_uint4(0u, 0u, 0u, 0u);
    uint4 w;
    w.x = k < len ? __ldcs(row + k) : 0u;
    w.y = k + STEP < len ? __ldcs(row + k + STEP) : 0u;
    w.z = k + 2 * STEP < len ? __ldcs(row + k + 2 * STEP) : 0u;
    w.w = k + 3 * STEP < len ? __ldcs(row + k + 3 * STEP) : 0u;
    return w;
}
// how many of them the row has, k < len
template <int STEP>
__device__ __forceinline__ uint32_t row_valid(uint32_t len, uint32_t k)
{
    return min((len - k + STEP - 1u) / STEP, 4u);
}

// ---------------------------------------------------------------------------
// density + EOS, mixed precision
// ---------------------------------------------------------------------------
// the row of one particle: plain FP32 weights m_j W-shape(r), Kahan sum.  A
// lane takes the row in chunks of four words (one 16-byte load; rows start on
// 32-byte boundaries and are reserved in multiples of 8 words, so a chunk
// never leaves the reservation), loaded one chunk ahead of its use, and
// issues the chunk's four record gathers together.  Words past the row end
// in the last chunk are not used as indices.
template <int TPP, int ZW, int KERN, bool GH>
__device__ __forceinline__ void density_row(const PairArgs& a, const uint32_t* row, uint32_t len,
                                            int gl, const PairSide& I, float inv2h, float& sum, float& comp,
                                            float& sumd, float& compd)
{
    const int kn = a.kernel_n;
    const PairSrc src = pair_src(a);
    uint32_t k = 4u * (uint32_t)gl;
    uint4 w = row_words<1>(row, len, k);
    for (; k < len; k += 4u * TPP) {
        const uint4 wn = row_words<1>(row, len, k + 4u * TPP);
        const uint32_t nv = row_valid<1>(len, k);
        const uint32_t cw[4] = {w.x, nv > 1u ? w.y : w.x, nv > 2u ? w.z : w.x, nv > 3u ? w.w : w.x};
        float4 q[4];
#pragma unroll
        for (int u = 0; u < 4; u++) q[u] = src.r5[cw[u] & kColMask];
        float dx[4], dy[4], dz[4];
        // all four words within the stencil (all but the few pairs with a big
        // particle): the stencil offsets without the per-pair branch
        if (((cw[0] >> kColBits) != kFarCode) & ((cw[1] >> kColBits) != kFarCode) &
            ((cw[2] >> kColBits) != kFarCode) & ((cw[3] >> kColBits) != kFarCode)) {
#pragma unroll
            for (int u = 0; u < 4; u++)
                rel_dx<ZW>(stencil_offset(cw[u] >> kColBits), I.s_f, I.sz_f, I.lz_f, I.ncz_f, I.ri.x, I.ri.y, I.ri.z, q[u], dx[u],
                           dy[u], dz[u]);
        } else {
#pragma unroll
            for (int u = 0; u < 4; u++) col_dx<ZW>(src, I, cw[u], q[u], dx[u], dy[u], dz[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; u++)
            if ((uint32_t)u < nv) density_term<KERN, GH>(dx[u], dy[u], dz[u], inv2h, kn, q[u].w, sum, comp, sumd, compd);
        w = wn;
    }
}

#ifndef SPH_DEN_MINB
#define SPH_DEN_MINB 4                  // resident 256-thread CTAs per SM the registers are sized for
#endif
template <int TPP, int KERN, bool GH>
__global__ void __launch_bounds__(256, SPH_DEN_MINB) k_density_mixed(PairArgs a)
{
    wait_before();
    const float kb8 = (float)(8.0 * a.kb);
    if (*a.status & kStBad) return;
    const GroupIdx G = group_idx<TPP>();
    const int64_t gs = ((int64_t)gridDim.x * blockDim.x) / TPP;
    const float gam = (float)a.gamma;
    int64_t kb, ke;
    pair_range(a, kb, ke);
    const int64_t k0 = kb + ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / TPP;
    RowAhead ahead = row_ahead_read(a, pair_at(a, k0 + gs, ke));
    for (int64_t k = k0; k < ke; k += gs) {
        const int64_t i = pair_at(a, k, ke);
        row_ahead_prefetch<TPP>(a, ahead, G.gl);
        ahead = row_ahead_read(a, pair_at(a, k + 2 * gs, ke));
        const PatchDev* P = a.pd + a.patch_of[i];
        const PairSide I = pair_side(a, P, i);
        const float inv2h = a.r.rv[i].w;                   // 1 / (2 h_i)
        const uint32_t* row = a.col + a.rowstart[i];
        const uint32_t len = a.cnt[i];
        float sum = 0.0f, comp = 0.0f, sumd = 0.0f, compd = 0.0f;
        if (P->zmode) density_row<TPP, 1, KERN, GH>(a, row, len, G.gl, I, inv2h, sum, comp, sumd, compd);
        else density_row<TPP, 0, KERN, GH>(a, row, len, G.gl, I, inv2h, sum, comp, sumd, compd);
        group_kahan_reduce<TPP>(sum, comp, G.gmask);
        if (GH) group_kahan_reduce<TPP>(sumd, compd, G.gmask);
        if (G.gl == 0) density_finish<GH>(a, i, I.ri.w, inv2h, kb8, gam, sum, comp, sumd, compd);
    }
}

// ---------------------------------------------------------------------------
// density + EOS, FP64
// ---------------------------------------------------------------------------
template <int TPP, int KERN, bool GH>
__global__ void __launch_bounds__(256) k_density_fp64(PairArgs a)
{
    wait_before();
    const int kn = a.kernel_n;
    if (*a.status & kStBad) return;
    const GroupIdx G = group_idx<TPP>();
    const int64_t gs = ((int64_t)gridDim.x * blockDim.x) / TPP;
    int64_t kb, ke;
    pair_range(a, kb, ke);
    // A group sums TPP particles, one after the other, before its lanes finish
    // one each: the epilogue's divisions and square root, some 60 operations on
    // the FP64 pipe, cost a warp the same for one lane as for all (125,000
    // particles at 8 lanes: 606 -> 516 us).
    for (int64_t k0 = kb + ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / TPP; k0 < ke; k0 += gs * TPP) {
        int64_t mine = -1;
        double sum_i = 0.0, sumd_i = 0.0;
        for (int b = 0; b < TPP; b++) {
            const int64_t k = k0 + b * gs;
            if (k >= ke) break;
            const int64_t i = pair_at(a, k, ke);
            const double xi = a.s.x[i], yi = a.s.y[i], zi = a.s.z[i], lz = a.pd[a.patch_of[i]].lz;
            const double w = a.f.w[i];
            const uint32_t* row = a.col + a.rowstart[i];
            const uint32_t len = a.cnt[i];
            double sum = 0.0, sumd = 0.0;
            for (uint32_t q = G.gl; q < len; q += TPP)
                density_pair_fp64<KERN, GH>(a, xi, yi, zi, w, lz, kn, __ldcs(row + q) & kColMask, sum, sumd);
            sum = group_sum<TPP>(sum, G.gmask);
            if (GH) sumd = group_sum<TPP>(sumd, G.gmask);
            if (G.gl == b) {
                mine = i;
                sum_i = sum;
                sumd_i = sumd;
            }
        }
        if (mine >= 0) density_finish_fp64<GH>(a, mine, sum_i, sumd_i);
    }
}

// ---------------------------------------------------------------------------
// momentum + energy, mixed precision
// ---------------------------------------------------------------------------
// The row in chunks of four words: a lane loads its chunk (row_words) one
// chunk ahead of its use, sums the chunk's four pair terms plainly and adds that sum with Kahan
// compensation (the plain sum of four terms errs by at most 3 eps times their
// magnitudes, the order of one term's own rounding).
template <int TPP, int ZW, int KERN, bool GH>
__device__ __forceinline__ void momentum_row(const PairArgs& a, const uint32_t* row, uint32_t len,
                                             int gl, const PairSide& I, const float4& vi, const float4& ti, float wi5,
                                             const MomConst& K, MomAcc& A)
{
    const int kn = a.kernel_n;
    const PairSrc src = pair_src(a);
    constexpr int kStep = TPP >= 4 ? TPP : 1;
    uint32_t k = kStep == 1 ? 4u * (uint32_t)gl : (uint32_t)gl;
    uint4 w = row_words<kStep>(row, len, k);
    for (; k < len; k += 4u * TPP) {
        const uint4 wn = row_words<kStep>(row, len, k + 4u * TPP);
        const uint32_t cws[4] = {w.x, w.y, w.z, w.w};
        const uint32_t nv = row_valid<kStep>(len, k);
        float bx, by, bz, bu;
        momentum_chunk<ZW, KERN, GH>(src, I, vi, ti, wi5, K, kn, cws, nv, bx, by, bz, bu, GlobalRecs{src});
        mom_acc_add(A, bx, by, bz, bu);
        w = wn;
    }
}

// Resident 256-thread CTAs per SM that the registers are sized for.  The packed
// pairs of the Wendland kernel need 112 registers (at 80 they spill: 10^6
// particles 512 -> 557 us).  The scalar loop of the Sinc kernel and of the
// grad-h form needs 100 to 105, waits on its gathers and special functions,
// and gains more from the third CTA than its 8 bytes of spill cost: 250,000
// particles, Sinc 209 -> 189 us, Wendland with grad-h 148 -> 127 us; with h
// varying 10 to 1, 491 -> 420 us and 322 -> 261 us.
template <int KERN, bool GH>
constexpr int mom_minb()
{
    return KERN == SPH_KERNEL_WENDLAND && !GH ? 2 : 3;
}

template <int TPP, int KERN, bool GH>
__global__ void __launch_bounds__(256, mom_minb<KERN, GH>()) k_momentum_mixed(PairArgs a)
{
    wait_before();
    const float gscale = (float)KernF<KERN>::grad_scale(a.kb, a.kernel_n);
    if (*a.status & kStBad) return;
    const GroupIdx G = group_idx<TPP>();
    const int64_t gs = ((int64_t)gridDim.x * blockDim.x) / TPP;
    const MomConst K = {0.25f * (float)a.eps, 0.5f * (float)a.beta, 0.5f * (float)a.alpha};
    int64_t kb, ke;
    pair_range(a, kb, ke);
    const int64_t k0 = kb + ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / TPP;
    RowAhead ahead = row_ahead_read(a, pair_at(a, k0 + gs, ke));
    for (int64_t k = k0; k < ke; k += gs) {
        const int64_t i = pair_at(a, k, ke);
        row_ahead_prefetch<TPP>(a, ahead, G.gl);
        ahead = row_ahead_read(a, pair_at(a, k + 2 * gs, ke));
        const PatchDev* P = a.pd + a.patch_of[i];
        const PairSide I = pair_side(a, P, i);
        const float4 vi = a.r.rv[i];
        const float4 ti = a.r.rt[i];
        const float wi2 = vi.w * vi.w;
        const float wi5 = wi2 * wi2 * vi.w;
        const uint32_t* row = a.col + a.rowstart[i];
        const uint32_t len = a.cnt[i];
        MomAcc A = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (P->zmode) momentum_row<TPP, 1, KERN, GH>(a, row, len, G.gl, I, vi, ti, wi5, K, A);
        else momentum_row<TPP, 0, KERN, GH>(a, row, len, G.gl, I, vi, ti, wi5, K, A);
        group_kahan_reduce<TPP>(A.sx, A.cx, G.gmask);
        group_kahan_reduce<TPP>(A.sy, A.cy, G.gmask);
        group_kahan_reduce<TPP>(A.sz, A.cz, G.gmask);
        group_kahan_reduce<TPP>(A.su, A.cu, G.gmask);
        if (G.gl == 0) momentum_finish(a, i, gscale, A);
    }
}

// ---------------------------------------------------------------------------
// momentum + energy, FP64
// ---------------------------------------------------------------------------
template <int TPP, int KERN, bool GH>
__global__ void __launch_bounds__(256) k_momentum_fp64(PairArgs a)
{
    wait_before();
    if (*a.status & kStBad) return;
    const GroupIdx G = group_idx<TPP>();
    const int64_t gs = ((int64_t)gridDim.x * blockDim.x) / TPP;
    const int kn = a.kernel_n;
    const double S80 = KernF<KERN>::grad_scale(a.kb, kn);
    int64_t kb, ke;
    pair_range(a, kb, ke);
    for (int64_t k = kb + ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / TPP; k < ke; k += gs) {
        const int64_t i = pair_at(a, k, ke);
        const PatchDev* P = a.pd + a.patch_of[i];
        const SideD I = side_fp64(a, P, i);
        const uint32_t* row = a.col + a.rowstart[i];
        const uint32_t len = a.cnt[i];
        MomAccD S = {0.0, 0.0, 0.0, 0.0};
        for (uint32_t k = G.gl; k < len; k += TPP) momentum_pair_fp64<KERN, GH>(a, I, __ldcs(row + k) & kColMask, kn, S);
        S.ax = group_sum<TPP>(S.ax, G.gmask);
        S.ay = group_sum<TPP>(S.ay, G.gmask);
        S.az = group_sum<TPP>(S.az, G.gmask);
        S.du = group_sum<TPP>(S.du, G.gmask);
        if (G.gl == 0) momentum_finish_fp64(a, i, S80, S);
    }
}

#define SPH_DISPATCH_TPP(KERNEL, KERN, GH, tpp, g, L, a)                                \
    switch (tpp) {                                                                      \
    case 1: launch_next(KERNEL<1, KERN, GH>, (g).x, (g).y, 0, (L).stream, a); break;    \
    case 2: launch_next(KERNEL<2, KERN, GH>, (g).x, (g).y, 0, (L).stream, a); break;    \
    case 4: launch_next(KERNEL<4, KERN, GH>, (g).x, (g).y, 0, (L).stream, a); break;    \
    case 16: launch_next(KERNEL<16, KERN, GH>, (g).x, (g).y, 0, (L).stream, a); break;  \
    case 32: launch_next(KERNEL<32, KERN, GH>, (g).x, (g).y, 0, (L).stream, a); break;  \
    default: launch_next(KERNEL<8, KERN, GH>, (g).x, (g).y, 0, (L).stream, a); break;   \
    }
#define SPH_DISPATCH_GH(KERNEL, KERN, tpp, g, L, a)                                     \
    if ((a).grad_h) {                                                                   \
        SPH_DISPATCH_TPP(KERNEL, KERN, true, tpp, g, L, a);                             \
    } else {                                                                            \
        SPH_DISPATCH_TPP(KERNEL, KERN, false, tpp, g, L, a);                            \
    }
#define SPH_DISPATCH(KERNEL, tpp, g, L, a)                                              \
    if ((a).kernel == SPH_KERNEL_SINC) {                                                \
        SPH_DISPATCH_GH(KERNEL, SPH_KERNEL_SINC, tpp, g, L, a);                         \
    } else {                                                                            \
        SPH_DISPATCH_GH(KERNEL, SPH_KERNEL_WENDLAND, tpp, g, L, a);                     \
    }

// {blocks, threads}: blocks of 256 threads that stride over the particles,
// of 64 while 256 would leave the SMs unevenly filled (8000 particles at 8
// lanes are 250 blocks of 256 for 152 SMs: some get two, some one)
// per_sm: blocks of 256 for each SM.  The mixed sums, whose two to four
// resident blocks hide latency, are best at 8 (from 16 on 2 to 8 % slower: a
// block is done before its prefetches pay); the FP64 momentum sum is bound by
// the FP64 pipe and loses only in its last round, so it takes 16 (125,000
// particles 1234 -> 1196 us, 64,000 with h 10 to 1 1375 -> 1346 us, 10^6 as
// before).
static uint2 pair_grid(const Launch& L, int64_t n, int tpp, int per_sm = 8)
{
    const int64_t cap = (int64_t)L.sms * per_sm;
    int64_t blocks = (n * tpp + 255) / 256;
    if (blocks < cap) return make_uint2((unsigned)((n * tpp + 63) / 64), 64u);
    return make_uint2((unsigned)cap, 256u);
}

int launch_density(const Launch& L, const PairArgs& a, int tpp, int mixed)
{
    if (a.n <= 0) return 0;
    const uint2 g = pair_grid(L, a.n, tpp);
    if (mixed) {
        SPH_DISPATCH(k_density_mixed, tpp, g, L, a);
    } else {
        SPH_DISPATCH(k_density_fp64, tpp, g, L, a);
    }
    return 1;
}

int launch_momentum(const Launch& L, const PairArgs& a, int tpp, int mixed)
{
    if (a.n <= 0) return 0;
    const uint2 g = pair_grid(L, a.n, tpp, mixed ? 8 : 16);
    if (mixed) {
        SPH_DISPATCH(k_momentum_mixed, tpp, g, L, a);
    } else {
        SPH_DISPATCH(k_momentum_fp64, tpp, g, L, a);
    }
    return 1;
}

// One launch per run of octaves that share a lanes-per-particle value (the
// bin sizes stay on the device, so every launch takes the full grid and
// strides over its range; a launch whose range is empty returns at once).
template <class F>
static int binned_launches(PairArgs a, int w, F&& launch_one)
{
    if (a.n <= 0 || !a.order) return 0;
    int launches = 0;
    int o = 0;
    while (o < kPairOctaves) {
        const int t = octave_tpp(o, w);
        int e = o;
        while (e + 1 < kPairOctaves && octave_tpp(e + 1, w) == t) e++;
        a.bin_lo = o;
        a.bin_hi = e;
        launches += launch_one(a, t);
        o = e + 1;
    }
    return launches;
}

int launch_density_binned(const Launch& L, PairArgs a, int w, int mixed)
{
    return binned_launches(a, w, [&](const PairArgs& b, int t) { return launch_density(L, b, t, mixed); });
}

int launch_momentum_binned(const Launch& L, PairArgs a, int w, int mixed)
{
    return binned_launches(a, w, [&](const PairArgs& b, int t) { return launch_momentum(L, b, t, mixed); });
}

}  // namespace sphg
