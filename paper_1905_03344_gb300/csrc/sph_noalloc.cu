// sph_noalloc.cu -- sph_conserved_noalloc: the conserved sums of particle
// arrays the caller already holds on the device, computed without allocating
// anything.  For callers that cannot call cudaMalloc: code running while a
// stream is being captured into a CUDA graph, an allocator-owning host
// framework that forbids other allocations, or a process that has handed
// all device memory to its own pool.
//
// The per-block partial sums live in a file-scope device array of fixed size
// (kStaticBlocks x 8 doubles, 256 KB), which every GPU that loads the
// library keeps until the process exits.  Host code cannot use the array's
// name as a device address; its address is looked up once per device with
// cudaGetSymbolAddress, with that device current, on the first call made on
// that device, and passed to the kernels.  That first call should therefore
// come before any stream capture.  The address is kept for the life of the
// process: a device reset (cudaDeviceReset, or a new primary context on that
// device) makes it stale, and the entry point must not be called on that
// device afterwards.  All calls share the one array: it is
// overwritten by every call (each block writes its own slot before the final
// sum reads it, so nothing needs clearing), and calls whose kernels overlap on
// the GPU race on it.
#include <mutex>
#include <string>

#include "sph_internal.cuh"

namespace {

constexpr int kStaticBlocks = 4096;                   // partial-sum slots
constexpr int kStaticChunk = 4096;                    // particles per slot at the largest n
constexpr int64_t kStaticMaxN = (int64_t)kStaticBlocks * kStaticChunk;  // 16,777,216
constexpr int kMaxDevices = 64;

__device__ __align__(256) double g_partials[kStaticBlocks * 8];

std::mutex g_setup_mutex;
double* g_partials_addr[kMaxDevices] = {};
int g_sms[kMaxDevices] = {};
thread_local std::string g_noalloc_error;

// The 7 sums of a block's share of the particles (chunk of them) into its
// slot (M, Px, Py, Pz, Lz, Ekin, Eint).  Eight blocks for every SM, so that
// the shares are even: bound by the FP64 pipe (12 operations a particle, 45 us
// at 2 M) with 17 us of reads under it.
__global__ void __launch_bounds__(256) k_cons_partials(int64_t n, int64_t chunk, const double* __restrict__ x,
                                                       const double* __restrict__ y, const double* __restrict__ vx,
                                                       const double* __restrict__ vy, const double* __restrict__ vz,
                                                       const double* __restrict__ m, const double* __restrict__ u, double* part)
{
    __shared__ double sh[7][8];
    const int64_t b0 = (int64_t)blockIdx.x * chunk;
    const int64_t b1 = b0 + chunk < n ? b0 + chunk : n;
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    for (int64_t i = b0 + threadIdx.x; i < b1; i += blockDim.x) sphg::cons_accum(x[i], y[i], vx[i], vy[i], vz[i], m[i], u[i], acc);
    acc[5] *= 0.5;
    const double sum = sphg::block_sum7(acc, sh);
    if (threadIdx.x < 7) part[(int64_t)blockIdx.x * 8 + threadIdx.x] = sum;
}

// one block per quantity: the compensated sum of the slots
__global__ void __launch_bounds__(256) k_cons_final(int nblocks, const double* part, double* out)
{
    __shared__ double sh_s[256], sh_c[256];
    const double s = sphg::block_neumaier(part + blockIdx.x, nblocks, 8, sh_s, sh_c);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
}

sph_status noalloc_fail(sph_status s, const std::string& msg)
{
    g_noalloc_error = msg;
    return s;
}

}  // namespace

extern "C" sph_status sph_conserved_noalloc(int64_t n, const double* x, const double* y, const double* vx,
                                            const double* vy, const double* vz, const double* m,
                                            const double* u, double* out, void* cuda_stream)
{
    if (n < 0 || n > kStaticMaxN)
        return noalloc_fail(SPH_EINVAL, "sph_conserved_noalloc: n must be in [0, 16777216] (fixed scratch)");
    if (!out) return noalloc_fail(SPH_EINVAL, "sph_conserved_noalloc: out is NULL");
    if (n > 0 && (!x || !y || !vx || !vy || !vz || !m || !u))
        return noalloc_fail(SPH_EINVAL, "sph_conserved_noalloc: NULL field pointer");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return noalloc_fail(SPH_ECUDA, std::string("sph_conserved_noalloc: no usable device: ") +
                                           cudaGetErrorString(e));
    double* part = nullptr;
    int sms = 1;
    {
        // once per device, with that device current: the device address of the
        // file-scope scratch array
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        if (!g_partials_addr[dev]) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_partials);
            if (e != cudaSuccess || !p)
                return noalloc_fail(SPH_ECUDA, std::string("sph_conserved_noalloc: cudaGetSymbolAddress: ") +
                                                   cudaGetErrorString(e));
            e = cudaDeviceGetAttribute(&g_sms[dev], cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess)
                return noalloc_fail(SPH_ECUDA, std::string("sph_conserved_noalloc: device attribute: ") +
                                                   cudaGetErrorString(e));
            g_partials_addr[dev] = (double*)p;
        }
        part = g_partials_addr[dev];
        sms = g_sms[dev];
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // eight even shares per SM, of 256 particles or more, in the slots there are
    int64_t want = (int64_t)sms * 8 < kStaticBlocks ? (int64_t)sms * 8 : kStaticBlocks;
    const int64_t chunk = ((n + want - 1) / want + 255) / 256 * 256;
    const int nblocks = n > 0 ? (int)((n + chunk - 1) / chunk) : 0;
    if (nblocks > 0) k_cons_partials<<<nblocks, 256, 0, st>>>(n, chunk, x, y, vx, vy, vz, m, u, part);
    k_cons_final<<<7, 256, 0, st>>>(nblocks, part, out);
    e = cudaGetLastError();
    if (e != cudaSuccess)
        return noalloc_fail(SPH_ECUDA, std::string("sph_conserved_noalloc: launch: ") + cudaGetErrorString(e));
    return SPH_OK;
}

extern "C" const char* sph_noalloc_last_error(void) { return g_noalloc_error.c_str(); }
