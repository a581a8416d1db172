// c = S v without any device allocation, for callers that cannot call cudaMalloc.
//
// Some callers of this library may not allocate device memory at the point where they need a sketch: code running
// inside a region whose memory plan is fixed in advance (a captured or replayed sequence of work, a real-time loop
// with a no-allocation rule), or a host application whose device memory is owned by another allocator or memory
// pool that must not be bypassed.  A solver handle allocates (CSR copy, gather lists, workspaces), so this entry
// point needs none: the per-block partial sums live in one file-scope static __device__ array of fixed size, which
// every GPU that loads the library holds until the process exits.  The caller passes only its input and output.
//
// The embedding is the same one a handle created with the same seed applies (same SplitMix64 draw rule, see
// sketch_column), so results agree with sfgmres_sketch_apply up to summation rounding.  A CTA takes chunks of at most 992
// columns, draws their rows on the fly, and sums a chunk's terms exactly in 64-bit fixed point relative to the chunk's
// largest exponent with shared-memory integer atomics (integer addition is order independent, so the result is
// deterministic); at most 992 terms of at most 2^53 meet in a sum, so none can overflow and no count of the terms is
// needed.  The chunk sums are added in chunk order into the CTA's partial, the partials in a fixed order.
//
// What bounds it: the draws (two 64-bit mixes per nonzero) and the shared-memory atomics, both in every SM at once; the
// chunks of at most two CTAs per SM keep the second kernel's sums short, and that kernel reads 32 sketch rows of a partial per
// warp with 16 warps over the partials.  n = 1,000,003, s = 240, zeta = 8: 43 + 5 us; with every row drawn twice (once to count the
// terms) into local memory, 977 partials and a thread per row of the second kernel, 102 + 72 us.
#include "../../include/sfgmres.h"
#include "common.cuh"

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>

namespace sfg {

// Largest number of (block, sketch row) partials the static scratch holds: 2^20 doubles = 8 MiB.
constexpr int64_t kNoallocScratch = int64_t(1) << 20;
constexpr int64_t kNoallocMaxCols = 65536;  // with 2^20 / s partials, the largest n (a documented limit)
constexpr int kChunkCols = 992;           // columns per chunk, at most: fewer than 1023 terms per sum
constexpr int kChunkMin = 128;            // and at least (short vectors: more CTAs)
constexpr int kNoallocCtas = 304;         // CTAs of the partials kernel, at most (two per SM)

static __device__ __align__(256) double g_noalloc_scratch[kNoallocScratch];

void set_global_error(const std::string& msg);  // api.cu: the message sfgmres_last_error(NULL) returns

// ZETA: nonzeros per column as a compile-time count (rows and signs in registers), 0: any count.
template <int ZETA>
__global__ void __launch_bounds__(512, 2)
    k_noalloc_partials(int64_t n, int chunk, int s, int zeta_any, uint64_t seed, const double* __restrict__ v,
                       double* __restrict__ part) {
    extern __shared__ unsigned char smem_raw[];
    long long* acc = reinterpret_cast<long long*>(smem_raw);  // [s] the chunk's sums
    double* tot = reinterpret_cast<double*>(acc + s);         // [s] the CTA's partial
    __shared__ int wmax[2][16];
    const int zeta = ZETA > 0 ? ZETA : zeta_any;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int r = threadIdx.x; r < s; r += blockDim.x) {
        acc[r] = 0;
        tot[r] = 0.0;
    }
    int par = 0;  // wmax alternates, so that a warp may write the next chunk's while another reads this one's
    for (int64_t c0 = (int64_t)blockIdx.x * chunk; c0 < n; c0 += (int64_t)gridDim.x * chunk, par ^= 1) {
        const int len = (int)min((int64_t)chunk, n - c0);
        double x[2];  // chunk <= 2 x 512 columns: this thread's
        int emax = 1;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int j = u * (int)blockDim.x + (int)threadIdx.x;
            x[u] = (j < len) ? v[c0 + j] : 0.0;
            emax = max(emax, exp_of(x[u]));
        }
        emax = (int)__reduce_max_sync(0xffffffffu, (unsigned)emax);
        if (lane == 0) wmax[par][warp] = emax;
        __syncthreads();  // also: acc and tot are set
        int Eb = 1;
        for (int q = 0; q < nw; ++q) Eb = max(Eb, wmax[par][q]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int j = u * (int)blockDim.x + (int)threadIdx.x;
            if (j >= len) break;
            const long long q = to_fixed(x[u], Eb, 0);
            int rows[ZETA > 0 ? ZETA : kMaxZeta], neg[ZETA > 0 ? ZETA : kMaxZeta];
            if constexpr (ZETA > 0) sketch_column_n<ZETA>(seed, c0 + j, s, rows, neg);
            else sketch_column(seed, c0 + j, zeta, s, rows, neg);
#pragma unroll
            for (int l = 0; l < zeta; ++l)
                atomicAdd(reinterpret_cast<unsigned long long*>(acc + rows[l]), (unsigned long long)(neg[l] ? -q : q));
        }
        __syncthreads();
        const double unit = ldexp(1.0, Eb - 1075);
        for (int r = threadIdx.x; r < s; r += blockDim.x) {
            tot[r] += (Eb >= 2047) ? (double)NAN : (double)acc[r] * unit;
            acc[r] = 0;  // the next chunk's atomics come after its first barrier
        }
    }
    for (int r = threadIdx.x; r < s; r += blockDim.x) part[(int64_t)blockIdx.x * s + r] = tot[r];
}

// a + b as a rounded sum and what the rounding took away.
__device__ __forceinline__ void two_sum(double& a, double& lost, double b) {
    const double t = a + b, bv = t - a;
    lost += (a - (t - bv)) + (b - bv);
    a = t;
}

// c[r] = scale * the sum of part[b*s + r] over b: a CTA per 32 sketch rows (a lane each), warp w sums the partials w, w + 16,
// ... and the warps' sums are added in order.
//
// CARRY, for vectors of up to 32,768 entries, whose partials are of 128 columns each: the warps' sums are joined by a tree that
// carries what its roundings lose.  Added one after another such partials cost up to 1.4 times the error of sums that are exact
// over 1024 columns (3,000 entries; 1.2 at 10,000, 1.0 at 30,000, less beyond, where chunks are longer).  Back to back, a call
// of 2,000 entries takes 11.1 us against 10.7, of 32,000 16.4 against 14.3; longer ones are as before (n = 1,000,003, s = 240: 51.2,
// and 71.8 with every addition carrying its loss).
constexpr int64_t kCarryCols = 32768;

template <bool CARRY>
__global__ void __launch_bounds__(512) k_noalloc_reduce(int nblk, int s, double scale, const double* __restrict__ part,
                                                        double* __restrict__ c) {
    __shared__ double sh[16][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = blockIdx.x * 32 + lane;
    double a = 0.0;
    if (r < s) {
#pragma unroll 8
        for (int b = warp; b < nblk; b += 16) a += part[(int64_t)b * s + r];
    }
    sh[warp][lane] = a;
    if constexpr (!CARRY) {
        __syncthreads();
        if (warp == 0 && r < s) {
            for (int w = 1; w < 16; ++w) a += sh[w][lane];
            c[r] = scale * a;
        }
    } else {
        __shared__ double sl[16][32];
        double lost = 0.0;
#pragma unroll
        for (int h = 8; h > 0; h >>= 1) {  // a level reads [h, 2h) and the next writes below h: one barrier each
            __syncthreads();
            if (warp >= h) continue;
            const double t = sh[warp + h][lane];
            if (h < 8) lost += sl[warp + h][lane];
            two_sum(a, lost, t);
            sh[warp][lane] = a;
            sl[warp][lane] = lost;
        }
        if (warp == 0 && r < s) c[r] = scale * (isfinite(a) ? a + lost : a);
    }
}

// Dynamic shared memory of k_noalloc_partials for s sketch rows: a 64-bit sum and an FP64 partial per row.
static size_t partials_smem(int s) { return (size_t)s * (sizeof(long long) + sizeof(double)); }

using PartialsKernel = void (*)(int64_t, int, int, int, uint64_t, const double*, double*);
static PartialsKernel partials_kernel(int zeta) {
    switch (zeta) {
        case 1: return k_noalloc_partials<1>;
        case 2: return k_noalloc_partials<2>;
        case 4: return k_noalloc_partials<4>;
        case 8: return k_noalloc_partials<8>;
        default: return k_noalloc_partials<0>;
    }
}

// Once per device, with that device current: look up the device address of the scratch array (cudaGetSymbolAddress;
// in host code the array's name is only a host-side stand-in) and allow k_noalloc_partials the dynamic shared memory
// of the largest sketch (4096 rows need 64 KiB, above the default limit).  Both results are cached per device.
static cudaError_t device_setup(double** out) {
    static std::mutex mu;
    static double* cache[64] = {nullptr};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (!cache[dev]) {
        for (int z : {0, 1, 2, 4, 8}) {
            e = cudaFuncSetAttribute((const void*)partials_kernel(z), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)partials_smem(kMaxS));
            if (e != cudaSuccess) return e;
        }
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        cache[dev] = static_cast<double*>(p);
    }
    *out = cache[dev];
    return cudaSuccess;
}

// Launch with the error of this launch alone as the result (the launch API returns it; an error left behind by
// unrelated earlier work is neither reported nor cleared here).  A failed launch's own error is cleared.
template <typename... KArgs, typename... Args>
static cudaError_t launch(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                          Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

}  // namespace sfg

extern "C" int sfgmres_sketch_apply_noalloc(int64_t n, int32_t s, int32_t zeta, uint64_t sketch_seed,
                                            const double* v, double* c, void* stream) {
    using namespace sfg;
    if (!v || !c) {
        set_global_error("sfgmres_sketch_apply_noalloc: v and c must not be NULL");
        return SFGMRES_ERR_INVALID_ARG;
    }
    if (n < 1 || n > INT32_MAX) {
        set_global_error("sfgmres_sketch_apply_noalloc: n must be in [1, 2^31-1]");
        return SFGMRES_ERR_INVALID_ARG;
    }
    if (zeta < 1 || zeta > kMaxZeta || s < zeta || s > kMaxS) {
        set_global_error("sfgmres_sketch_apply_noalloc: need 1 <= zeta <= 16 and zeta <= s <= 4096");
        return SFGMRES_ERR_INVALID_ARG;
    }
    const int64_t max_blocks = kNoallocScratch / s;
    const int64_t max_n = max_blocks * kNoallocMaxCols;
    if (n > max_n) {
        set_global_error("sfgmres_sketch_apply_noalloc: n exceeds the static scratch limit (n <= 65536 * floor(2^20"
                         " / s) = " + std::to_string(max_n) + " for s = " + std::to_string(s) + ")");
        return SFGMRES_ERR_INVALID_ARG;
    }
    double* part = nullptr;
    cudaError_t e = device_setup(&part);
    if (e != cudaSuccess) {
        set_global_error(std::string("sfgmres_sketch_apply_noalloc: device set-up (cudaFuncSetAttribute / "
                                     "cudaGetSymbolAddress): ") + cudaGetErrorString(e));
        return SFGMRES_ERR_CUDA;
    }
    int64_t chunk = (n + kNoallocCtas - 1) / kNoallocCtas;
    chunk = std::min<int64_t>(kChunkCols, std::max<int64_t>(kChunkMin, (chunk + 31) / 32 * 32));
    const int64_t nblk = std::min<int64_t>(std::min<int64_t>((n + chunk - 1) / chunk, kNoallocCtas), max_blocks);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    e = launch(partials_kernel(zeta), (unsigned)nblk, 512, partials_smem(s), st, n, (int)chunk, (int)s, (int)zeta,
               sketch_seed, v, part);
    if (e != cudaSuccess) {
        set_global_error(std::string("sfgmres_sketch_apply_noalloc: launch of the block partials kernel: ") +
                         cudaGetErrorString(e));
        return SFGMRES_ERR_CUDA;
    }
    e = launch(n <= kCarryCols ? k_noalloc_reduce<true> : k_noalloc_reduce<false>, (unsigned)((s + 31) / 32), 512, 0, st,
               (int)nblk, (int)s, 1.0 / std::sqrt((double)zeta), (const double*)part, c);
    if (e != cudaSuccess) {
        set_global_error(std::string("sfgmres_sketch_apply_noalloc: launch of the reduction kernel: ") +
                         cudaGetErrorString(e));
        return SFGMRES_ERR_CUDA;
    }
    return SFGMRES_OK;
}
