// Transpose of the CSR matrix (for the adjoint solve A^T x = b) and the pattern gradient used by differentiation.
//
// The transpose is built once on the device: column counts, their prefix sum, a counting fill, then a sort of each
// transposed row by original row index (ties by source position), so the layout -- and hence every sum formed from
// it -- is deterministic.  The source position of every transposed entry is kept, so new values of A are carried
// over by a gather without rebuilding the structure.
#include "kernels.h"

#include <algorithm>

namespace sfg {

__global__ void k_count_cols(int64_t nnz, const int* __restrict__ col, int* __restrict__ counts) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(counts + col[p], 1);
}

// Exclusive prefix sum of counts[0..len) into out[0..len] (single block).
__global__ void k_scan_plain(const int* __restrict__ counts, int* __restrict__ out, int len) {
    __shared__ int sums[1024];
    const int tid = threadIdx.x, T = blockDim.x;
    const int chunk = (len + T - 1) / T;
    const int a = min(len, tid * chunk), bnd = min(len, a + chunk);
    int local = 0;
    for (int i = a; i < bnd; ++i) local += counts[i];
    sums[tid] = local;
    __syncthreads();
    for (int off = 1; off < T; off <<= 1) {
        int v = (tid >= off) ? sums[tid - off] : 0;
        __syncthreads();
        sums[tid] += v;
        __syncthreads();
    }
    int run = sums[tid] - local;
    for (int i = a; i < bnd; ++i) {
        out[i] = run;
        run += counts[i];
    }
    if (tid == T - 1) out[len] = sums[T - 1];
}

__global__ void k_fill_transpose(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                 const int* __restrict__ rpT, int* __restrict__ cursor, int* __restrict__ colT,
                                 int* __restrict__ srcT) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    for (int p = rp[r]; p < rp[r + 1]; ++p) {
        const int c = col[p];
        const int pos = rpT[c] + atomicAdd(cursor + c, 1);
        colT[pos] = r;
        srcT[pos] = p;
    }
}

// Insertion sort of each transposed row by (original row, source position); rows are short.
__global__ void k_sort_rows(int n, const int* __restrict__ rpT, int* __restrict__ colT, int* __restrict__ srcT,
                            int* __restrict__ maxlen) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int a = rpT[r], e = rpT[r + 1];
    for (int i = a + 1; i < e; ++i) {
        const int c = colT[i], sidx = srcT[i];
        int j = i - 1;
        while (j >= a && (colT[j] > c || (colT[j] == c && srcT[j] > sidx))) {
            colT[j + 1] = colT[j];
            srcT[j + 1] = srcT[j];
            --j;
        }
        colT[j + 1] = c;
        srcT[j + 1] = sidx;
    }
    atomicMax(maxlen, e - a);
}

__global__ void k_gather_vals(int64_t nnz, const int* __restrict__ src, const double* __restrict__ val,
                              double* __restrict__ out) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x)
        out[q] = val[src[q]];
}

void launch_transpose(int n, int64_t nnz, const int* rp, const int* col, int* counts, int* rpT, int* colT,
                      int* srcT, int* maxlen, cudaStream_t st) {
    const int g = (int)std::min<int64_t>((nnz + 255) / 256, 152 * 16);
    k_count_cols<<<std::max(g, 1), 256, 0, st>>>(nnz, col, counts);
    k_scan_plain<<<1, 1024, 0, st>>>(counts, rpT, n);
    cudaMemsetAsync(counts, 0, (size_t)n * sizeof(int), st);
    k_fill_transpose<<<(n + 255) / 256, 256, 0, st>>>(n, rp, col, rpT, counts, colT, srcT);
    k_sort_rows<<<(n + 255) / 256, 256, 0, st>>>(n, rpT, colT, srcT, maxlen);
    g_launches += 4;
}

void launch_gather_vals(int64_t nnz, const int* src, const double* val, double* out, cudaStream_t st) {
    const int g = (int)std::min<int64_t>((nnz + 255) / 256, 152 * 16);
    k_gather_vals<<<std::max(g, 1), 256, 0, st>>>(nnz, src, val, out);
    ++g_launches;
}

// out[p] += alpha * u[row(p)] * v[col(p)] over the stored entries (one thread per row, entries in order).
__global__ void k_pattern_outer(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                const double* __restrict__ u, const double* __restrict__ v, double alpha,
                                double* __restrict__ out) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const double ur = alpha * u[r];
    for (int p = rp[r]; p < rp[r + 1]; ++p) out[p] += ur * v[col[p]];
}

void launch_pattern_outer(int n, const int* rp, const int* col, const double* u, const double* v, double alpha,
                          double* out, cudaStream_t st) {
    k_pattern_outer<<<(n + 255) / 256, 256, 0, st>>>(n, rp, col, u, v, alpha, out);
    ++g_launches;
}

// One CTA (256 threads) per row block: stable counting sort of the block's rows by length (rows beyond kSortedMax entries last,
// in order), so the order -- and every sum formed in it -- is deterministic; and the class boundaries (cls, see kernels.h).
// The rows the sorted copy takes, a thread each, end where a slice of 32 rows would be less than half full or so long that
// its chain of loads (a round per 8 entries, some 1.2 us) outlasts the time the block's entries need on an SM (about
// a nanosecond each): then a warp per row, or 8 lanes, is the better use.  Blocks of fewer than 2048 rows have too few slices to
// even out over 16 warps beyond 16 entries (400,000 Zipf rows in blocks of 1344, FP64: 117 us per step with the longer rows in
// the copy, 107 without; 1M in blocks of 3296: 164 and 177).
__global__ void __launch_bounds__(256) k_bin_rows(const int* __restrict__ rp, const int* __restrict__ lb_m0,
                                                  const int* __restrict__ lb_len, uint16_t* __restrict__ perm,
                                                  int* __restrict__ cls) {
    constexpr int NK = kSortedMax + 2, NW = 8;
    __shared__ int cnt[NK], cur[NK], wc[NW][NK];
    const int L = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = lb_m0[L], len = lb_len[L];
    auto row_len = [&](int k) { return rp[m0 + k + 1] - rp[m0 + k]; };
    auto key_of = [&](int k) { return min(row_len(k), kSortedMax + 1); };
    for (int q = tid; q < NK; q += blockDim.x) cnt[q] = 0;
    for (int q = tid; q < NW * NK; q += blockDim.x) wc[q / NK][q % NK] = 0;
    __syncthreads();
    for (int k = tid; k < len; k += blockDim.x) atomicAdd(&cnt[key_of(k)], 1);
    __syncthreads();
    if (tid == 0) {
        int run = 0;
        for (int b = 0; b < NK; ++b) {
            cur[b] = run;
            run += cnt[b];
        }
        cls[2 * L] = cur[65];
    }
    const unsigned lt = (1u << lane) - 1u;
    for (int base = 0; base < len; base += blockDim.x) {
        __syncthreads();
        const int k = base + tid;
        const bool ok = k < len;
        const int key = ok ? key_of(k) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        const bool lead = ok && lane == __ffs(peers) - 1;
        if (lead) wc[warp][key] = __popc(peers);
        __syncthreads();
        if (ok) {
            int pos = cur[key] + __popc(peers & lt);
            for (int w = 0; w < warp; ++w) pos += wc[w][key];
            perm[m0 + pos] = (uint16_t)k;
        }
        __syncthreads();
        if (lead) {  // one lane per warp and key
            atomicAdd(&cur[key], __popc(peers));
            wc[warp][key] = 0;
        }
    }
    __syncthreads();
    if (warp == 0) {
        const int most = len < 2048 ? 16 : max(16, (rp[m0 + len] - rp[m0]) / 256);
        int q = (len + 31) / 32 - 1;
        for (; q >= 0; --q) {
            const int i = 32 * q + lane;
            const unsigned l = i < len ? (unsigned)row_len(perm[m0 + i]) : 0u;
            const int sum = (int)__reduce_add_sync(0xffffffffu, l), w = (int)__reduce_max_sync(0xffffffffu, l);
            if (w <= 16 || (w <= kSortedMax && w <= most && 32 * w <= 2 * sum)) break;
        }
        if (lane == 0) cls[2 * L + 1] = min(len, 32 * (q + 1));
    }
}

void launch_bin_rows(int nl, const int* rp, const int* lb_m0, const int* lb_len, uint16_t* perm, int* cls,
                     cudaStream_t st) {
    k_bin_rows<<<nl, 256, 0, st>>>(rp, lb_m0, lb_len, perm, cls);
    ++g_launches;
}

// ---- the length-binned SpMV's sorted copy (SELL-32 over each row block's length order) ----
// Slice base[L] + q holds rows 32q .. 32q+31 of block L's order (local rows perm[m0 + 32q + lane]), those below the block's
// boundary cls[2L + 1]; it is as wide as its longest row and stored like the SELL-32 copy below.

// One CTA per row block: row lengths and slice widths (0 beyond the boundary).
__global__ void k_sorted_len(const int* __restrict__ rp, const int* __restrict__ lb_m0, const int* __restrict__ lb_len,
                             const uint16_t* __restrict__ perm, const int* __restrict__ cls,
                             const int* __restrict__ base, uint16_t* __restrict__ len, int* __restrict__ wid) {
    const int L = blockIdx.x, m0 = lb_m0[L], nr = lb_len[L], na = cls[2 * L + 1];
    const int lane = threadIdx.x & 31;
    for (int q = threadIdx.x >> 5; 32 * q < nr; q += blockDim.x >> 5) {
        const int i = 32 * q + lane;
        int l = 0;
        if (i < na) {
            const int k = m0 + perm[m0 + i];
            l = rp[k + 1] - rp[k];
        }
        const int64_t s = base[L] + q;
        len[s * 32 + lane] = (uint16_t)l;
        const int w = (int)__reduce_max_sync(0xffffffffu, (unsigned)l);
        if (lane == 0) wid[s] = w;
    }
}

// Columns (when scol is not null) and values in slice order, one warp per slice.
template <typename MT>
__global__ void k_sorted_fill(const int* __restrict__ rp, const int* __restrict__ col, const double* __restrict__ val,
                              const int* __restrict__ lb_m0, const int* __restrict__ lb_len,
                              const uint16_t* __restrict__ perm, const int* __restrict__ cls,
                              const int* __restrict__ base, const int* __restrict__ off, int* __restrict__ scol,
                              MT* __restrict__ sval) {
    const int L = blockIdx.x, m0 = lb_m0[L], na = cls[2 * L + 1];
    const int lane = threadIdx.x & 31;
    for (int q = threadIdx.x >> 5; 32 * q < na; q += blockDim.x >> 5) {
        const int i = 32 * q + lane;
        int a = 0, l = 0;
        if (i < na) {
            const int k = m0 + perm[m0 + i];
            a = rp[k];
            l = rp[k + 1] - a;
        }
        const int o = off[base[L] + q], w = off[base[L] + q + 1] - o;
        const int64_t at = (int64_t)o * 32 + lane;
#pragma unroll 4
        for (int e = 0; e < w; ++e) {
            if (scol) scol[at + (int64_t)e * 32] = (e < l) ? col[a + e] : 0;
            sval[at + (int64_t)e * 32] = (e < l) ? (MT)val[a + e] : MT(0);
        }
    }
}

void launch_sorted_build(int nl, int ns, const int* rp, const int* lb_m0, const int* lb_len, const uint16_t* perm,
                         const int* cls, const int* base, uint16_t* len, int* wid, int* off, cudaStream_t st) {
    k_sorted_len<<<nl, 512, 0, st>>>(rp, lb_m0, lb_len, perm, cls, base, len, wid);
    k_scan_plain<<<1, 1024, 0, st>>>(wid, off, ns);
    g_launches += 2;
}

void launch_sorted_fill(int nl, const int* rp, const int* col, const double* val, const int* lb_m0, const int* lb_len,
                        const uint16_t* perm, const int* cls, const int* base, const int* off, int* scol, double* sval,
                        float* sval32, cudaStream_t st) {
    if (sval) k_sorted_fill<double><<<nl, 512, 0, st>>>(rp, col, val, lb_m0, lb_len, perm, cls, base, off, scol, sval);
    if (sval32)
        k_sorted_fill<float><<<nl, 512, 0, st>>>(rp, col, val, lb_m0, lb_len, perm, cls, base, off, nullptr, sval32);
    g_launches += (sval ? 1 : 0) + (sval32 ? 1 : 0);
}

// ---- SELL-32 copy of a matrix with short rows ----
// Slice s holds rows moff[q] + 32 c .. of system q (c = s - sl0[q]); entry e of the slice's lane l sits at
// (off[s] + e) * 32 + l, so the 32 lanes of a warp read entry e of their rows with one coalesced load.  A slice is
// as wide as its longest row; a lane past its row's end (or past the system's last row) holds column 0, value 0,
// and its length says so.

__device__ __forceinline__ int sell_system(const int* __restrict__ sl0, int nsys, int64_t s) {
    int lo = 0, hi = nsys - 1;  // the last q with sl0[q] <= s
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sl0[mid] <= s) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// One warp per slice: row lengths and the slice width.
__global__ void k_sell_len(int ns, const int* __restrict__ sl0, int nsys, const int* __restrict__ moff,
                           const int* __restrict__ rp, uint8_t* __restrict__ len, int* __restrict__ wid) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t s = w0; s < ns; s += nwarps) {
        const int q = sell_system(sl0, nsys, s);
        const int r = moff[q] + 32 * (int)(s - sl0[q]) + lane;
        const int l = (r < moff[q + 1]) ? rp[r + 1] - rp[r] : 0;
        len[s * 32 + lane] = (uint8_t)l;
        const int w = (int)__reduce_max_sync(0xffffffffu, (unsigned)l);
        if (lane == 0) wid[s] = w;
    }
}

// One warp per slice: columns and values in slice order (entry order within each row).
__global__ void k_sell_fill(int ns, const int* __restrict__ sl0, int nsys, const int* __restrict__ moff,
                            const int* __restrict__ rp, const int* __restrict__ col, const double* __restrict__ val,
                            const int* __restrict__ off, const uint8_t* __restrict__ len, int* __restrict__ scol,
                            double* __restrict__ sval) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t s = w0; s < ns; s += nwarps) {
        const int q = sell_system(sl0, nsys, s);
        const int r = moff[q] + 32 * (int)(s - sl0[q]) + lane;
        const int l = len[s * 32 + lane];
        const int a = (l > 0) ? rp[r] : 0;
        const int64_t base = (int64_t)off[s] * 32 + lane;
        const int w = off[s + 1] - off[s];
        for (int e = 0; e < w; ++e) {
            if (scol) scol[base + (int64_t)e * 32] = (e < l) ? col[a + e] : 0;
            sval[base + (int64_t)e * 32] = (e < l) ? val[a + e] : 0.0;
        }
    }
}

static int sell_grid(int ns) { return (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)ns + 7) / 8, 152 * 64)); }

void launch_sell_build(int ns, const int* sl0, int nsys, const int* moff, const int* rp, uint8_t* len, int* wid,
                       int* off, cudaStream_t st) {
    k_sell_len<<<sell_grid(ns), 256, 0, st>>>(ns, sl0, nsys, moff, rp, len, wid);
    k_scan_plain<<<1, 1024, 0, st>>>(wid, off, ns);
    g_launches += 2;
}

void launch_sell_fill(int ns, const int* sl0, int nsys, const int* moff, const int* rp, const int* col,
                      const double* val, const int* off, const uint8_t* len, int* scol, double* sval,
                      cudaStream_t st) {
    k_sell_fill<<<sell_grid(ns), 256, 0, st>>>(ns, sl0, nsys, moff, rp, col, val, off, len, scol, sval);
    ++g_launches;
}

}  // namespace sfg
