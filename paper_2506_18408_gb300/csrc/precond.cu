// Zero-fill incomplete LU (ILU(0)) right preconditioning in a multicolour order, on the device (the "-p" runs of
// Section 4: ILU(0) preconditioning; Table 1).
//
// The rows are ordered colour by colour (P: a greedy colouring of the pattern of A + A^T, computed once on the host
// when the handle's matrix is set up; no two coupled rows share a colour), and M = P^T L U P with L U the ILU(0)
// factorisation of the permuted matrix P A P^T.  Because rows of one colour are not coupled, the diagonal colour
// blocks of L are identities and those of U diagonal, so
//  * the factorisation is one pass per colour, every row of the colour independent (row r eliminates with the
//    finished rows k < r of earlier colours, in increasing k, dropping updates outside the pattern: the IKJ form), and
//  * M^{-1} u needs one pass per colour forward (y_r = u_perm(r) - sum_{k<r} l_rk y_k) and one per colour backward (z_r = (y_r
//    - sum_{k>r} u_rk z_k) / u_rr), one thread per row, instead of a wavefront of ~3N dependent levels of the natural order.
//    Rows of the first colour have no earlier columns, so their y is u and their forward pass is left out; rows of the last
//    colour have no later ones, so their z follows from their y in the same pass: 2 ncol - 2 passes, two for the red-black
//    order of a stencil.
// A pass is bound by HBM and the latency of its gathers.  The factors are read through rows_staged (rows of at most 16 entries:
// coalesced copies a group of rows ahead), vectors by original index (y, z and out share that order), and the division by
// the pivot is a product with its stored reciprocal and one correction step (three FP64 instructions for some twelve on a pipe
// that takes 17 cycles per warp and instruction).  96^3, red-black: two passes of 13.2 us per application against four of 6.7
// and 10.5 us (solve 22.2 -> 19.8 ms).
// The permuted matrix is stored in CSR with sorted columns (permuted indices), its diagonal position per row, and
// the position of every entry in A's CSR, so new values of A refresh the factors without rebuilding the structure.
#include "kernels.h"
#include "spmv.cuh"

#include <algorithm>

namespace sfg {

// lu[p] = val[src[p]]: the values of P A P^T in its own CSR order.
__global__ void k_ilu_gather(int64_t nnz, const int* __restrict__ src, const double* __restrict__ val,
                             double* __restrict__ lu) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < nnz) lu[p] = val[src[p]];
}

// ILU(0) of the rows [r0, r1) of one colour, one thread per row: for each entry (r, k) with k < r (earlier colours,
// already final), l_rk = a_rk / u_kk, then a_rj -= l_rk u_kj for the entries j > k that row r and row k both hold
// (a merge of the two sorted rows).  A zero pivot sets bit 0 of *bad.
__global__ void k_ilu0_colour(int r0, int r1, const int* __restrict__ rp, const int* __restrict__ col,
                              const int* __restrict__ diag, double* __restrict__ lu, int* __restrict__ bad) {
    const int r = r0 + (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (r >= r1) return;
    const int a = rp[r], e = rp[r + 1], dr = diag[r];
    for (int p = a; p < dr; ++p) {
        const int k = col[p];
        const double ukk = lu[diag[k]];
        if (ukk == 0.0) {
            atomicOr(bad, 1);
            return;
        }
        const double l = lu[p] / ukk;
        lu[p] = l;
        int q = p + 1;                             // row r's entries after column k
        int s = diag[k] + 1;                       // row k's entries after its diagonal
        const int se = rp[k + 1];
        while (q < e && s < se) {
            const int cq = col[q], cs = col[s];
            if (cq == cs) {
                lu[q] -= l * lu[s];
                ++q;
                ++s;
            } else if (cq < cs) {
                ++q;
            } else {
                ++s;
            }
        }
    }
    if (lu[dr] == 0.0) atomicOr(bad, 1);
}

// Whether the cycle of the plan's single problem has stopped before step i (nothing of step i is used then).
__device__ __forceinline__ bool ilu_idle(const Plan& P, int i) {
    if (i < 0) return false;
    const CycleState* c = P.cyc;
    return c->stopped || c->brk_step <= i || (P.pflag[0] & 1);
}

// piv[r] = (u_rr, 1 / u_rr); a pivot whose reciprocal overflows sets bit 1 of *bad.
__global__ void k_ilu_pivots(int n, const int* __restrict__ diag, const double* __restrict__ lu,
                             double2* __restrict__ piv, int* __restrict__ bad) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const double d = lu[diag[r]];
    const double inv = 1.0 / d;
    piv[r] = make_double2(d, inv);
    if (isinf(inv)) atomicOr(bad, 2);
}

// ocol[p] = the original index of entry p's column, with kLaterColour set where that column is not of the first colour.
constexpr unsigned kLaterColour = 0x80000000u;
__global__ void k_ilu_ocol(int64_t nnz, int first, const int* __restrict__ col, const int* __restrict__ perm,
                           int* __restrict__ ocol) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < nnz) ocol[p] = (int)((unsigned)perm[col[p]] | (col[p] >= first ? kLaterColour : 0u));
}

// The entries of a row before (forward) or after (backward) its diagonal.
template <bool FWD>
struct TriangleRows {
    const int* diag;  // of the pass's first row
    int len;
    __device__ __forceinline__ int load(int k) const { return k < len ? __ldg(diag + k) : 0; }
    __device__ __forceinline__ void cut(int d, int a, int& off, int& l) const {
        if constexpr (FWD) {
            l = d - a;
        } else {
            off = d + 1 - a;
            l -= off;
        }
    }
};

// One pass over the rows [r0, r1) of a colour, the CTA's part of `chunk` rows.  Forward: y = u - sum of l y, and with `final`
// (the last colour) z = y / u_rr into out, else y.  Backward: z = (y - sum of u z) / u_rr into out, with `first` y = u.
// DIV: some pivot's reciprocal overflows, so the pass divides.  Chosen per factorisation: a division for such rows alone costs
// all others its branch (a 1M-row solve 19.7 -> 22.2 ms, with the operands scaled instead 20.4 ms).
template <bool FWD, bool STAGED, bool DIV>
__global__ void __launch_bounds__(512, 2) k_ilu_pass(const Plan P, int i, int r0, int r1, int chunk, bool edge,
                                                     int maxlen, const double* __restrict__ u, double* y, double* out) {
    if (ilu_idle(P, i)) return;
    extern __shared__ __align__(16) unsigned char smem[];
    const IluDev& I = P.ilu;
    const int s0 = r0 + blockIdx.x * chunk, len = min(chunk, r1 - s0);
    const int* __restrict__ diag = I.diag + s0;
    const int* __restrict__ perm = I.perm + s0;
    const double2* __restrict__ piv = I.piv + s0;
    auto get = [&](int c) -> double {
        const unsigned o = (unsigned)c & ~kLaterColour;
        if constexpr (FWD) return ((unsigned)c & kLaterColour) ? y[o] : __ldg(u + o);
        else return out[o];
    };
    int at = 0;
    double v0 = 0.0;
    double2 pv = make_double2(1.0, 1.0);
    auto pre = [&](int k) {
        if (k >= len) return;
        at = __ldg(perm + k);
        v0 = (FWD || edge) ? __ldg(u + at) : y[at];
        if (!FWD || edge) pv = __ldg(piv + k);
    };
    auto emit = [&](int k, double sum) {
        if (k >= len) return;
        const double v = v0 - sum;
        if (FWD && !edge) {
            y[at] = v;
        } else {
            const double t = v * pv.y;
            out[at] = DIV ? v / pv.x : fma(fma(-t, pv.x, v), pv.y, t);
        }
    };
    const TriangleRows<FWD> part{diag, len};
    if constexpr (STAGED) {
        rows_staged<double, double>(I.rp + s0, I.ocol, I.lu, len, smem, maxlen, get, part, pre, emit);
    } else {
        for (int k = threadIdx.x; k < len; k += blockDim.x) {
            pre(k);
            const int a = I.rp[s0 + k];
            int off = 0, l = I.rp[s0 + k + 1] - a;
            part.cut(part.load(k), a, off, l);
            double sum = 0.0;
            for (int q = a + off; q < a + off + l; ++q) sum += I.lu[q] * get(I.ocol[q]);
            emit(k, sum);
        }
    }
}

cudaError_t launch_ilu_factor(const IluHost& H, const double* val, int* bad, cudaStream_t st) {
    const IluDev& I = H.dev;
    k_ilu_gather<<<(unsigned)((H.nnz + 255) / 256), 256, 0, st>>>(H.nnz, H.src, val, I.lu);
    for (int c = 0; c < H.ncol; ++c) {
        const int r0 = H.starts[c], r1 = H.starts[c + 1];
        if (r1 > r0) k_ilu0_colour<<<(unsigned)((r1 - r0 + 255) / 256), 256, 0, st>>>(r0, r1, I.rp, I.col, I.diag, I.lu, bad);
    }
    if (H.n > 0) k_ilu_pivots<<<(unsigned)((H.n + 255) / 256), 256, 0, st>>>(H.n, I.diag, I.lu, H.piv, bad);
    g_launches += 2 + H.ncol;
    return cudaGetLastError();
}

cudaError_t launch_ilu_columns(const IluHost& H, int* ocol, cudaStream_t st) {
    if (H.nnz > 0)
        k_ilu_ocol<<<(unsigned)((H.nnz + 255) / 256), 256, 0, st>>>(H.nnz, H.ncol > 0 ? H.starts[1] : 0, H.dev.col,
                                                                   H.dev.perm, ocol);
    ++g_launches;
    return cudaGetLastError();
}

template <bool FWD, bool DIV>
static void ilu_pass(const Plan& P, int i, int c, bool edge, const double* u, double* out) {
    const IluHost& H = *P.ilu_host;
    const int r0 = H.starts[c], r1 = H.starts[c + 1];
    if (r1 <= r0) return;
    // about two CTAs per SM, whole rounds of 512 rows
    const int per = (r1 - r0 + 2 * P.sms - 1) / (2 * P.sms), chunk = std::max(512, (per + 511) / 512 * 512);
    const unsigned grid = (unsigned)((r1 - r0 + chunk - 1) / chunk);
    if (H.maxlen <= 16) {
        const size_t sm = 16 * (size_t)stage_bytes<double>(H.maxlen);
        set_smem((const void*)k_ilu_pass<FWD, true, DIV>, sm);
        k_ilu_pass<FWD, true, DIV><<<grid, 512, sm, P.st>>>(P, i, r0, r1, chunk, edge, H.maxlen, u, H.dev.y, out);
    } else {
        k_ilu_pass<FWD, false, DIV><<<grid, 512, 0, P.st>>>(P, i, r0, r1, chunk, edge, H.maxlen, u, H.dev.y, out);
    }
    ++g_launches;
}

template <bool DIV>
static void ilu_apply(const Plan& P, int i, const double* u, double* out) {
    const int ncol = P.ilu_host->ncol;
    for (int c = std::min(1, ncol - 1); c < ncol; ++c) ilu_pass<true, DIV>(P, i, c, c == ncol - 1, u, out);
    for (int c = ncol - 2; c >= 0; --c) ilu_pass<false, DIV>(P, i, c, c == 0, u, out);
}

void launch_ilu_apply(const Plan& P, int i, const double* u, double* out) {
    if (P.ilu_host->divide) ilu_apply<true>(P, i, u, out);
    else ilu_apply<false>(P, i, u, out);
}

}  // namespace sfg
