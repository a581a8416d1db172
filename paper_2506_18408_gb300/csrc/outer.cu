// Outer FGMRES (Algorithm 1) on the device for every problem of a batch, FP64 throughout.
//
// Outer step j:  w = A z_j (fused with the first batch of dot products v_l^T w), two classical Gram-Schmidt passes
// against v_0..v_j (the reorthogonalised form of the orthogonalisation loop of Algorithm 1), h_{j+1,j} = ||w||,
// v_{j+1} = w / h_{j+1,j} (stored unnormalised with its scale nu), then one Givens rotation of the Hessenberg
// column, which gives the FGMRES residual estimate |g_{j+1}| and the FFOM residual |g_{j+1}| / |c_j| (Eq. 4: the
// FFOM residual is h_{j+1,j} |gamma_j|; in rotated form this is the FGMRES residual divided by the cosine of the
// last rotation).  The FFOM residual feeds rule C3 of the next inner cycle through the bound of Eq. 5.
// Row-block kernels skip the blocks of problems that are done; per-problem kernels reduce their problem's block
// partials in block order, so every sum has a fixed order.
#include "kernels.h"
#include "spmv.cuh"

#include <algorithm>

namespace sfg {

__device__ __forceinline__ bool outer_idle(const Plan& P, int p) { return (P.pflag[p] & 1) != 0; }

// A x over rows [k0, k0 + len) of a block, emit(k, (A x)_k) once per row k; smem: the shape's scratch (the block's rows, or the
// stage area).  The length-binned shape takes whole blocks only.  The shapes that go through shared memory end the SpMV with
// a block barrier.
template <int V, int U, typename Emit>
__device__ __forceinline__ void block_spmv(const Plan& P, const BlockInfo& bi, int k0, int len,
                                           const double* __restrict__ x, unsigned char* smem, Emit&& emit) {
    const int m0 = bi.v0 - bi.cs + k0;
    if constexpr (V == kVecStaged) {
        spmv_rows_staged<double, double, double>(P.rp + m0, P.col, P.val, x + bi.cs, len, smem, P.maxlen, [](int) {},
                                                 [&](int k, double v) {
                                                     if (k < len) emit(k0 + k, v);
                                                 });
    } else {
        double* yb = reinterpret_cast<double*>(smem);
        SortedRows<double> so{};
        if constexpr (V == 0) so = sorted_rows<double>(P, bi);
        spmv_rows_to_smem<V, U, double, double, double>(P.rp, P.col, P.val, x + bi.cs, m0, m0 + len, yb, P.perm, so);
        __syncthreads();
        for (int k = threadIdx.x; k < len; k += blockDim.x) emit(k0 + k, yb[k]);
    }
}

// The shape of an FP64 SpMV kernel of the outer iteration that needs `fixed` bytes of shared memory besides: staged entries
// for matrices of one thread per row where two 512-thread CTAs fit on an SM, and its dynamic shared memory.  128^3: w = A z with
// its dots 94 -> 73 us, the residual 78 -> 55 us, y = A x 55 -> 46 us per launch.
static int outer_vec(const Plan& p, size_t fixed, size_t* smem) {
    const size_t stage = 16 * (size_t)stage_bytes<double>(p.maxlen);
    if (p.vec == 1 && 2 * (fixed + stage + 4096) <= 226 * 1024) {
        *smem = fixed + stage;
        return kVecStaged;
    }
    *smem = std::max<size_t>(fixed, (size_t)p.Bn * sizeof(double));
    return p.vec;
}

// rb = b - A x (x may be null: rb = b); npart[b] = ||rb||^2 over the block, npart2[b] = ||b||^2 over the block.
template <int V, int U>
__global__ void __launch_bounds__(512, 2)
    k_residual(const Plan P, const double* __restrict__ bv, const double* __restrict__ x, double* __restrict__ rb,
               int only_final) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[32];
    const int b = blockIdx.x;
    const BlockInfo bi = block_info(P, b);
    const int fl = P.pflag[bi.prob];
    if (only_final ? !(fl & 2) : (fl & 1)) return;
    double a1 = 0.0, a2 = 0.0;
    auto row = [&](int k, double ax) {
        const double bb = bv[bi.v0 + k];
        const double rr = bb - ax;
        if (rb) rb[bi.v0 + k] = rr;
        a1 += rr * rr;
        a2 += bb * bb;
    };
    if (x) {
        block_spmv<V, U>(P, bi, 0, bi.len, x, smem, row);
    } else {
        for (int k = threadIdx.x; k < bi.len; k += blockDim.x) row(k, 0.0);
    }
    a1 = block_sum(a1, red);
    a2 = block_sum(a2, red);
    if (threadIdx.x == 0) {
        P.npart[b] = a1;
        P.npart2[b] = a2;
    }
}

void launch_residual(const Plan& p, const double* b, const double* x, double* rb, bool only_final) {
    size_t sm = 0;
    const int vec = x ? outer_vec(p, 0, &sm) : 1;
    SFG_SPMV_DISPATCH(vec, (set_smem((const void*)k_residual<VV, UU>, sm),
                            k_residual<VV, UU><<<p.nblk, 512, sm, p.st>>>(p, b, x, rb, only_final ? 1 : 0)));
    ++g_launches;
}

// Per problem (one warp each): beta = ||r0||, ||b||, tol * ||b||, nu_0 = 1/beta, g_0 = beta.
__global__ void k_init_state(const Plan P, double tol) {
    const int p = blockIdx.x, lane = threadIdx.x;
    double a1 = 0.0, a2 = 0.0;
    for (int q = P.prob_b0[p] + lane; q < P.prob_b0[p + 1]; q += 32) {
        a1 += P.npart[q];
        a2 += P.npart2[q];
    }
    a1 = warp_sum(a1);
    a2 = warp_sum(a2);
    if (lane == 0) {
        OuterState* ost = P.ost + p;
        const double beta = sqrt(a1), bn = sqrt(a2);
        ost->j = 0;
        ost->conv_est = 0;
        ost->breakdown = 0;
        ost->nan = (!isfinite(a1) || !isfinite(a2)) ? 1 : 0;
        ost->sync_fail = 0;
        ost->beta = beta;
        ost->bnorm = bn;
        ost->est = beta;
        ost->ffom = beta;
        ost->true_res2 = a1;
        ost->tol_abs = tol * bn;
        const int64_t o = (int64_t)p * (P.jmax + 1);
        P.nu[o] = (beta > 0.0) ? 1.0 / beta : 0.0;
        P.g[o] = beta;
    }
}

void launch_init_state(const Plan& p, double tol) {
    k_init_state<<<p.P, 32, 0, p.st>>>(p, tol);
    ++g_launches;
}

// Per problem flagged "finalise now": ost[p].true_res2 = sum of its blocks' npart.
__global__ void k_true_res(const Plan P) {
    const int p = blockIdx.x;
    if (!(P.pflag[p] & 2)) return;
    double a = 0.0;
    for (int q = P.prob_b0[p] + threadIdx.x; q < P.prob_b0[p + 1]; q += 32) a += P.npart[q];
    a = warp_sum(a);
    if (threadIdx.x == 0) P.ost[p].true_res2 = a;
}

void launch_true_residual_reduce(const Plan& p) {
    k_true_res<<<p.P, 32, 0, p.st>>>(p);
    ++g_launches;
}

// Dots of the block's part of v_0..v_j with the block vector wb (smem): opart[b*ldo + l].  With few columns every column's
// rows are cut into `nseg` segments so that all warps work (a warp per column left 15 of 16 idle at j = 0); the segments'
// sums are added in order.
__device__ __forceinline__ void block_dots(const Plan& P, const BlockInfo& bi, int b, int j,
                                           const double* __restrict__ wb) {
    __shared__ double seg_sh[16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int ldo = P.jmax + 1, cols = j + 1, nseg = max(1, nw / cols);
    for (int t = warp; t < cols * nseg; t += nw) {
        const int l = t / nseg, g = t % nseg;
        const double* vl = P.Vb + (int64_t)l * P.N + bi.v0;
        const int k1 = (int)((int64_t)bi.len * (g + 1) / nseg);
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        int k = (int)((int64_t)bi.len * g / nseg) + lane;
        for (; k + 96 < k1; k += 128) {
            double v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = vl[k + 32 * u];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u] = fma(v[u], wb[k + 32 * u], acc[u]);
        }
        for (; k < k1; k += 32) acc[0] = fma(vl[k], wb[k], acc[0]);
        const double a = warp_sum((acc[0] + acc[1]) + (acc[2] + acc[3]));
        if (lane == 0) {
            if (nseg == 1) P.opart[(int64_t)b * ldo + l] = a;
            else seg_sh[t] = a;
        }
    }
    if (nseg == 1) return;
    __syncthreads();
    if ((int)threadIdx.x < cols) {
        double a = 0.0;
        for (int g = 0; g < nseg; ++g) a += seg_sh[threadIdx.x * nseg + g];
        P.opart[(int64_t)b * ldo + threadIdx.x] = a;
    }
}

// w = A z_j into smem and Wo; opart[b*ldo + l] = Vb_l(block) . w(block) for l <= j; and the true residual of inner cycle
// j, r_hat_j = v_j - A z_j (v_j = nu_j Vb_j), for the bound of Eq. 5: its block partial of ||r_hat_j||^2 goes to npart2
// (free during outer steps).
template <int V, int U>
__global__ void __launch_bounds__(512, 2) k_outer_spmv(const Plan P, int j) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[32];
    const int b = blockIdx.x;
    const BlockInfo bi = block_info(P, b);
    if (outer_idle(P, bi.prob)) return;
    double* wb = reinterpret_cast<double*>(smem);  // [Bn], then the stage area
    const double nuj = P.nu[(int64_t)bi.prob * (P.jmax + 1) + j];
    const double* vj = P.Vb + (int64_t)j * P.N + bi.v0;
    double r2 = 0.0;
    block_spmv<V, U>(P, bi, 0, bi.len, P.Z + (int64_t)j * P.N, V == kVecStaged ? smem + (size_t)P.Bn * sizeof(double) : smem,
                     [&](int k, double w) {
                         wb[k] = w;
                         P.Wo[bi.v0 + k] = w;
                         const double rr = nuj * vj[k] - w;
                         r2 += rr * rr;
                     });
    __syncthreads();
    block_dots(P, bi, b, j, wb);
    r2 = block_sum(r2, red);
    if (threadIdx.x == 0) P.npart2[b] = r2;
}

// out[p*ldo + l] = nu[p][l] * sum over the blocks of problem p of opart[b*ldo + l]  (one warp per (p, l)).
__global__ void k_reduce_cols(const Plan P, int ncols, double* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (w >= (int64_t)P.P * ncols) return;
    const int p = (int)(w / ncols), l = (int)(w % ncols);
    if (outer_idle(P, p)) return;
    const int ldo = P.jmax + 1;
    double acc = 0.0;
    for (int q = P.prob_b0[p] + lane; q < P.prob_b0[p + 1]; q += 32) acc += P.opart[(int64_t)q * ldo + l];
    acc = warp_sum(acc);
    if (lane == 0) out[(int64_t)p * ldo + l] = P.nu[(int64_t)p * ldo + l] * acc;
}

// One classical Gram-Schmidt subtraction w <- w - sum_{l<=j} h_l v_l with v_l = nu_l Vb_l.
//  final == 0: result back into Wo and the next pass's dots into opart
//  final == 1: result into Vb_{j+1} (unnormalised) and ||w||^2 partials into npart
__global__ void __launch_bounds__(512, 2)
    k_outer_cgs(const Plan P, int j, int final_pass, const double* __restrict__ h) {
    extern __shared__ double sm[];
    double* cf = sm;            // [j+1]
    double* wb = sm + (j + 1);  // [Bn]
    __shared__ double red[32];
    const int b = blockIdx.x;
    const BlockInfo bi = block_info(P, b);
    const int p = bi.prob;
    if (outer_idle(P, p)) return;
    const int N = P.N;
    const int64_t o = (int64_t)p * (P.jmax + 1);
    for (int l = threadIdx.x; l <= j; l += blockDim.x) cf[l] = h[o + l] * P.nu[o + l];
    __syncthreads();
    double* dst = P.Vb + (int64_t)(j + 1) * N;
    double nacc = 0.0;
    for (int k = threadIdx.x; k < bi.len; k += blockDim.x) {
        const int r = bi.v0 + k;
        double w = P.Wo[r];
        for (int l = 0; l <= j; ++l) w -= cf[l] * P.Vb[(int64_t)l * N + r];
        if (final_pass) {
            dst[r] = w;
            nacc += w * w;
        } else {
            P.Wo[r] = w;
            wb[k] = w;
        }
    }
    if (final_pass) {
        nacc = block_sum(nacc, red);
        if (threadIdx.x == 0) P.npart[b] = nacc;
        return;
    }
    __syncthreads();
    block_dots(P, bi, b, j, wb);
}

// Per problem (one warp): Hessenberg column j = h1 + h2 (and h_{j+1,j} = ||w||), Givens update, residual
// estimates, histories.
__global__ void k_outer_givens(const Plan P, int j) {
    const int p = blockIdx.x, lane = threadIdx.x;
    if (outer_idle(P, p)) return;
    const int ldo = P.jmax + 1, J = P.jmax;
    double a = 0.0, ar = 0.0;
    for (int q = P.prob_b0[p] + lane; q < P.prob_b0[p + 1]; q += 32) {
        a += P.npart[q];
        ar += P.npart2[q];
    }
    a = warp_sum(a);
    ar = warp_sum(ar);
    if (lane != 0) return;
    OuterState* ost = P.ost + p;
    const CycleState* cyc = P.cyc + p;
    const int64_t oh = (int64_t)p * J, og = (int64_t)p * ldo;
    P.ires_hist[oh + j] = sqrt(ar);  // ||v_j - A z_j||: the factor ||r_hat_j|| of the bound of Eq. 5
    P.rho_hist[oh + j] = cyc->rho;   // the cycle's sketched estimate of it (rule C3)
    if (P.gsync && P.gsync[1]) {  // the inner cycle's grid-wide wait gave up: its results are not valid
        ost->sync_fail = 1;
        ost->nan = 1;
    }
    P.k_hist[oh + j] = cyc->k;
    P.reason_hist[oh + j] = cyc->reason;
    if (cyc->k == 0) {  // inner cycle produced no correction
        ost->breakdown = 2;
        return;
    }
    if (cyc->reason == 6) ost->nan = 1;
    const double* h1 = P.h1 + og;
    const double* h2 = P.h2 + og;
    double* cs = P.cs + oh;
    double* sn = P.sn + oh;
    double* g = P.g + og;
    const double hn = sqrt(a);
    double* colj = P.H + og * J + (int64_t)j * ldo;
    for (int l = 0; l <= j; ++l) colj[l] = h1[l] + h2[l];
    colj[j + 1] = hn;
    for (int l = 0; l < j; ++l) {
        const double x0 = colj[l], x1 = colj[l + 1];
        colj[l] = cs[l] * x0 + sn[l] * x1;
        colj[l + 1] = -sn[l] * x0 + cs[l] * x1;
    }
    const double aa = colj[j], bb = colj[j + 1];
    const double r = hypot(aa, bb);
    double c = 1.0, s = 0.0;
    if (r > 0.0) {
        c = aa / r;
        s = bb / r;
    }
    cs[j] = c;
    sn[j] = s;
    colj[j] = r;
    colj[j + 1] = 0.0;
    const double gj = g[j];
    g[j] = c * gj;
    g[j + 1] = -s * gj;
    const double est = fabs(g[j + 1]);
    const double ffom = (c != 0.0) ? est / fabs(c) : INFINITY;
    P.nu[og + j + 1] = (hn > 0.0) ? 1.0 / hn : 0.0;
    if (P.outer_variant == 1 && c == 0.0) {  // FFOM: the square system of this step is singular; keep step j's x
        ost->breakdown = 2;
        return;
    }
    const double e = (P.outer_variant == 1) ? ffom : est;  // the variant's residual estimate
    ost->j = j + 1;
    ost->est = e;
    ost->ffom = ffom;
    ost->breakdown = (hn == 0.0) ? 1 : 0;
    ost->conv_est = (e <= ost->tol_abs) ? 1 : 0;
    if (!isfinite(est) || !isfinite(hn) || !isfinite(r)) ost->nan = 1;
    P.est_hist[oh + j] = e / ost->bnorm;
    P.ffom_hist[oh + j] = ffom / ost->bnorm;
}

void launch_outer_step(const Plan& p, int j) {
    size_t sm;
    const int vec = outer_vec(p, (size_t)p.Bn * sizeof(double), &sm);
    SFG_SPMV_DISPATCH(vec, (set_smem((const void*)k_outer_spmv<VV, UU>, sm),
                            k_outer_spmv<VV, UU><<<p.nblk, 512, sm, p.st>>>(p, j)));
    const int ncols = j + 1, wpb = 8;
    const int rgrid = (int)(((int64_t)p.P * ncols + wpb - 1) / wpb);
    k_reduce_cols<<<rgrid, 32 * wpb, 0, p.st>>>(p, ncols, p.h1);
    const size_t sm2 = (size_t)(p.Bn + j + 1) * sizeof(double);
    set_smem((const void*)k_outer_cgs, sm2);
    k_outer_cgs<<<p.nblk, 512, sm2, p.st>>>(p, j, 0, p.h1);
    k_reduce_cols<<<rgrid, 32 * wpb, 0, p.st>>>(p, ncols, p.h2);
    k_outer_cgs<<<p.nblk, 512, (size_t)(j + 1) * sizeof(double), p.st>>>(p, j, 1, p.h2);
    k_outer_givens<<<p.P, 32, 0, p.st>>>(p, j);
    g_launches += 6;
}

// Per problem flagged "finalise now" (one warp): y = R^{-1} g over the rotated J x J triangle, J = the problem's
// outer iteration count.
__global__ void k_final_y(const Plan P) {
    extern __shared__ double rhs[];
    const int p = blockIdx.x;
    if (!(P.pflag[p] & 2)) return;
    const int ldo = P.jmax + 1, J = P.ost[p].j;
    const double* H = P.H + (int64_t)p * ldo * P.jmax;
    const double* g = P.g + (int64_t)p * ldo;
    double* y = P.yo + (int64_t)p * P.jmax;
    const int lane = threadIdx.x;
    // FFOM: the square system before the last rotation (c, s) has last diagonal c r_JJ and last right-hand side
    // g_J / c; the rows above are those of R
    const double cl = (P.outer_variant == 1 && J > 0) ? P.cs[(int64_t)p * P.jmax + J - 1] : 1.0;
    for (int l = lane; l < J; l += 32) rhs[l] = (l == J - 1) ? g[l] / cl : g[l];
    __syncwarp();
    for (int l = J - 1; l >= 0; --l) {
        const double yl = rhs[l] / (H[(int64_t)l * ldo + l] * ((l == J - 1) ? cl : 1.0));
        for (int q = lane; q < l; q += 32) rhs[q] -= H[(int64_t)l * ldo + q] * yl;
        if (lane == 0) y[l] = yl;
        __syncwarp();
    }
}

// x = x0 + Z y over the blocks of flagged problems, each block in pieces of kFinalRows rows (one CTA each, grid y; two rows and
// four columns in flight per thread).  Bound by HBM; 128^3, 7 columns: 59 -> 32 us against a CTA per row block.
constexpr int kFinalThreads = 256, kFinalRows = 512;
__global__ void __launch_bounds__(kFinalThreads) k_final_x(const Plan P, const double* __restrict__ x0,
                                                           double* __restrict__ x) {
    __shared__ double yy[kMaxM];
    const BlockInfo bi = block_info(P, blockIdx.x);
    const int p = bi.prob, k0 = blockIdx.y * kFinalRows;
    if (!(P.pflag[p] & 2) || k0 >= bi.len) return;
    const int J = P.ost[p].j;
    const int64_t N = P.N;
    for (int l = threadIdx.x; l < J; l += kFinalThreads) yy[l] = P.yo[(int64_t)p * P.jmax + l];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kFinalRows / kFinalThreads; ++u) {
        const int k = k0 + u * kFinalThreads + threadIdx.x;
        if (k >= bi.len) break;
        const int64_t r = bi.v0 + k;
        double acc = x0 ? x0[r] : 0.0;
#pragma unroll 4
        for (int l = 0; l < J; ++l) acc += yy[l] * P.Z[(int64_t)l * N + r];
        x[r] = acc;
    }
}

void launch_final_x(const Plan& p, int J, const double* x0, double* x) {
    k_final_y<<<p.P, 32, (size_t)std::max(J, 1) * sizeof(double), p.st>>>(p);
    k_final_x<<<dim3(p.nblk, (p.Bn + kFinalRows - 1) / kFinalRows), kFinalThreads, 0, p.st>>>(p, x0, x);
    g_launches += 2;
}

// y = A x; staged entries: each block in pieces of kPlainRows rows (one CTA each, grid y), which come and go on the two CTAs of 64
// registers a thread that an SM holds, so that their waits and ends do not fall together.
constexpr int kPlainRows = 2048;
template <int V, int U>
__global__ void __launch_bounds__(512, 2)
    k_spmv_plain(const Plan P, const double* __restrict__ x, double* __restrict__ y) {
    extern __shared__ __align__(16) unsigned char smem[];
    const BlockInfo bi = block_info(P, blockIdx.x);
    const int k0 = blockIdx.y * kPlainRows;
    if (k0 >= bi.len) return;
    const int len = (V == kVecStaged) ? min(kPlainRows, bi.len - k0) : bi.len;
    block_spmv<V, U>(P, bi, k0, len, x, smem, [&](int k, double v) { y[bi.v0 + k] = v; });
}

void launch_spmv_f64(const Plan& p, const double* x, double* y) {
    size_t sm;
    const int vec = outer_vec(p, 0, &sm);
    const int pieces = (vec == kVecStaged) ? (p.Bn + kPlainRows - 1) / kPlainRows : 1;
    SFG_SPMV_DISPATCH(vec, (set_smem((const void*)k_spmv_plain<VV, UU>, sm),
                            k_spmv_plain<VV, UU><<<dim3(p.nblk, pieces), 512, sm, p.st>>>(p, x, y)));
    ++g_launches;
}

}  // namespace sfg
