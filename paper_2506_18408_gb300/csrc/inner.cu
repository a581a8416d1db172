// One sketched-GMRES cycle on the device for every problem of a batch (Section 3; Eq. 3 with r0 = v_j and zero
// initial guess).
//
// Storage: the basis vectors are kept unnormalised, b_l = sigma_l u_l; scale factors live in scalars and a stored
// vector is only ever rescaled by a power of two.  Per inner step i (0-based; the paper's i+1):
//   k_inner_spmv  w' = A u_i, the truncated-Arnoldi dot products u_l^T w' for the last t basis vectors
//                 (Section 4.1), ||u_i||^2, and the per-block partial sketch S w' -- one pass over A; the row block of
//                 w' stays in shared memory for the sketch gather lists.  In FP64 the sketch partials are accumulated
//                 exactly in 64-bit fixed point (integer adds), which keeps the scarce FP64 pipe for the SpMV.
//   k_inner_axpy  sigma_i = 1/||u_i||, h_l = b_l^T A b_i, the sketched column S A b_i = sigma_i S w', and the next
//                 stored vector u_{i+1} = 2^p_i (w' - sum_l sigma_l^2 (u_l^T w') u_l), with 2^p_i the power of two
//                 just below sigma_i (an exact rescaling that keeps stored norms O(||A||) instead of growing like
//                 ||A||^i).
//   k_inner_qr    per problem a cluster of CTAs: Gram-Schmidt with one reorthogonalisation pass of S A b_i against Q
//                 (Section 3, C2), the condition proxy max|r_ll|/min|r_ll| (rule C2), the running sketched residual
//                 (rule C3) and C1.  It runs on a second stream, overlapping the next step's SpMV; a step that runs
//                 past the end of a problem's cycle is discarded.
// After the cycle: k_inner_ls solves R_k y = (Q^T S v)_k and k_inner_gemv forms z_j = B_k y_k (FP64 output).
// The step kernels (k_inner_spmv, k_inner_axpy and the fused k_inner_step) live in inner_step.cuh and are
// instantiated per precision in inner_f64.cu, inner_f32.cu and inner_bf16.cu; this file holds the QR, the least
// squares, z, the cycle reset and the launchers.
#include "inner_step.cuh"

#include <cooperative_groups.h>
#include <type_traits>

namespace cg = cooperative_groups;

namespace sfg {

// ---------------------------------------------------------------------------------------------------------------
// Sketched QR update of column i, one cluster of nq CTAs per problem (cluster index = problem); CTA q owns the sketch rows
// [s q / nq, s (q+1) / nq) of Q and of the working vectors.  Q is stored CTA by CTA: the slice of CTA q holds its rows of
// column l at slice[l * nrp + r] (nrp odd, so that threads taking consecutive columns of one row read distinct
// shared-memory banks), which makes the columns 0..i-1 that an update needs one contiguous stretch.
//
// An update is a chain of dependent steps (two Gram-Schmidt passes, the norm, the residual), so what counts is the
// latency of each and the FP64 instructions on its path: a warp's FP64 instruction holds its quarter of the SM's FP64 pipe
// for some 67 cycles on this GPU.  Hence: as many SMs as the cluster can have share the 4 s i multiply-adds; the slice, the
// new column and e come into shared memory in one wave of asynchronous 16-byte copies, and both products of both
// passes run there (STAGED; a slice that does not fit is read from L2 in the same layout); products are split so that all
// four warps work; scalars are formed by one thread (the two that need a division by two, in different warps).
//  * projection a = Q^T p: column l by thread wp of group gp (Gp groups of rows), the CTAs' parts exchanged through
//    distributed shared memory and summed in rank order (the same values in every CTA, so every decision is the same);
//  * subtraction p -= Q a: row r by thread ws of group gs (Gs groups of columns).
// A thread's part of a product is one running sum, or with LONG (qr_long) the sums over even and odd terms: a chain twice
// as long has 1.4 times the rounding error.
// Group partials are added in group order: every sum has a fixed order.  Five cluster barriers per update: one per pass, one
// for ||p||^2 and p^T e together (d_i = p^T e / r_ii), one for the updated residual norm, and a last one before any
// CTA leaves.  Each CTA reads the stop state itself (written by earlier launches; the one field another stream may change
// meanwhile, the breakdown step, only ever moves to values above i).  CTAs are small (128 threads, at most 56 registers) so
// they fit beside the inner step's CTAs.
//
// An update takes (clock64 of CTA 0) 11 us at s = 120, i = 15 on 4 CTAs, 15 us at s = 400, i = 50 on 16 and 27 us at s = 1000,
// i = 100 on 16; the earlier form, which streamed column- and row-major copies of Q from L2 on 8 CTAs, took 58 us per update
// of an 80^3 cycle at s = 1000, m = 200 (that cycle 13.4 -> 8.4 ms).

// Sum of v over groups of 16 lanes (every lane gets its group's sum).
__device__ __forceinline__ double half_warp_sum(double v) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums of x and y over the CTA's threads, of which the first nws warps hold values; valid in warp 0: x in lanes 0-15, y in
// lanes 16-31 (half the additions of two separate trees).
__device__ __forceinline__ double qr_pair_sum(double x, double y, double (*red)[4], int nws) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double v = 0.0;
    if (warp < nws) {
        const double ox = __shfl_xor_sync(0xffffffffu, x, 16), oy = __shfl_xor_sync(0xffffffffu, y, 16);
        v = half_warp_sum(lane < 16 ? x + ox : y + oy);
    }
    if (nws > 1) {
        if ((lane & 15) == 0) red[lane >> 4][warp] = v;
        __syncthreads();
        if (warp == 0) {
            v = red[lane >> 4][0];
            for (int w = 1; w < nws; ++w) v += red[lane >> 4][w];
        }
    }
    return v;
}

template <bool STAGED, bool LONG>
__global__ void __launch_bounds__(kQrThreads, 9) k_inner_qr(const Plan P, int i) {
    cg::cluster_group cl = cg::this_cluster();
    cl.barrier_arrive();  // waited for before the first access to another CTA's shared memory: all CTAs have started
    const int q = (int)cl.block_rank(), nq = (int)cl.num_blocks();
    const int prob = blockIdx.x / nq;
    const int s = P.s, m = P.m, nrp = P.qr.nrp;
    double* __restrict__ Qg = P.Q + ((int64_t)prob * nq + q) * P.qr.slice;
    CycleState* cyc = P.cyc + prob;
    const int rlo = (int)((int64_t)s * q / nq), rhi = (int)((int64_t)s * (q + 1) / nq), nr = rhi - rlo;
    double* __restrict__ e = P.e + (int64_t)prob * s + rlo;
    extern __shared__ __align__(16) double qsm[];
    const int ns = STAGED ? (i * nrp + 1) & ~1 : 0;
    const double* Q = STAGED ? qsm : Qg;  // columns 0..i-1 of the slice
    double* p = qsm + ns;                 // [nrp] this CTA's rows of the working vector
    double* es = p + nrp;                 // [nrp] its rows of e
    double* a = es + nrp;                 // [m] full projections
    double* part = a + m;                 // [2][m] partial projections over this CTA's rows, one buffer per pass
    __shared__ double red[2][4];
    __shared__ double sum_sh[3][16];      // every CTA's ||p||^2, p^T e and (CTA 0) ||e||^2 partials
    __shared__ double bc[4];              // scalars formed once for the CTA
    __shared__ double grp[kQrThreads];    // group partials of a split projection, rank sum or subtraction
    const int tid = threadIdx.x;
    if constexpr (STAGED) {
        // i * nrp doubles rounded up to 16 bytes (the slice has room for the rounding)
        const unsigned dst = (unsigned)__cvta_generic_to_shared(qsm);
        for (int u = tid; u < ns / 2; u += kQrThreads)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * u), "l"(Qg + 2 * u) : "memory");
    }
    // the cycle state as earlier launches left it (the same for every CTA of the cluster)
    const double dmax0 = cyc->dmax, dmin0 = cyc->dmin, thr = cyc->cond_thr;
    const int code = (cyc->stopped || (P.pflag[prob] & 1)) ? 1 : (cyc->brk_step <= i ? 2 : 0);
    for (int r = tid; r < nr; r += kQrThreads) {
        p[r] = P.C[((int64_t)prob * m + i) * s + rlo + r];
        es[r] = e[r];
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    cl.barrier_wait();
    if (code) {
        if (code == 2 && q == 0 && tid == 0) {
            cyc->stopped = 1;  // u_i has zero (or non-finite) norm: the cycle keeps k = i columns
            cyc->reason = cyc->brk_reason;
        }
        return;  // the whole cluster returns
    }
    // projection split: Gp groups of rows (Gp * i <= 128 threads), Wp threads per group over the columns
    int Gp = 1;
    while (Gp < 8 && 2 * Gp * i <= kQrThreads && 2 * Gp * 2 <= nr) Gp *= 2;
    const int Wp = kQrThreads / Gp, gp = tid / Wp, wp = tid % Wp;
    const int pr0 = nr * gp / Gp, pr1 = nr * (gp + 1) / Gp;
    int Gr = 1;  // rank-sum split: Gr groups of ranks (a power of two; Gr * i <= 128 threads)
    while (2 * Gr < nq && 2 * Gr * i <= kQrThreads) Gr *= 2;
    // subtraction split: Wr threads over the rows (a power of two from 32 to 128, so that Gs Wr = 128 and every
    // thread has a group), Gs groups of columns
    int Wr = 32;
    while (Wr < nr && Wr < kQrThreads) Wr *= 2;
    const int Gs = kQrThreads / Wr, gs = tid / Wr, ws = tid % Wr;
    const int sl0 = i * gs / Gs, sl1 = i * (gs + 1) / Gs;
    const int nws = (min(nr, kQrThreads) + 31) / 32;  // warps whose threads hold rows in the per-row loops
    __syncthreads();
    for (int pass = 0; pass < 2 && i > 0; ++pass) {
        double* ap = part + pass * m;
        for (int l = wp; l < i; l += Wp) {
            const double* ql = Q + l * nrp;
            double v = 0.0;
            if constexpr (LONG) {
                v = dot2(ql + pr0, 1, p + pr0, pr1 - pr0);
            } else {
#pragma unroll 8
                for (int r = pr0; r < pr1; ++r) v = fma(ql[r], p[r], v);
            }
            if (Gp == 1) ap[l] = v;
            else grp[gp * i + l] = v;
        }
        if (Gp > 1) {
            __syncthreads();
            for (int l = tid; l < i; l += kQrThreads) {
                double v = grp[l];
                for (int g = 1; g < Gp; ++g) v += grp[g * i + l];
                ap[l] = v;
            }
        }
        cl.sync();  // this pass's partials of every CTA are in place
        auto rank_sum = [&](int l, int r0, int r1) -> double {
            double v = 0.0;
#pragma unroll 4
            for (int r2 = r0; r2 < r1; ++r2) v += cl.map_shared_rank(ap, r2)[l];
            return v;
        };
        if (Gr > 1) {
            if (tid < Gr * i) grp[tid] = rank_sum(tid % i, nq / Gr * (tid / i), nq / Gr * (tid / i + 1));
            __syncthreads();
            if (tid < i) {
                double v = grp[tid];
                for (int g = 1; g < Gr; ++g) v += grp[g * i + tid];
                a[tid] = v;
            }
        } else {
            for (int l = tid; l < i; l += kQrThreads) a[l] = rank_sum(l, 0, nq);
        }
        __syncthreads();
        for (int r0 = 0; r0 < nr; r0 += Wr) {
            const int r = r0 + ws;
            double v = 0.0;
            if (r < nr) {
                if constexpr (LONG) {
                    v = dot2(Q + sl0 * nrp + r, nrp, a + sl0, sl1 - sl0);
                } else {
#pragma unroll 8
                    for (int l = sl0; l < sl1; ++l) v = fma(Q[l * nrp + r], a[l], v);
                }
                if (Gs == 1) p[r] -= v;
                else grp[gs * Wr + ws] = v;
            }
        }
        if (Gs > 1) {  // then nr <= Wr
            __syncthreads();
            if (tid < nr) {
                double v = grp[tid];
                for (int g = 1; g < Gs; ++g) v += grp[g * Wr + tid];
                p[tid] -= v;
            }
        }
        if (q == 0) {  // column i of R: the sum of the two passes' projections
            double* __restrict__ Ri = P.R + ((int64_t)prob * m + i) * m;
            for (int l = tid; l < i; l += kQrThreads) Ri[l] = pass ? Ri[l] + a[l] : a[l];
        }
        __syncthreads();
    }
    // r_ii = ||p|| and p^T e from one exchange
    const int lane = tid & 31, warp = tid >> 5;
    double pp = 0.0, pe = 0.0;
    for (int r = tid; r < nr; r += kQrThreads) {
        pp = fma(p[r], p[r], pp);
        pe = fma(p[r], es[r], pe);
    }
    {
        const double v = qr_pair_sum(pp, pe, red, nws);
        if (warp == 0 && (lane & 15) < nq) cl.map_shared_rank(&sum_sh[lane >> 4][q], lane & 15)[0] = v;
    }
    cl.sync();
    if (warp < 2) {  // the ranks' sums by a tree; one warp forms r_ii and its reciprocal, another the condition proxy
        const double v = half_warp_sum((lane & 15) < nq ? sum_sh[lane >> 4][lane & 15] : 0.0);
        if (tid == 0) {
            const double rii0 = sqrt(v);
            bc[0] = rii0;
            bc[3] = 1.0 / rii0;
        } else if (tid == 16) {
            bc[1] = v;
        } else if (tid == 32) {
            const double rii0 = sqrt(v);
            const double dmx = fmax(dmax0, rii0);
            const double dmn = (i == 0) ? rii0 : fmin(dmin0, rii0);
            bc[2] = (dmn > 0.0) ? dmx / dmn : INFINITY;
        }
    }
    __syncthreads();
    const double rii = bc[0], pet = bc[1], kappa = bc[2], inv = bc[3];
    const double dmax = fmax(dmax0, rii);
    const double dmin = (i == 0) ? rii : fmin(dmin0, rii);
    if (!(kappa <= thr)) {  // C2 (also rii == 0 or NaN): drop column i, keep k = i
        if (q == 0 && tid == 0) {
            cyc->stopped = 1;
            cyc->k = i;
            cyc->reason = (i == 0) ? 5 : 2;
        }
        cl.sync();  // no CTA leaves while another may still reach its shared memory
        return;
    }
    const unsigned long long keep = l2_keep_policy();  // Q is read again at every update of the cycle
    const double di = pet * inv;
    double ee = 0.0;
    for (int r = tid; r < nr; r += kQrThreads) {
        const double qv = p[r] * inv;
        st_keep(Qg + i * nrp + r, qv, keep);
        const double ev = es[r] - di * qv;
        e[r] = ev;
        ee = fma(ev, ev, ee);
    }
    ee = qr_pair_sum(ee, 0.0, red, nws);
    if (tid == 0) cl.map_shared_rank(&sum_sh[2][q], 0)[0] = ee;
    cl.sync();  // the last access to another CTA's shared memory has been made
    if (q != 0 || warp != 0) return;
    ee = half_warp_sum(lane < nq ? sum_sh[2][lane & 15] : 0.0);
    if (lane == 0) {
        const double rh = sqrt(ee);
        P.R[((int64_t)prob * m + i) * m + i] = rii;
        P.d[(int64_t)prob * m + i] = di;
        P.rho[(int64_t)prob * m + i] = rh;
        cyc->dmax = dmax;
        cyc->dmin = dmin;
        cyc->k = i + 1;
        cyc->rho = rh;
        if (cyc->c3_on && cyc->c3_scale * rh <= cyc->c3_tol) {
            cyc->stopped = 1;
            cyc->reason = 3;
        } else if (i + 1 == m) {
            cyc->stopped = 1;
            cyc->reason = 1;
        }
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Per problem (one CTA): y = R_k^{-1} d by back substitution, coef_l = y_l sigma_l, in panels of 32 columns from the last.
// A panel's triangle is one warp's: lane q holds row q of the right-hand side, its row of the triangle (one wave of loads)
// and 1 / r_qq (the divisions of all rows at once); step l forms y_l in lane l (the product with the reciprocal and one
// correction step, as accurate as the division), shuffles it to the other lanes, and the rows above l subtract r_ql y_l.
// The other rows then subtract the panel's 32 products, a thread per row, whose entries of the panel were loaded while the
// triangle was solved.  A chain of k dependent steps, bound by FP64 and shuffle
// latency: 22 us on the mean of a 128^3 solve's cycles (k = 77) and 57 us at k = 200, against 70 and 182 us with a block barrier
// pair and a division on the path of every column.
constexpr int kLsThreads = 128;
__global__ void __launch_bounds__(kLsThreads) k_inner_ls(const Plan P) {
    extern __shared__ double rhs[];  // [k]
    __shared__ double ysh[32];
    const int p = blockIdx.x, m = P.m;
    if (P.pflag[p] & 1) return;
    const double* __restrict__ R = P.R + (int64_t)p * m * m;  // column-major: R[l*m + q] = R_{q,l}
    const double* __restrict__ d = P.d + (int64_t)p * m;
    const double* __restrict__ sigma = P.sigma + (int64_t)p * (m + 1);
    double* __restrict__ y = P.y + (int64_t)p * m;
    double* __restrict__ coef = P.coef + (int64_t)p * m;
    const int k = P.cyc[p].k;
    const int tid = threadIdx.x;
    for (int l = tid; l < k; l += kLsThreads) rhs[l] = d[l];
    __syncthreads();
    for (int l0 = (k - 1) & ~31; l0 >= 0; l0 -= 32) {  // columns l0 .. l1 - 1
        const int w = min(32, k - l0);
        double rq[32];  // warp 0: row l0 + lane of the triangle; the others: their first row's entries of the panel
        const int first = (tid < 32) ? l0 + tid : tid - 32;
        const bool mine = (tid < 32) ? tid < w : first < l0;
#pragma unroll
        for (int c = 0; c < 32; ++c)
            rq[c] = (mine && c < w && (tid >= 32 || tid <= c)) ? R[(int64_t)(l0 + c) * m + first] : 0.0;
        if (tid < 32) {
            double r = mine ? rhs[first] : 0.0;
            double rqq = 1.0;
#pragma unroll
            for (int c = 0; c < 32; ++c)
                if (c == tid && mine) rqq = rq[c];
            const double inv = 1.0 / rqq;
            double yq = 0.0;
#pragma unroll
            for (int c = 31; c >= 0; --c) {
                if (c >= w) continue;
                double t = r * inv;
                t = fma(fma(-t, rqq, r), inv, t);
                const double yl = __shfl_sync(0xffffffffu, t, c);
                if (tid == c) yq = yl;
                if (tid < c) r = fma(-rq[c], yl, r);
            }
            if (mine) {
                ysh[tid] = yq;
                y[first] = yq;
                coef[first] = yq * sigma[first];
            } else {
                ysh[tid] = 0.0;
            }
        }
        __syncthreads();
        if (tid >= 32) {
            for (int q = first; q < l0; q += kLsThreads - 32) {
                double r = rhs[q];
#pragma unroll
                for (int c = 31; c >= 0; --c)
                    r = fma(-((q == first) ? rq[c] : (c < w ? R[(int64_t)(l0 + c) * m + q] : 0.0)), ysh[c], r);
                rhs[q] = r;
            }
        }
        __syncthreads();
    }
}

// z = sum_{l<k} coef_l u_l, FP64 output.  FP64 basis: FP64 FMAs.  FP32/BF16 basis: the FP64 coefficients are split into
// two FP32 parts and the sum is carried as an unevaluated FP32 pair (TwoSum, and FMA for the exact product error),
// close to FP64 accuracy on the FP32 pipe.  Every row's sum runs over l in order.
//
// A pass over the k basis vectors with one multiply-add per value: bound by HBM for FP32 and BF16 bases, by the FP64 pipe
// for FP64 ones.
// Each row block is cut into pieces of kGemvThreads x R rows, one CTA each (grid y), so that the GPU holds as many
// threads as fit whatever the block size, and a thread loads L columns of its R rows (kGemvThreads apart: coalesced at
// any alignment) before it uses them.  Means over the cycles of a 128^3 solve: FP64 (77 columns) 530 -> 287 us (1.1 TFLOP/s,
// this GPU's FP64 rate), FP32 (93 columns) 775 -> 148 us (5.4 TB/s), both against one CTA of 256 threads per row block with
// one row's column in flight per thread.
constexpr int kGemvThreads = 256;
template <typename VT> struct GemvShape { static constexpr int R = 4, L = 4; };       // FP32, BF16
template <> struct GemvShape<double> { static constexpr int R = 2, L = 4; };

template <typename VT>
__global__ void __launch_bounds__(kGemvThreads) k_inner_gemv(const Plan P, double* __restrict__ z) {
    constexpr int R = GemvShape<VT>::R, L = GemvShape<VT>::L;
    constexpr bool F64 = sizeof(VT) == 8;
    using AT = typename std::conditional<F64, double, float>::type;
    __shared__ double cf[F64 ? kMaxM : 1];
    __shared__ float ch[F64 ? 1 : kMaxM], clo[F64 ? 1 : kMaxM];
    const BlockInfo bi = block_info(P, blockIdx.x);
    const int k0 = blockIdx.y * (kGemvThreads * R);  // the CTA's first row within the block
    if (k0 >= bi.len) return;
    const int p = bi.prob;
    if (P.pflag[p] & 1) return;
    const int k = P.cyc[p].k;
    const int64_t N = P.N;
    const double* coef = P.coef + (int64_t)p * P.m;
    for (int l = threadIdx.x; l < k; l += kGemvThreads) {
        const double c = coef[l];
        if constexpr (F64) {
            cf[l] = c;
        } else {
            const float hi = (float)c;
            ch[l] = hi;
            clo[l] = (float)(c - (double)hi);
        }
    }
    __syncthreads();
    const VT* ub = (const VT*)P.U + bi.v0 + k0 + threadIdx.x;
    bool ok[R];
#pragma unroll
    for (int r = 0; r < R; ++r) ok[r] = k0 + (int)threadIdx.x + r * kGemvThreads < bi.len;
    AT sh[R], sl[R];
#pragma unroll
    for (int r = 0; r < R; ++r) sh[r] = sl[r] = AT(0);
    auto add = [&](int l, int r, AT u) {
        if constexpr (F64) {
            sh[r] = fma(cf[l], u, sh[r]);
        } else {
            const float pr = ch[l] * u;
            const float pe = fmaf(ch[l], u, -pr) + clo[l] * u;  // exact product error + low-part term
            const float t1 = sh[r] + pr;                         // TwoSum(sh, pr)
            const float bv = t1 - sh[r];
            const float err = (sh[r] - (t1 - bv)) + (pr - bv);
            sh[r] = t1;
            sl[r] += err + pe;
        }
    };
    int l = 0;
    for (; l + L <= k; l += L) {
        AT u[L][R];
#pragma unroll
        for (int q = 0; q < L; ++q)
#pragma unroll
            for (int r = 0; r < R; ++r) u[q][r] = ok[r] ? ld_plain(ub + (l + q) * N + r * kGemvThreads) : AT(0);
#pragma unroll
        for (int q = 0; q < L; ++q)
#pragma unroll
            for (int r = 0; r < R; ++r) add(l + q, r, u[q][r]);
    }
    for (; l < k; ++l)
#pragma unroll
        for (int r = 0; r < R; ++r) add(l, r, ok[r] ? ld_plain(ub + l * N + r * kGemvThreads) : AT(0));
    double* zb = z + bi.v0 + k0 + threadIdx.x;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (ok[r]) {
            if constexpr (F64) zb[r * kGemvThreads] = sh[r];
            else zb[r * kGemvThreads] = (double)sh[r] + (double)sl[r];
        }
}

template <typename VT>
static void inner_gemv(const Plan& p, double* z) {
    constexpr int rows = kGemvThreads * GemvShape<VT>::R;
    k_inner_gemv<VT><<<dim3(p.nblk, (p.Bn + rows - 1) / rows), kGemvThreads, 0, p.st>>>(p, z);
}

template <typename VT>
__global__ void k_export_basis(const Plan P, int count, double* __restrict__ out) {
    const BlockInfo bi = block_info(P, blockIdx.x);
    const double* sigma = P.sigma + (int64_t)bi.prob * (P.m + 1);
    const VT* Ub = (const VT*)P.U;
    for (int kk = threadIdx.x; kk < bi.len; kk += blockDim.x) {
        const int64_t r = bi.v0 + kk;
        for (int l = 0; l < count; ++l)
            out[(int64_t)l * P.N + r] = sigma[l] * (double)ld_plain(Ub + (int64_t)l * P.N + r);
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Start of inner cycle j, per problem: reset the cycle state (C3 scale = FFOM residual of the previous outer step,
// beta at the first, Eq. 5); a problem that is done is marked stopped so every inner kernel skips it.
__global__ void k_cycle_reset(const Plan P, int j, int c3_on, double cond_thr) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P.P) return;
    CycleState* cyc = P.cyc + p;
    cyc->stopped = (P.pflag[p] & 1) ? 1 : 0;
    cyc->k = 0;
    cyc->reason = 0;
    cyc->brk_step = INT_MAX;
    cyc->brk_reason = 0;
    cyc->dmax = 0.0;
    cyc->dmin = INFINITY;
    cyc->rho = INFINITY;
    cyc->cond_thr = cond_thr;
    if (p == 0 && P.gsync) {  // the fused step's grid counters (0: phase-1 partials, 2: sketch partials), give-up flag
        P.gsync[0] = 0;
        P.gsync[1] = 0;
        P.gsync[2] = 0;
    }
    if (j >= 0) {
        const OuterState* ost = P.ost + p;
        const double sc = (j == 0) ? ost->beta : ost->ffom;
        cyc->c3_scale = sc;
        cyc->c3_tol = ost->tol_abs;
        cyc->c3_on = (c3_on && isfinite(sc)) ? 1 : 0;
    } else {
        cyc->c3_scale = INFINITY;
        cyc->c3_tol = 0.0;
        cyc->c3_on = 0;
    }
    P.sigma[(int64_t)p * (P.m + 1)] = 1.0;
}

void launch_cycle_start(const Plan& p, int j, const double* v, const double* vscale, int vstride, int c3_on,
                        double cond_thr) {
    k_cycle_reset<<<(p.P + 127) / 128, 128, 0, p.st>>>(p, j, c3_on, cond_thr);
    launch_sketch_partials(p, v, vscale, vstride, p.U, p.cpart);
    launch_sketch_reduce(p, p.cpart, p.c0, p.e);
    ++g_launches;
}

void launch_inner_spmv(const Plan& p, int i) {
    if (p.prec == kFP64) inner_spmv_f64(p, i);
    else if (p.prec == kFP32) inner_spmv_f32(p, i);
    else inner_spmv_bf16(p, i);
    ++g_launches;
}

bool launch_inner_step(const Plan& p, int i, bool last) {
    if (!p.gsync) return false;
    bool ok;
    if (p.prec == kFP64) ok = inner_step_f64(p, i, last);
    else if (p.prec == kFP32) ok = inner_step_f32(p, i, last);
    else ok = inner_step_bf16(p, i, last);
    if (ok) ++g_launches;
    return ok;
}

void launch_inner_axpy(const Plan& p, int i, bool last) {
    if (p.prec == kFP64) inner_axpy_f64(p, i, last);
    else if (p.prec == kFP32) inner_axpy_f32(p, i, last);
    else inner_axpy_bf16(p, i, last);
    ++g_launches;
}

// The kernel for a shape, with the attributes that its launches need.
using QrKernel = void (*)(const Plan, int);
static cudaError_t qr_kernel(const QrShape& q, int s, int m, int i, QrKernel* fn) {
    const bool lg = qr_long(s, q.cluster, i);
    if (q.staged) *fn = lg ? k_inner_qr<true, true> : k_inner_qr<true, false>;
    else *fn = lg ? k_inner_qr<false, true> : k_inner_qr<false, false>;
    set_smem((const void*)*fn, qr_smem(q, m, m - 1));
    return q.cluster > kQrPortable
               ? cudaFuncSetAttribute((const void*)*fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)
               : cudaSuccess;
}

bool qr_places(const QrShape& q, int s, int m) {
    QrKernel fn;
    int clusters = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)q.cluster, 1, 1);
    cfg.blockDim = dim3(kQrThreads, 1, 1);
    cfg.dynamicSmemBytes = qr_smem(q, m, m - 1);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = q.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (qr_kernel(q, s, m, m - 1, &fn) == cudaSuccess && cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) == cudaSuccess)
        return clusters > 0;
    cudaGetLastError();
    return false;
}

cudaError_t launch_inner_qr(const Plan& p, int i, cudaStream_t st) {
    const QrShape& q = p.qr;
    QrKernel fn;
    const cudaError_t e = qr_kernel(q, p.s, p.m, i, &fn);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(q.cluster * p.P), 1, 1);
    cfg.blockDim = dim3(kQrThreads, 1, 1);
    cfg.dynamicSmemBytes = qr_smem(q, p.m, i);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = q.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    ++g_launches;
    return cudaLaunchKernelEx(&cfg, fn, p, i);
}

void launch_inner_finish(const Plan& p, double* z) {
    set_smem((const void*)k_inner_ls, (size_t)p.m * sizeof(double));
    k_inner_ls<<<p.P, kLsThreads, (size_t)p.m * sizeof(double), p.st>>>(p);
    if (p.prec == kFP64) inner_gemv<double>(p, z);
    else if (p.prec == kFP32) inner_gemv<float>(p, z);
    else inner_gemv<__nv_bfloat16>(p, z);
    g_launches += 2;
}

void launch_export_basis(const Plan& p, double* out, int count) {
    if (p.prec == kFP64) k_export_basis<double><<<p.nblk, 256, 0, p.st>>>(p, count, out);
    else if (p.prec == kFP32) k_export_basis<float><<<p.nblk, 256, 0, p.st>>>(p, count, out);
    else k_export_basis<__nv_bfloat16><<<p.nblk, 256, 0, p.st>>>(p, count, out);
    ++g_launches;
}

}  // namespace sfg
