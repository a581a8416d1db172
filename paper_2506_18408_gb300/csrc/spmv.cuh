// CSR SpMV over one row block, result into shared memory (used by the inner and outer steps).
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace sfg {

// CNT entries (compile-time count) of one row chunk: loads first, then exactly CNT FMAs.  Lanes whose row has
// fewer entries in this chunk are predicated off; the warp issues no instruction for slots no lane needs.
template <int CNT, typename MT, typename XT, typename AT>
__device__ __forceinline__ void row_chunk(const int* __restrict__ col, const MT* __restrict__ val,
                                          const XT* __restrict__ x, int a, int len, int pk, AT& sum) {
    int c[CNT];
    AT v[CNT];
#pragma unroll
    for (int q = 0; q < CNT; ++q) {
        if (pk + q < len) {
            c[q] = __ldg(col + a + pk + q);
            v[q] = (AT)__ldg(val + a + pk + q);
        }
    }
#pragma unroll
    for (int q = 0; q < CNT; ++q)
        if (pk + q < len) sum += v[q] * load_as(x + c[q], AT());
}

// out[r - r0] = sum_p val[p] * x[col[p]] for rows r in [r0, r1), one thread per row.
// Warps walk the rows together; each row is read in chunks of up to 4 entries whose count is the longest row of
// the warp in that chunk, dispatched to a compile-time count, so the number of FMA instructions a warp issues is
// exactly its longest row (with no shuffle tree): the FP64 pipe, scarce on this GPU, does only useful work.
// The next row group's extents are fetched while the current one is summed.  Sums run in entry order.
template <typename MT, typename XT, typename AT>
__device__ __forceinline__ void spmv_rows_scalar(const int* __restrict__ rp, const int* __restrict__ col,
                                                 const MT* __restrict__ val, const XT* __restrict__ x, int r0,
                                                 int r1, AT* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    int rw = r0 + (threadIdx.x & ~31);
    int a = 0, len = 0;
    if (rw + lane < r1) {
        a = __ldg(rp + rw + lane);
        len = __ldg(rp + rw + lane + 1) - a;
    }
    for (; rw < r1; rw += blockDim.x) {  // warp-uniform loop
        const int rn = rw + (int)blockDim.x + lane;
        int an = 0, lenn = 0;
        if (rn < r1) {
            an = __ldg(rp + rn);
            lenn = __ldg(rp + rn + 1) - an;
        }
        const int maxlen = (int)__reduce_max_sync(0xffffffffu, (unsigned)len);
        AT sum = AT(0);
        for (int pk = 0; pk < maxlen; pk += 4) {
            switch (min(maxlen - pk, 4)) {
                case 1: row_chunk<1>(col, val, x, a, len, pk, sum); break;
                case 2: row_chunk<2>(col, val, x, a, len, pk, sum); break;
                case 3: row_chunk<3>(col, val, x, a, len, pk, sum); break;
                case 4: row_chunk<4>(col, val, x, a, len, pk, sum); break;
                default: row_chunk<4>(col, val, x, a, len, pk, sum); break;
            }
        }
        if (rw + lane < r1) out[rw + lane - r0] = sum;
        a = an;
        len = lenn;
    }
}

// ---- one thread per row with the entries staged in shared memory ----
// A warp takes 32 consecutive rows at a time.  Their entries are one stretch of the CSR arrays, which the warp copies
// into its own part of shared memory with asynchronous 16-byte copies (from the 16-byte boundary at or below; the
// arrays are padded, so a copy may run past the last entry), one group of rows ahead: a group's columns and values are there
// when its turn comes, every copy is coalesced whatever the row lengths, and what a row waits for is one round of gathers of x
// (up to eight in flight per lane).  Used by the FP32 and BF16 inner cycles and by the FP64 kernels of the outer iteration.  Read straight from global memory, lanes 7 entries apart touch 20 sectors per load, and a
// row of 7 entries waits for two rounds of loads and gathers.  A group's values go to registers before its last products,
// which frees the buffer for the next group's copy.  Rows are summed in entry order, a warp issuing as many products as its
// longest row.  128^3 solve to 1e-12 with FP32 inner cycles: 45.8 -> 42.3 ms.  FP64 inner cycles keep the SELL-32 copy (staged:
// 46.4 -> 57.6 ms, the buffers of two CTAs beside their blocks of w' leave 28 KB of L1).
constexpr int kVecStaged = -2;  // template value of the lanes-per-row parameter for this form

template <typename MT>
__host__ __device__ constexpr int stage_bytes(int maxlen) {  // one warp's buffer for rows of at most maxlen entries
    return 32 * maxlen * (4 + (int)sizeof(MT)) + 32;
}

__device__ __forceinline__ void cp_async16(unsigned dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Starts the copy of entries [a0, a1) into a warp's buffer (columns at cdst, values at vdst).
template <typename MT>
__device__ __forceinline__ void stage_issue(const int* __restrict__ col, const MT* __restrict__ val, int a0, int a1,
                                            unsigned cdst, unsigned vdst, int lane) {
    constexpr int VP = 16 / (int)sizeof(MT);
    const int ca = a0 & ~3, va = a0 & ~(VP - 1);
    // unsigned: a lane's offset may pass 2^31 - 1 entries before it ends the loop
    for (unsigned u = lane; ca + 4 * u < (unsigned)a1; u += 32) cp_async16(cdst + 16 * u, col + ca + 4 * u);
    for (unsigned u = lane; va + VP * u < (unsigned)a1; u += 32) cp_async16(vdst + 16 * u, val + va + VP * u);
}

// Entries pk .. pk+CNT-1 of the lane's row (its first entry at cs, vs in shared memory), get(c) the factor of column c;
// `release` runs once the values are in registers.
template <int CNT, typename MT, typename AT, typename Get, typename Release>
__device__ __forceinline__ void staged_chunk(const int* cs, const MT* vs, Get&& get, int len, int pk, AT& sum,
                                             Release&& release) {
    AT xv[CNT], v[CNT];
#pragma unroll
    for (int q = 0; q < CNT; ++q) xv[q] = (pk + q < len) ? get(cs[pk + q]) : AT(0);
#pragma unroll
    for (int q = 0; q < CNT; ++q) v[q] = (pk + q < len) ? (AT)vs[pk + q] : AT(0);
    release();
#pragma unroll
    for (int q = 0; q < CNT; ++q)
        if (pk + q < len) sum += v[q] * xv[q];
}

// The whole of every row (the default of rows_staged's Part).
struct WholeRows {
    __device__ __forceinline__ int load(int) const { return 0; }
    __device__ __forceinline__ void cut(int, int, int&, int&) const {}
};

// For the len rows from matrix row r0 on (row pointers rpm = rp + r0): pre(k) before local row k's products (loads that
// should be in flight with them), then emit(k, sum of val * get(col) over the row's entries, or over the part that
// part.cut(part.load(k), first entry, offset, count) leaves of them; load runs a group ahead).  Lanes past the last row call
// all with k >= len.  buf: the CTA's stage area (blockDim / 32 buffers of stage_bytes(maxlen)).
template <typename MT, typename AT, typename Get, typename Part, typename Pre, typename Emit>
__device__ __forceinline__ void rows_staged(const int* __restrict__ rpm, const int* __restrict__ col,
                                            const MT* __restrict__ val, int len, unsigned char* buf, int maxlen,
                                            Get&& get, Part part, Pre&& pre, Emit&& emit) {
    const int lane = threadIdx.x & 31;
    unsigned char* mine = buf + (threadIdx.x >> 5) * stage_bytes<MT>(maxlen);
    int* cbuf = reinterpret_cast<int*>(mine);
    MT* vbuf = reinterpret_cast<MT*>(mine + 128 * maxlen + 16);
    const unsigned cdst = (unsigned)__cvta_generic_to_shared(cbuf), vdst = (unsigned)__cvta_generic_to_shared(vbuf);
    constexpr int VP = 16 / (int)sizeof(MT);
    int kw = threadIdx.x & ~31;
    if (kw >= len) return;
    // first entry and length of the lane's row in the group at k0 (past the last row: its end, 0)
    auto extent = [&](int k0, int& a, int& l, int& d) {
        a = __ldg(rpm + min(k0 + lane, len));
        l = __ldg(rpm + min(k0 + lane + 1, len)) - a;
        d = part.load(k0 + lane);
    };
    auto issue = [&](int a, int l) {
        stage_issue(col, val, __shfl_sync(0xffffffffu, a, 0), __shfl_sync(0xffffffffu, a + l, 31), cdst, vdst, lane);
    };
    int a, rl, d, an = 0, rln = 0, dn = 0;
    extent(kw, a, rl, d);
    issue(a, rl);
    if (kw + (int)blockDim.x < len) extent(kw + blockDim.x, an, rln, dn);
    for (; kw < len; kw += blockDim.x) {  // warp-uniform loop
        const bool more = kw + (int)blockDim.x < len;
        pre(kw + lane);
        const int a0 = __shfl_sync(0xffffffffu, a, 0);
        int off = 0;
        if (kw + lane < len) part.cut(d, a, off, rl);
        const int* cs = cbuf + (a + off - (a0 & ~3));
        const MT* vs = vbuf + (a + off - (a0 & ~(VP - 1)));
        const int wm = (int)__reduce_max_sync(0xffffffffu, (unsigned)rl);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        AT sum = AT(0);
        auto release = [&]() {  // every lane has read the buffer: the next group's entries may come in
            __syncwarp();
            if (more) issue(an, rln);
        };
        int pk = 0;
        for (; pk + 8 < wm; pk += 8) staged_chunk<8>(cs, vs, get, rl, pk, sum, [] {});
        switch (wm - pk) {
            case 1: staged_chunk<1>(cs, vs, get, rl, pk, sum, release); break;
            case 2: staged_chunk<2>(cs, vs, get, rl, pk, sum, release); break;
            case 3: staged_chunk<3>(cs, vs, get, rl, pk, sum, release); break;
            case 4: staged_chunk<4>(cs, vs, get, rl, pk, sum, release); break;
            case 5: staged_chunk<5>(cs, vs, get, rl, pk, sum, release); break;
            case 6: staged_chunk<6>(cs, vs, get, rl, pk, sum, release); break;
            case 7: staged_chunk<7>(cs, vs, get, rl, pk, sum, release); break;
            case 8: staged_chunk<8>(cs, vs, get, rl, pk, sum, release); break;
            default: release(); break;  // rows without entries
        }
        emit(kw + lane, sum);
        a = an;
        rl = rln;
        d = dn;
        if (kw + 2 * (int)blockDim.x < len) extent(kw + 2 * (int)blockDim.x, an, rln, dn);
    }
}

// rows_staged of whole rows against a vector x: A x.
template <typename MT, typename XT, typename AT, typename Pre, typename Emit>
__device__ __forceinline__ void spmv_rows_staged(const int* __restrict__ rpm, const int* __restrict__ col,
                                                 const MT* __restrict__ val, const XT* __restrict__ x, int len,
                                                 unsigned char* buf, int maxlen, Pre&& pre, Emit&& emit) {
    rows_staged<MT, AT>(rpm, col, val, len, buf, maxlen, [&](int c) { return load_as(x + c, AT()); }, WholeRows(), pre,
                        emit);
}

// Same result with each row handled by a sub-warp of V lanes; a warp processes U sub-warp rows at once (all their
// loads issued before the FMAs).  For a fixed unroll slot the warp's sub-warps read consecutive rows, so the
// col/val streams are read in contiguous segments.  Per-row sums are combined by a fixed xor-shuffle tree.
// Suited to long or irregular rows.
template <int V, int U, typename MT, typename XT, typename AT>
__device__ __forceinline__ void spmv_rows_vector(const int* __restrict__ rp, const int* __restrict__ col,
                                                 const MT* __restrict__ val, const XT* __restrict__ x, int r0,
                                                 int r1, AT* __restrict__ out) {
    constexpr int SUBS = 32 / V;
    constexpr int TILE = SUBS * U;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int sub = lane / V, sl = lane % V;
    for (int tb = r0 + warp * TILE; tb < r1; tb += nwarps * TILE) {
        int beg[U], len[U];
        int maxlen = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int row = tb + u * SUBS + sub;
            if (row < r1) {
                beg[u] = __ldg(rp + row);
                len[u] = __ldg(rp + row + 1) - beg[u];
            } else {
                beg[u] = 0;
                len[u] = 0;
            }
            maxlen = max(maxlen, len[u]);
        }
        AT sum[U];
#pragma unroll
        for (int u = 0; u < U; ++u) sum[u] = AT(0);
        for (int p = sl; p < maxlen; p += V) {
            int c[U];
            AT v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (p < len[u]) {
                    c[u] = __ldg(col + beg[u] + p);
                    v[u] = (AT)__ldg(val + beg[u] + p);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (p < len[u]) sum[u] += v[u] * load_as(x + c[u], AT());
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int o = V / 2; o > 0; o >>= 1) sum[u] += __shfl_xor_sync(0xffffffffu, sum[u], o);
            const int row = tb + u * SUBS + sub;
            if (sl == 0 && row < r1) out[row - r0] = sum[u];
        }
    }
}

// Rows [lo, hi) of a block's length-sorted order (local offsets pm[i]), each handled by a sub-warp of V lanes, U rows
// per sub-warp at once, each lane taking E entries of a row per pass (all loads of a pass issued before its FMAs,
// so E * U gathers per lane are in flight); a lane's entries are p, p + V, p + 2V, ... in that order and the per-row
// sums are combined by a fixed xor-shuffle tree.
template <int V, int U, int E, typename MT, typename XT, typename AT>
__device__ __forceinline__ void spmv_sorted_vector(const int* __restrict__ rpm, const int* __restrict__ col,
                                                   const MT* __restrict__ val, const XT* __restrict__ x,
                                                   const uint16_t* __restrict__ pm, int lo, int hi,
                                                   AT* __restrict__ out) {
    constexpr int SUBS = 32 / V;
    constexpr int TILE = SUBS * U;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int sub = lane / V, sl = lane % V;
    for (int tb = lo + warp * TILE; tb < hi; tb += nwarps * TILE) {
        int beg[U], len[U], kk[U];
        int maxlen = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = tb + u * SUBS + sub;
            kk[u] = -1;
            beg[u] = 0;
            len[u] = 0;
            if (i < hi) {
                kk[u] = pm[i];
                const int* rq = rpm + kk[u];
                beg[u] = __ldg(rq);
                len[u] = __ldg(rq + 1) - beg[u];
            }
            maxlen = max(maxlen, len[u]);
        }
        maxlen = (int)__reduce_max_sync(0xffffffffu, (unsigned)maxlen);
        AT sum[U];
#pragma unroll
        for (int u = 0; u < U; ++u) sum[u] = AT(0);
        for (int p0 = sl; p0 < maxlen; p0 += E * V) {
            int c[U][E];
            AT v[U][E];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int p = p0 + e * V;
                    if (p < len[u]) {
                        c[u][e] = __ldg(col + beg[u] + p);
                        v[u][e] = (AT)__ldg(val + beg[u] + p);
                    }
                }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (p0 + e * V < len[u]) sum[u] += v[u][e] * load_as(x + c[u][e], AT());
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int o = V / 2; o > 0; o >>= 1) sum[u] += __shfl_xor_sync(0xffffffffu, sum[u], o);
            if (sl == 0 && kk[u] >= 0) out[kk[u]] = sum[u];
        }
    }
}

// CNT entries of the lane's row in a slice of the sorted copy (cp, vp: the lane's first; consecutive entries 32 apart),
// entries past the row's end (rl) not gathered.  The matrix streams through once: loads that do not stay in the caches.
template <int CNT, typename MT, typename XT, typename AT>
__device__ __forceinline__ void sorted_chunk(const int* __restrict__ cp, const MT* __restrict__ vp,
                                             const XT* __restrict__ x, int rl, int pk, AT& sum) {
    int c[CNT];
    AT xv[CNT], v[CNT];
#pragma unroll
    for (int q = 0; q < CNT; ++q) c[q] = __ldcs(cp + (pk + q) * 32);
#pragma unroll
    for (int q = 0; q < CNT; ++q) v[q] = (AT)__ldcs(vp + (pk + q) * 32);
#pragma unroll
    for (int q = 0; q < CNT; ++q) xv[q] = (pk + q < rl) ? load_as(x + c[q], AT()) : AT(0);
#pragma unroll
    for (int q = 0; q < CNT; ++q)
        if (pk + q < rl) sum += v[q] * xv[q];
}

// *out = the lane's row in a slice of w entries per row (out: a shared slot, null for lanes without a row).
//
// Up to 16 entries are one running sum.  A longer row's error would grow with its length (one running sum had 1.4 to 4.4
// times the error of lanes' sums joined by a tree at 17 to 512 entries), so it is summed in chunks of at most eight of nearly one
// size, each as two interleaved sums; the chunks' sums are added in groups, two of them up to 64 entries and of four chunks
// beyond, and the groups into *out, the third and later ones with what that addition lost carried into the next group.  Against
// the lanes' sums (8 up to 64 entries, else 32) that measures 1.02 to 1.05 of the error at 17 to 32 entries, 1.00 to 0.95 up to
// 64, 1.03 at 65, 0.98 at 96, 0.83 at 256 and 0.71 at 512 (a dominant entry anywhere in the row, normal values; FP32 and FP64
// alike).  The total stays in shared memory and a chunk's columns are loaded with the one before: eight gathers in flight
// leave a thread of the FP64 kernels' 56 registers no room for a second set of sums.
// Cycles of 60 steps on Zipf rows with one running sum and so, ms: FP64 2M rows 18.0 and 17.9, 1M 10.05 and 10.20, 700,000 9.84 and 9.79;
// FP32 2M 14.4 and 14.7, 1M 7.87 and 7.75.  (Eight running sums per row: 18.8, 10.5 and 10.0 with eight loads in flight, which spill,
// 17.2, 10.7 and 11.0 with four.)
template <typename MT, typename XT, typename AT>
__device__ __forceinline__ void sorted_row(const int* __restrict__ cp, const MT* __restrict__ vp,
                                           const XT* __restrict__ x, int rl, int w, AT* out) {
    int pk = 0;
    AT sum = AT(0);
    if (w <= 16) {
        for (; pk + 8 < w; pk += 8) sorted_chunk<8>(cp, vp, x, rl, pk, sum);
        switch (w - pk) {
            case 1: sorted_chunk<1>(cp, vp, x, rl, pk, sum); break;
            case 2: sorted_chunk<2>(cp, vp, x, rl, pk, sum); break;
            case 3: sorted_chunk<3>(cp, vp, x, rl, pk, sum); break;
            case 4: sorted_chunk<4>(cp, vp, x, rl, pk, sum); break;
            case 5: sorted_chunk<5>(cp, vp, x, rl, pk, sum); break;
            case 6: sorted_chunk<6>(cp, vp, x, rl, pk, sum); break;
            case 7: sorted_chunk<7>(cp, vp, x, rl, pk, sum); break;
            case 8: sorted_chunk<8>(cp, vp, x, rl, pk, sum); break;
            default: break;
        }
        if (out) *out = sum;
        return;
    }
    const int chunks = (w + 7) / 8, step = (w + chunks - 1) / chunks, group = chunks <= 8 ? (chunks + 1) / 2 : 4;
    int c[8], left = group;
    bool first = true;
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if (q < step) c[q] = __ldcs(cp + q * 32);
    for (; pk < w; pk += step) {
        const int cnt = min(step, w - pk), next = min(step, w - pk - step);
        AT v[8], xv[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = (q < cnt) ? (AT)__ldcs(vp + (pk + q) * 32) : AT(0);
#pragma unroll
        for (int q = 0; q < 8; ++q) xv[q] = (q < cnt && pk + q < rl) ? load_as(x + c[q], AT()) : AT(0);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < next) c[q] = __ldcs(cp + (pk + step + q) * 32);
        AT s0 = AT(0), s1 = AT(0);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < cnt && pk + q < rl) {
                if (q & 1) s1 += v[q] * xv[q];
                else s0 += v[q] * xv[q];
            }
        sum += s0 + s1;
        if (--left == 0 && next > 0) {  // a group but the last
            left = group;
            if (first) {
                if (out) *out = sum;
                sum = AT(0);
                first = false;
            } else {
                const AT t0 = out ? *out : AT(0), t = t0 + sum, d = t - t0;
                const AT lost = (t0 - (t - d)) + (sum - d);
                if (out) *out = t;
                sum = isfinite(t) ? lost : AT(0);
            }
        }
    }
    if (out) *out += sum;
}

// Length-binned SpMV of one block for matrices with irregular rows: out[k] for the block's local rows k, matrix rows
// m0 + k.  The block's rows come in a precomputed order pm[0 .. len) (local offsets), by length.  The first so.na, those of the
// sorted copy, take one thread each, 32 rows of (nearly) one length per warp from a slice that the warp reads
// coalesced: every FP64 instruction does 32 rows' products and no sum needs a shuffle tree (with 8 lanes or a warp per row
// the trees and half-empty passes doubled the FP64 instructions of a 2M-row Zipf matrix, on a GPU whose FP64 pipe takes 17
// cycles per warp and instruction).  Warps take the slices longest first, in alternating direction, so that their loads
// even out.  2M rows, FP64, one running sum per row: 270 -> 235 us per launch; whole steps 1M rows 227 -> 164 us, 1.5M FP32 213 ->
// 179 us (sorted_row has what its order of sums costs beside that).
// The rows that the copy leaves (too long for the block, or slices that would be half empty) take 8 lanes (up to 64 entries) or a
// warp from the CSR arrays.  Every row's sum runs over its entries in a fixed order.
template <typename MT, typename XT, typename AT>
__device__ __forceinline__ void spmv_rows_binned(const int* __restrict__ rp, const int* __restrict__ col,
                                                 const MT* __restrict__ val, const XT* __restrict__ x, int m0, int len,
                                                 const uint16_t* __restrict__ perm, const SortedRows<MT>& so,
                                                 AT* __restrict__ out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const uint16_t* pm = perm + m0;
    const int* rpm = rp + m0;
    const int ns = (so.na + 31) / 32;
    for (int t0 = 0, flip = 0; t0 < ns; t0 += nwarps, flip ^= 1) {
        const int t = t0 + (flip ? nwarps - 1 - warp : warp);
        if (t >= ns) continue;
        const int s = ns - 1 - t, i = 32 * s + lane;
        const int o = __ldg(so.off + s), w = __ldg(so.off + s + 1) - o, rl = so.len[(int64_t)s * 32 + lane];
        const int k = (i < so.na) ? pm[i] : -1;
        const int* cp = so.col + (int64_t)o * 32 + lane;
        const MT* vp = so.val + (int64_t)o * 32 + lane;
        sorted_row<MT, XT, AT>(cp, vp, x, rl, w, k >= 0 ? out + k : nullptr);
    }
    const int mid = max(so.na, so.n64);
    spmv_sorted_vector<8, 2, 2, MT, XT, AT>(rpm, col, val, x, pm, so.na, mid, out);
    spmv_sorted_vector<32, 2, 4, MT, XT, AT>(rpm, col, val, x, pm, mid, len, out);
}

// V == 0: length-binned (perm, so as for spmv_rows_binned); V == 1: one thread per row; else V lanes per row.
template <int V, int U, typename MT, typename XT, typename AT>
__device__ __forceinline__ void spmv_rows_to_smem(const int* __restrict__ rp, const int* __restrict__ col,
                                                  const MT* __restrict__ val, const XT* __restrict__ x, int r0,
                                                  int r1, AT* __restrict__ out, const uint16_t* perm,
                                                  const SortedRows<MT>& so) {
    if constexpr (V == 0) spmv_rows_binned<MT, XT, AT>(rp, col, val, x, r0, r1 - r0, perm, so, out);
    else if constexpr (V == 1) spmv_rows_scalar<MT, XT, AT>(rp, col, val, x, r0, r1, out);
    else spmv_rows_vector<V, U, MT, XT, AT>(rp, col, val, x, r0, r1, out);
}

// Dispatch on the lanes-per-row width chosen at run time (-2 = one thread per row with staged entries, 0 = length-binned, 1 =
// one thread per row, else 2..32).
#define SFG_SPMV_DISPATCH(V_RUNTIME, CALL)                       \
    switch (V_RUNTIME) {                                         \
        case -2: { constexpr int VV = -2, UU = 1; CALL; } break; \
        case 0: { constexpr int VV = 0, UU = 1; CALL; } break;   \
        case 1: { constexpr int VV = 1, UU = 1; CALL; } break;   \
        case 2: { constexpr int VV = 2, UU = 4; CALL; } break;   \
        case 4: { constexpr int VV = 4, UU = 4; CALL; } break;   \
        case 8: { constexpr int VV = 8, UU = 4; CALL; } break;   \
        case 16: { constexpr int VV = 16, UU = 2; CALL; } break; \
        default: { constexpr int VV = 32, UU = 2; CALL; } break; \
    }

}  // namespace sfg
