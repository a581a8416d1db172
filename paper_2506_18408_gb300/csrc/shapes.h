// Shape rules of the launchers that need no device: plain C++.
#pragma once

#include <algorithm>
#include <cstddef>

namespace sfg {

constexpr int kQrCluster = 16;   // most CTAs of the cluster that runs a sketched QR update
constexpr int kQrThreads = 128;  // threads of such a CTA
constexpr int kQrPortable = 8;   // the largest cluster that every device of the architecture places

// Shape of the sketched-QR update.
struct QrShape {
    int cluster = 8;     // CTAs per problem (one cluster)
    int nrp = 0;         // rows of Q per CTA, padded to an odd number
    int slice = 0;       // doubles of one CTA's slice of Q (nrp * m, even)
    bool staged = false; // the slice is kept in shared memory during an update
};

// Dynamic shared memory of update i: the staged columns, the CTA's rows of p and e, the projections and their parts.
inline size_t qr_smem(const QrShape& q, int m, int i) {
    return ((size_t)(q.staged ? (i * q.nrp + 1) & ~1 : 0) + 2 * (size_t)q.nrp + 3 * (size_t)m) * sizeof(double);
}

// Whether a thread's part of one of update i's products (k_inner_qr: rows of a group, columns of a group) passes 16 terms.  Two
// sums where the parts are short cost a 64^2 solve (8 terms) 1.5 %; where they are long, 0.5 % of an 80^3 cycle at s = 1000, m = 200, and
// four sums 2.5 %.
inline bool qr_long(int s, int cluster, int i) {
    const int nr = (s + cluster - 1) / cluster;
    int gp = 1, wr = 32;
    while (gp < 8 && 2 * gp * i <= kQrThreads && 4 * gp <= nr) gp *= 2;
    while (wr < nr && wr < kQrThreads) wr *= 2;
    return (nr + gp - 1) / gp > 16 || (i * wr + kQrThreads - 1) / kQrThreads > 16;
}

// The shape for P problems, sketch size s and basis size m, given the shared memory a QR CTA may take; binned: the step's SpMV
// is the length-binned one.  The cluster, on which the rounding of the sums depends, is the same for steps of one and of two
// launches.
//
// Few CTAs where an update's FP64 work is small (its latency is then the exchanges, which grow with the CTAs), many where it
// is large.  Whole solves, 2 / 4 / 8 / 16 CTAs: s = 80, m = 20 (2D 32^2) 2.40 / 2.51 / 2.54 / 2.49 ms; s = 120, m = 30 (2D
// 64^2) 4.34 / 4.12 / 5.21 / 5.03 ms; s = 240, m = 60 (3D 32^3) 3.36 / 3.19 / 3.56 / 3.41 ms; s = 320, m = 80 (40^3) 4.96 / 4.47
// / 4.06 / 3.90 ms; s = 1000, m = 200 (80^3) 44.3 / 28.9 / 20.9 / 15.9 ms; beside the length-binned SpMV, s = 120, m = 30
// (30,000 Zipf rows) 19.6 / 20.8 / 20.8 / 20.9 ms.  Batches take what leaves the problems' clusters
// side by side on the GPU.
//
// Clusters beyond the portable size are taken where places(shape) says that the device can hold one (all of a cluster's CTAs lie in
// one group of SMs, which has fewer of them on a partition of a GPU): staged, else read from L2, else the portable size.
template <typename Places>
QrShape qr_shape(int P, int s, int m, size_t smem_left, bool binned, Places&& places) {
    const int most = P <= 4 ? kQrCluster : P <= 16 ? 8 : P <= 32 ? 4 : P <= 64 ? 2 : 1;
    const int want = std::min(most, s * m <= (binned ? 5000 : 3000) ? 2 : s * m <= 20000 ? 4 : kQrCluster);
    auto shape = [&](int cluster) {
        QrShape q;
        q.cluster = cluster;
        q.nrp = ((s + cluster - 1) / cluster) | 1;
        q.slice = (q.nrp * m + 1) & ~1;
        q.staged = true;
        q.staged = qr_smem(q, m, m - 1) + 3072 <= smem_left;  // its static shared memory and the reserve
        return q;
    };
    QrShape q = shape(want);
    if (want <= kQrPortable || places(q)) return q;
    if (q.staged) {
        q.staged = false;
        if (places(q)) return q;
    }
    return shape(kQrPortable);
}

}  // namespace sfg
