// How a selection, and the row copies of a small layer step, are handed to CTAs.  Plain arithmetic on the host, without device
// code, so that a host compiler can check it.  select.cu describes the kernels.
#pragma once
#include "common.cuh"

namespace pafu {

constexpr int kSelThreads = 256;            // block of a CTA with a short share; kSelThreadsMax with a long one
constexpr int kSelThreadsMax = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelWarpsMax = kSelThreadsMax / 32;
constexpr int kSelCluster = 8;              // at most this many CTAs cooperate on one stream
constexpr int kSelCapCta = 45056;           // candidates one CTA holds (176 KiB of keys)
constexpr int kSelCapCluster = kSelCluster * kSelCapCta;
constexpr int kSelBins = 1024;
constexpr int kSelList = 1024;              // most candidates in the bin of the k-th largest one that are ranked directly
constexpr size_t kSelSmemMax = 227 * 1024 - 2048;            // dynamic shared memory a CTA may ask for (static part left out)
constexpr size_t kSelFixedBytes = (size_t)(2 * kSelBins + (kSelCluster + 1) * kSelList) * 4;
static_assert((size_t)kSelCapCta * 4 + kSelFixedBytes <= kSelSmemMax, "a CTA's share does not fit");

// A share beyond this is sorted into bins only near where a sample has the k-th largest candidate.  That takes 0.5 us for ranking the sample and
// wins from 7500 candidates a CTA on; where a far outlier in the sample makes the plain range sweep twice, no sooner than here is
// that slower than three digits of the key were.
constexpr int kSelLong = 11264;
// Candidates a CTA: most before the cluster doubles, and most for a block of 256 threads.  Doubling from 2048 / 4096 / 8192 on: 4096 candidates 8.5 / 8.4 /
// 8.4 us, 6000 8.5 / 8.5 / 9.1, 7800 8.6 / 9.2 / 10.2, 10 000 8.6 / 8.5 / 9.7, 16 000 9.2 / 9.4 / 11.3, 30 000 10.6 / 10.6 / 11.9; up to 4096 one CTA also lets a
// small step select and copy in one launch.  From 6500 to 8192 four CTAs would be the better choice by 0.7 us.  In 256 threads and in
// 1024: 444 candidates 4.3 and 8.5 us, 2000 6.9 and 5.8; blocks of 512 were not tried.
constexpr int64_t kSelShare = 4096, kSelShort = 1024;

// Clusters of eight, one block an SM, that the GPU holds at once: 15 streams of 21 840 candidates 10.4 us, 16 18.8 (in clusters of four 11.3); 32
// streams 28.1, in clusters of four 11.6; 31 of 500 candidates beside one of 20 000 23.1 and 10.7; 16 of 45 000 24.1 and 16.4.
constexpr int kSelRoom8 = 15 * 8;

// Where other work covers the selection but leaves its SMs out (a rolling cache's append copies), its CTAs are kept few: a cache of
// 18 720 tokens, 30 layers of 12 heads, eight CTAs 1109 us, one 1098; 28 080 tokens 1660, two 1631; 18 720 of 2 heads 210 and 206.
constexpr int64_t kSelShareCovered = 24576;

struct SelLaunch {
    bool any_cluster = false, any_stream = false;
    int nc = 1;
    int64_t per_cta = 0;
    int threads() const { return per_cta <= kSelShort ? kSelThreads : kSelThreadsMax; }
};
inline SelLaunch plan_select(const StreamTable& st, bool covered = false) {
    SelLaunch pl;
    int64_t m_max = 0;
    for (int s = 0; s < st.n_streams; ++s) {
        const int64_t T = st.cu_T[s + 1] - st.cu_T[s], B = st.cu_B[s + 1] - st.cu_B[s];
        if (B == 0) continue;
        const int64_t M = B >= T ? 0 : T - st.n_sink[s] - st.n_recent[s];
        if (M > kSelCapCluster) { pl.any_stream = true; continue; }
        pl.any_cluster = true;
        if (M > m_max) m_max = M;
    }
    // CTAs per stream.  A histogram of 1024 candidates costs a CTA some 400 clocks (13 an add and warp, whether or not its
    // lanes collide), the barriers across CTAs and the trips through distributed shared memory two to three thousand.
    // They are doubled while all streams' clusters find room on the GPU at once, or one stream's candidates would not fit.
    auto fits = [&](int nc) { return st.n_streams * nc <= (nc < 8 ? 128 : kSelRoom8); };
    while (pl.nc < kSelCluster && m_max > pl.nc * (!fits(2 * pl.nc) ? (int64_t)kSelCapCta : covered ? kSelShareCovered : kSelShare)) pl.nc *= 2;
    pl.per_cta = ((m_max + pl.nc - 1) / pl.nc + 31) / 32 * 32;
    return pl;
}

// Selection and row copies in one launch: CTAs [first[s], first[s + 1]) select stream s side by side and share its rows.
constexpr int kSelCopyBatch = 4;            // 16-byte pieces of K and of V a thread has in flight
struct CopyShares {
    int32_t equal;                          // that many CTAs each, where it is the same for all; else 0
    uint16_t first[PAFU_MAX_STREAMS + 1];
};
struct SelCopyLaunch {
    bool small = false;
    int threads = 0, per_cta = 0;
    CopyShares shares;
};
// A step is small when one CTA selects each stream and the rows, K and V in and out, are few.  One launch saves the second kernel's
// start; two copy the always-kept rows while the selection runs, with more loads in flight.  Two / one, us a step: one stream kept whole (12 x
// 128) 44 MB 41.7 / 41.7, 52 MB 42.7 / 43.2, 68 MB 46 / 48.6; eight kept whole 46.6 / 46.5, 48.7 / 49.9, 52 / 54.5; mostly sink 45.5 / 45.4, 45.9 / 47.5,
// 49 / 53; all by salience (40 x 128) 71.2 / 69.0, 75.1 / 71.1, 76.9 / 74.9; four streams of the same 48.8 / 48.1, 51.6 / 49.9, 60.4 / 59.2.
// A stream gets as many CTAs as its rows keep busy with one batch each; where that is more than the GPU holds at once, all streams'
// shares grow alike, so that a long stream beside short ones has the GPU nearly to itself (30 000 rows of 512 bytes beside 31 short streams:
// selection and copies 17 us, in two launches 40, with as many CTAs for every stream 255).
// Two launches do worse with narrow rows (2 x 128, mostly sink, 52 MB 49.3 / 47.6, 60 MB 50.1 / 49.3, 68 MB 51.5 / 52.8) and behind more than
// eight selecting CTAs, where the rows are claimed one by one (16 streams, one kept whole, 61 MB 70.7 / 64.9).
constexpr int64_t kSelCopyBytes = (int64_t)64 << 20, kSelCopyAlways = (int64_t)44 << 20;      // of all rows; of always-kept ones
constexpr int kStaticSelect = 8;            // selecting CTAs up to which the row gather hands out fixed shares
inline SelCopyLaunch plan_select_copy(const StreamTable& st, int64_t chunks, int sms) {
    SelCopyLaunch cp;
    const SelLaunch pl = plan_select(st);
    const int n = st.n_streams;
    int64_t top = 0;
    for (int s = 0; s < n; ++s) top += st.cu_B[s + 1] - st.cu_B[s] < st.cu_T[s + 1] - st.cu_T[s] ? st.k[s] : 0;
    const int64_t total = st.cu_B[n] * chunks;
    const int64_t always = n <= kStaticSelect && chunks >= 64 ? kSelCopyAlways : kSelCopyBytes;
    cp.small = !pl.any_stream && pl.any_cluster && pl.nc == 1 && total * 64 <= kSelCopyBytes && (total - top * chunks) * 64 <= always;
    if (!cp.small) return cp;
    cp.per_cta = (int)pl.per_cta;
    cp.threads = pl.threads();
    int64_t batch = (int64_t)cp.threads * kSelCopyBatch;
    const int64_t most = sms > n ? sms : n;
    int64_t longest = 0;
    for (int s = 0; s < n; ++s) longest = st.cu_B[s + 1] - st.cu_B[s] > longest ? st.cu_B[s + 1] - st.cu_B[s] : longest;
    // with room to spare every stream gets what the longest one wants (three of 300 to 517 rows of 512 bytes 29.2 us a step, by rows 29.5)
    const int64_t equal = (longest * chunks + batch - 1) / batch;
    cp.shares.equal = 0;
    if (n * equal <= most) {
        cp.shares.equal = (int32_t)equal;
        for (int s = 0; s <= PAFU_MAX_STREAMS; ++s) cp.shares.first[s] = (uint16_t)((s < n ? s : n) * equal);
        return cp;
    }
    if (batch < (total + most - 1) / most) batch = (total + most - 1) / most;
    for (;; batch += batch / 64) {                           // ends: with the longest stream's rows in one batch there are n CTAs
        int64_t ctas = 0;
        for (int s = 0; s < n; ++s) {
            cp.shares.first[s] = (uint16_t)ctas;
            ctas += ((st.cu_B[s + 1] - st.cu_B[s]) * chunks + batch - 1) / batch;
        }
        for (int s = n; s <= PAFU_MAX_STREAMS; ++s) cp.shares.first[s] = (uint16_t)ctas;
        if (ctas <= most) return cp;
    }
}

}  // namespace pafu
