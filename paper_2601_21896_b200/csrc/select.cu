// Retained-token selection (Sec. 3.4 inference paragraph; Algorithm 2 "Top-k"; frame sink
// Sec. 4.1): kept = [0, n_sink) U top-k salient of the middle U [T - n_recent, T), written as
// ascending token indices, ties to the lower index.
//
// The step moves a few hundred KB, so it is latency-bound: what counts is the chain of barriers, the trips through
// distributed shared memory, and instructions that every warp executes (a scan by 32 warps costs four times the issue slots of
// one by eight, so short shares run in blocks of 256 threads and eight warps do what is done once).  One CTA, or a
// cluster of two, four or eight (the host picks by the stream length), works on one stream; CTA r holds the r-th part of the
// candidates in its shared memory.  Back to back, 444 / 4000 / 7800 / 21 840 / 87 360 / 200 000 / 360 000 candidates:
// 4.3 / 8.2 / 8.8 / 9.8 / 17.1 / 24.9 / 37.1 us; with three passes over digits of the key (11 + 11 + 10 bits, a tenth of the candidates left after
// the first), blocks of 1024 and one CTA up to 24 576 candidates 8.4 / 10.4 / 12.0 / 18.5 / 25.0 / 31.5 / 40.0.
//   1. fp32 scores map to order-preserving 32-bit keys (-0 folded onto +0, NaN lowest).
//   2. One histogram of 1024 equal steps between the smallest and the largest of 256 sampled scores (the same sample in
//      every CTA, so nothing is exchanged for it; values outside fall into the end bins).  One cluster barrier later
//      every CTA adds up all histograms through distributed shared memory and finds by itself the bin that holds the k-th
//      largest candidate.  Every CTA sends its few candidates of that bin to all others; one more barrier, and each ranks
//      them against one another by itself.
//      Long shares (more than kSelLong candidates a CTA): ranking m candidates costs m^2, and a bin of the whole range holds hundreds; the
//      adds into the histogram alone take 10 us at 45 000.  So the sample is ranked, and the steps lie between its places three standard
//      deviations around the k-th largest candidate's: most candidates then fall into the end bins, which are counted in
//      registers, the bins hold dozens, and an outlier in the sample does no harm (360 000 candidates with steps between the extremes
//      61 us, with outliers 63; so 37 and 38).
//   3. A bin that holds too many (ties, a far outlier in the sample) is narrowed down: the smallest and the largest of
//      its candidates are exchanged, and if they differ another histogram divides what lies between them, first in equal
//      steps of the score, then of the key (which ends: 2^32 keys, a factor of 1024 each time).
//   4. Ordered emission: every warp owns a contiguous stretch of the CTA's candidates.  What it keeps of them is known from the sweep that
//      found the bin's candidates and from who found which; with the counts of the warps and CTAs before it, it writes them in order:
//      the result is ascending and ties resolve to the lowest indices.
// Streams with more candidates than eight CTAs hold (360 448) use one CTA that re-reads L2 in every pass.
// A kernel launched behind these as a programmatic dependent may start at once (the trigger at
// their top): inside a layer step that is the row gather, which copies the rows that are kept
// whatever the scores say while the selection runs, and waits for the indices after that.
#include <cooperative_groups.h>

#include "select_plan.cuh"

namespace pafu {

namespace cg = cooperative_groups;

constexpr int kSelBatch = 8;                // independent loads a thread keeps in flight
constexpr int kSelStreamThreads = 1024;     // the streaming kernel's block
static_assert(kSelBins == 4 * kSelThreads, "four bins a thread");

__device__ __forceinline__ uint32_t score_key(float f) {
    uint32_t u = __float_as_uint(f);
    if ((u & 0x7fffffffu) > 0x7f800000u) return 0u;      // NaN: below -inf
    if (u == 0x80000000u) u = 0u;                        // -0 == +0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Exclusive prefix sum of one int per thread over a block of 1024; also returns the block total.
__device__ __forceinline__ int sel_exclusive_scan(int v, int* warp_sums, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
    }
    __syncthreads();                // protect warp_sums from the previous use
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int w = warp_sums[lane];
        int winc = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int n = __shfl_up_sync(0xffffffffu, winc, o);
            if (lane >= o) winc += n;
        }
        warp_sums[lane] = winc - w;  // exclusive offset of each warp
        if (lane == 31) warp_sums[32] = winc;
    }
    __syncthreads();
    *total = warp_sums[32];
    return warp_sums[warp] + inc - v;
}

// The score a key stands for (a NaN for key 0).
__device__ __forceinline__ float key_score(uint32_t key) { return __uint_as_float((key & 0x80000000u) ? key ^ 0x80000000u : ~key); }

struct SelShared {
    int sums[kSelWarps];
    uint32_t lo[kSelWarpsMax], hi[kSelWarpsMax];
    int bin, k_rem, bin_count;
    uint32_t thr;
    int need_eq, eq_total;
    int list_n;
    int warp_gt[kSelWarpsMax], warp_eq[kSelWarpsMax];   // candidates of each warp above the bin (the threshold) and in it (equal to it)
    uint8_t owner[kSelList];         // whose the CTA's candidates in the bin are
    // from every CTA: its candidates in the bin and above it, and the smallest and largest of those in it
    int in_bin[kSelCluster], above[kSelCluster];
    uint32_t cta_lo[kSelCluster], cta_hi[kSelCluster];
};

__device__ __forceinline__ void sel_barrier(cg::cluster_group& cluster, int nc) {
    if (nc > 1) cluster.sync(); else __syncthreads();
}

// The bin that holds the k_rem-th largest of what the CTAs' histograms `hist` (the same address in every CTA) count, to
// sh.bin, sh.k_rem, sh.bin_count.  The barrier at the top makes every histogram complete and visible.  (Eight warps do it
// whatever the block: a scan by 32 costs four times the issue slots.)
__device__ __forceinline__ void find_bin(cg::cluster_group& cluster, int nc, SelShared& sh, const int* hist, int k_rem) {
    sel_barrier(cluster, nc);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // bins from the top: thread t holds bins 1023 - 4 t .. 1020 - 4 t
    const int b_hi = kSelBins - 1 - 4 * tid;
    int c[4] = {0, 0, 0, 0}, own = 0, inc = 0;
    if (warp < kSelWarps) {
        const int* mine = hist + b_hi - 3;
        for (int r0 = 0; r0 < nc; r0 += 4) {
            int4 v[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) v[r] = r0 + r < nc ? *reinterpret_cast<const int4*>(cluster.map_shared_rank(mine, r0 + r)) : make_int4(0, 0, 0, 0);
#pragma unroll
            for (int r = 0; r < 4; ++r) { c[0] += v[r].w; c[1] += v[r].z; c[2] += v[r].y; c[3] += v[r].x; }
        }
        own = inc = c[0] + c[1] + c[2] + c[3];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int n = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += n;
        }
        if (lane == 31) sh.sums[warp] = inc;
    }
    __syncthreads();
    if (warp < kSelWarps) {
        int above = inc - own;
#pragma unroll
        for (int w = 0; w < kSelWarps - 1; ++w) above += w < warp ? sh.sums[w] : 0;
        if (above < k_rem && k_rem <= above + own) {
            int i = 0;
#pragma unroll
            for (int u = 0; u < 3; ++u)
                if (i == u && above + c[u] < k_rem) { above += c[u]; ++i; }
            sh.bin = b_hi - i; sh.k_rem = k_rem - above; sh.bin_count = i == 0 ? c[0] : i == 1 ? c[1] : i == 2 ? c[2] : c[3];
        }
    }
    __syncthreads();
}

// The selection of stream s by the CTAs of a cluster, or (ALONE) by one CTA for itself: `copies` CTAs then select the same stream
// side by side, number `copy` of them writes its share of the always-kept indices, number 0 the top-k ones, and every one
// leaves the top-k tokens in its shared memory (`top`).
template <bool ALONE>
__device__ __forceinline__ void select_stream(const float* __restrict__ scores, const StreamTable& st, int s, int copy, int copies, int32_t keys_bytes,
                                              int32_t* __restrict__ idx, int trigger_late, unsigned char* sel_smem, SelShared& sh, int* top) {
    if (!ALONE && !trigger_late) grid_dep_launch_dependents();
    cg::cluster_group cluster = cg::this_cluster();
    const int nc = ALONE ? 1 : (int)cluster.num_blocks();    // 1, 2, 4 or 8: the host's choice for this launch
    const int rank = ALONE ? 0 : (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int threads = (int)blockDim.x, warps = threads >> 5;
    uint32_t* keys = reinterpret_cast<uint32_t*>(sel_smem);
    int* hist = reinterpret_cast<int*>(sel_smem + keys_bytes);               // two histograms
    uint32_t* list = reinterpret_cast<uint32_t*>(hist + 2 * kSelBins);       // [kSelCluster][kSelList]: every CTA's candidates in the bin
    uint32_t* all = list + kSelCluster * kSelList;                           // [kSelList]: the same side by side
    if (tid < kSelThreads) *reinterpret_cast<int4*>(hist + 4 * tid) = make_int4(0, 0, 0, 0);
    if (tid == 0) sh.list_n = 0;
    const int T = (int)(st.cu_T[s + 1] - st.cu_T[s]), B = (int)(st.cu_B[s + 1] - st.cu_B[s]);
    // a stream that keeps everything is one long "sink"
    const bool everything = B >= T;
    const int ns = everything ? T : (int)st.n_sink[s], nr = everything ? 0 : (int)st.n_recent[s], k = everything ? 0 : (int)st.k[s];
    const int M = T - ns - nr;
    const float* first = scores + st.cu_T[s] + ns;
    int32_t* out = idx + st.cu_B[s];
    grid_dep_wait();
    if (!ALONE && trigger_late) grid_dep_launch_dependents();
    // cluster-uniform exits (before any cluster barrier)
    if (B == 0) return;
    if (M > nc * kSelCapCta) return;                         // the streaming kernel owns this stream

    // this CTA's candidates: [j_lo, j_lo + n) of the stream's M
    const int per_cta = ((M + nc - 1) / nc + 31) / 32 * 32;
    const int j_lo = rank * per_cta;
    const int n = max(0, min(M - j_lo, per_cta));
    const bool near_k = !ALONE && per_cta > kSelLong;
    if (k > 0) {
        const int step = M / kSelThreads;                    // 0: every candidate is in the sample
        const int js = step > 0 ? tid * step : tid;
        const float sample = js < M && tid < kSelThreads ? __ldg(first + js) : __uint_as_float(0x7fc00000u);
        for (int j0 = tid; j0 < n; j0 += threads * kSelBatch) {
            float v[kSelBatch];
#pragma unroll
            for (int u = 0; u < kSelBatch; ++u) v[u] = j0 + u * threads < n ? __ldg(first + j_lo + j0 + u * threads) : 0.f;
#pragma unroll
            for (int u = 0; u < kSelBatch; ++u)
                if (j0 + u * threads < n) keys[j0 + u * threads] = score_key(v[u]);
        }
        // the finite samples' range
        const uint32_t ks = score_key(sample);
        const bool finite = ks >= 0x00800000u && ks <= 0xff7fffffu;
        const uint32_t lo_w = __reduce_min_sync(0xffffffffu, finite ? ks : 0xffffffffu), hi_w = __reduce_max_sync(0xffffffffu, finite ? ks : 0u);
        if (lane == 0) { sh.lo[warp] = lo_w; sh.hi[warp] = hi_w; }
        if (near_k && tid < kSelThreads && tid % 2 == 0) hist[kSelBins + tid / 2] = (int)ks;
    }
    // always-kept tokens (spread over the cluster, or the CTAs side by side): position p < ns is token p, position ns + k + i is token T - nr + i
    for (int p = (ALONE ? copy : rank) * threads + tid; p < ns + nr; p += (ALONE ? copies : nc) * threads) {
        if (p < ns) out[p] = p; else out[p + k] = T - (ns + nr) + p;
    }
    if (k == 0) return;
    __syncthreads();
    uint32_t klo = 0u, khi = 0xffffffffu;                    // the keys still in question
    float lo = 0.f, scale = 0.f;                             // how they are divided: equal steps of the score,
    int shift = -1;                                          // or of the key (>= 0)
    auto steps = [&](float a, float b) {                     // between finite scores a < b
        lo = a;
        scale = (float)kSelBins / (b - a);
        if (!(scale <= 3.0e38f)) scale = 0.f;                // a range of a few denormals
    };
    {
        const uint32_t a = __reduce_min_sync(0xffffffffu, sh.lo[lane & (kSelWarps - 1)]), b = __reduce_max_sync(0xffffffffu, sh.hi[lane & (kSelWarps - 1)]);
        if (a < b) steps(key_score(a), key_score(b));        // at least two finite values
    }
    if (near_k) {
        // Between the places of every other sample three standard deviations around the k-th largest candidate's, and three times as far
        // out where the sample ends (eight threads rank a sample).
        constexpr int kRanked = kSelThreads / 2;
        static_assert(kRanked * 8 == kSelThreadsMax, "eight threads a sample");
        const float p = (float)k / (float)M * kRanked, d = 3.f * sqrtf(p * (1.f - p / kRanked)) + 1.f;
        const int r_hi = max(0, (int)(p - d)), r_lo = min(kRanked - 1, (int)(p + d) + 1);
        const uint32_t* ranked_keys = reinterpret_cast<const uint32_t*>(hist + kSelBins);
        const uint32_t key = ranked_keys[tid >> 3];
        int gt = 0, ge = 0;
#pragma unroll
        for (int e = 0; e < kRanked / 8; e += 4) {
            const uint4 o = *reinterpret_cast<const uint4*>(ranked_keys + (tid & 7) * (kRanked / 8) + e);
            gt += (o.x > key) + (o.y > key) + (o.z > key) + (o.w > key);
            ge += (o.x >= key) + (o.y >= key) + (o.z >= key) + (o.w >= key);
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) { gt += __shfl_xor_sync(0xffffffffu, gt, o); ge += __shfl_xor_sync(0xffffffffu, ge, o); }
        if (gt <= r_hi && r_hi < ge) sh.hi[kSelWarps] = key;                 // equal keys write the same
        if (gt <= r_lo && r_lo < ge) sh.lo[kSelWarps] = key;
        __syncthreads();
        const uint32_t l = sh.lo[kSelWarps], h = sh.hi[kSelWarps];
        if (l >= 0x00800000u && l < h && h <= 0xff7fffffu) {
            const float a = key_score(l), b = key_score(h), far = 3.f * (b - a);
            const float x = p < d ? b + far : b, y = p + d > kRanked ? a - far : a;
            if (x - y <= 3.0e38f) steps(y, x); else steps(a, b);
        }
    }
    // Monotone in the key: rounding is, and so are the clamps; infinities end up in the end bins, NaN (lowest) in bin 0, and with
    // scale = 0 everything in bin 0.
    auto bin_of = [&](uint32_t key) {
        int b = shift >= 0 ? (int)((key - klo) >> shift)
                           : min(max(__float2int_rz(__fmul_rn(__fsub_rn(key_score(key), lo), scale)), 0), kSelBins - 1);
        if (key < klo) b = -1;
        if (key > khi) b = kSelBins;
        return b;
    };
    // each warp's stretch of the candidates: whole groups of 32
    const int per_warp = ((n + 31) / 32 + warps - 1) / warps * 32;
    const int w0 = min(n, warp * per_warp), w1 = min(n, w0 + per_warp);
    const unsigned lt = (1u << lane) - 1u;
    uint32_t thr = 0u;
    int need_eq = k, eq_total = 0;
    int gt_before = 0, eq_before = 0;                        // in the CTAs before this one
    bool ranked = true;
#pragma unroll 1
    for (int level = 0;; ++level) {                          // cluster-uniform
        int* h = hist + (level & 1) * kSelBins;              // (every CTA is past its reads of the level before last)
        if (level > 0) {
            if (tid < kSelThreads) *reinterpret_cast<int4*>(h + 4 * tid) = make_int4(0, 0, 0, 0);
            __syncthreads();
        }
        if (near_k && level == 0) {                          // most candidates fall into the end bins: they are counted in registers
            int low = 0, high = 0;
#pragma unroll 4
            for (int j = tid; j < n; j += threads) {
                const int b = bin_of(keys[j]);
                low += b == 0;
                high += b == kSelBins - 1;
                if (b > 0 && b < kSelBins - 1) atomicAdd(h + b, 1);
            }
            low = __reduce_add_sync(0xffffffffu, low);
            high = __reduce_add_sync(0xffffffffu, high);
            if (lane == 0) { atomicAdd(h, low); atomicAdd(h + kSelBins - 1, high); }
        } else {
#pragma unroll 4
            for (int j = tid; j < n; j += threads) {
                const int b = bin_of(keys[j]);
                if ((unsigned)b < (unsigned)kSelBins) atomicAdd(h + b, 1);
            }
        }
        find_bin(cluster, nc, sh, h, need_eq);
        need_eq = sh.k_rem; eq_total = sh.bin_count;
        // ranking m keys costs a warp m / 32 turns of m comparisons, narrowing down two more sweeps over the CTA's share
        if (eq_total <= max(256, min(kSelList, per_cta / 32))) break;
        // ---- too many: what lies between the smallest and the largest of them
        const int bin = sh.bin;
        int above = 0, in = 0;
        uint32_t mn = 0xffffffffu, mx = 0u;
        for (int j0 = w0; j0 < w1; j0 += 32) {
            const uint32_t key = j0 + lane < w1 ? keys[j0 + lane] : 0u;
            const int b = j0 + lane < w1 ? bin_of(key) : -1;
            above += __popc(__ballot_sync(0xffffffffu, b > bin));
            in += __popc(__ballot_sync(0xffffffffu, b == bin));
            if (b == bin) { mn = min(mn, key); mx = max(mx, key); }
        }
        mn = __reduce_min_sync(0xffffffffu, mn); mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) { sh.lo[warp] = mn; sh.hi[warp] = mx; sh.warp_gt[warp] = above; sh.warp_eq[warp] = in; }
        __syncthreads();
        if (warp == 0) {
            const int a = __reduce_add_sync(0xffffffffu, lane < warps ? sh.warp_gt[lane] : 0), i = __reduce_add_sync(0xffffffffu, lane < warps ? sh.warp_eq[lane] : 0);
            mn = __reduce_min_sync(0xffffffffu, lane < warps ? sh.lo[lane] : 0xffffffffu); mx = __reduce_max_sync(0xffffffffu, lane < warps ? sh.hi[lane] : 0u);
            if (lane < nc) {
                SelShared* remote = cluster.map_shared_rank(&sh, lane);
                remote->in_bin[rank] = i; remote->above[rank] = a; remote->cta_lo[rank] = mn; remote->cta_hi[rank] = mx;
            }
        }
        sel_barrier(cluster, nc);
        mn = __reduce_min_sync(0xffffffffu, lane < nc ? sh.cta_lo[lane] : 0xffffffffu); mx = __reduce_max_sync(0xffffffffu, lane < nc ? sh.cta_hi[lane] : 0u);
        if (mn == mx) {                                      // all equal
            thr = mn;
            gt_before = __reduce_add_sync(0xffffffffu, lane < rank ? sh.above[lane] : 0);
            eq_before = __reduce_add_sync(0xffffffffu, lane < rank ? sh.in_bin[lane] : 0);
            ranked = false;
            break;
        }
        klo = mn; khi = mx;
        const bool finite = klo >= 0x00800000u && khi <= 0xff7fffffu;
        if (level == 0 && finite) steps(key_score(klo), key_score(khi));
        else shift = max(0, 22 - __clz(khi - klo));
    }
    if (ranked) {
        // ---- the bin's candidates, to segment `rank` of every CTA's list (any order: only their values matter now)
        const int bin = sh.bin, k_rem = need_eq;
        int above = 0;
#pragma unroll 4
        for (int j0 = w0; j0 < w1; j0 += 32) {
            const uint32_t key = j0 + lane < w1 ? keys[j0 + lane] : 0u;
            const int b = j0 + lane < w1 ? bin_of(key) : -1;
            above += __popc(__ballot_sync(0xffffffffu, b > bin));
            if (b == bin) {
                const int at = atomicAdd(&sh.list_n, 1);
                sh.owner[at] = (uint8_t)warp;
                for (int r = 0; r < nc; ++r) cluster.map_shared_rank(list, r)[rank * kSelList + at] = key;
            }
        }
        if (lane == 0) { sh.warp_gt[warp] = above; sh.warp_eq[warp] = 0; }
        __syncthreads();
        if (warp == 0) {
            const int a = __reduce_add_sync(0xffffffffu, lane < warps ? sh.warp_gt[lane] : 0);
            if (lane < nc) {
                SelShared* remote = cluster.map_shared_rank(&sh, lane);
                remote->in_bin[rank] = sh.list_n; remote->above[rank] = a;
            }
        }
        sel_barrier(cluster, nc);
        // ---- side by side, in the CTAs' order
        const int in_bin = lane < nc ? sh.in_bin[lane] : 0;
        const int n_all = __reduce_add_sync(0xffffffffu, in_bin), n_before = __reduce_add_sync(0xffffffffu, lane < rank ? in_bin : 0);
        gt_before = __reduce_add_sync(0xffffffffu, lane < rank ? sh.above[lane] : 0);
        uint32_t* flat = nc > 1 ? all : list;
        if (nc > 1 && warp < nc) {
            const int at = __reduce_add_sync(0xffffffffu, lane < warp ? in_bin : 0), m = sh.in_bin[warp];
            for (int i = lane; i < m; i += 32) all[at + i] = list[warp * kSelList + i];
        }
        if (nc > 1) __syncthreads();
        // ---- the key of the k_rem-th largest of them: every thread ranks its own
        for (int i = tid; i < n_all; i += threads) {
            const uint32_t key = flat[i];
            int gt = 0, eq = 0;
            int e = 0;
#pragma unroll 2
            for (; e + 4 <= n_all; e += 4) {
                const uint4 o = *reinterpret_cast<const uint4*>(flat + e);
                gt += (o.x > key) + (o.y > key) + (o.z > key) + (o.w > key);
                eq += (o.x == key) + (o.y == key) + (o.z == key) + (o.w == key);
            }
            for (; e < n_all; ++e) { gt += flat[e] > key; eq += flat[e] == key; }
            if (gt < k_rem && k_rem <= gt + eq) { sh.thr = key; sh.need_eq = k_rem - gt; sh.eq_total = eq; }   // equal keys write the same
        }
        __syncthreads();
        thr = sh.thr; need_eq = sh.need_eq; eq_total = sh.eq_total;
        // what the CTAs before this one keep of them (every warp for itself)
        for (int i0 = 0; i0 < n_before; i0 += 32) {
            const bool in = i0 + lane < n_before;
            const uint32_t key = in ? flat[i0 + lane] : 0u;
            gt_before += __popc(__ballot_sync(0xffffffffu, in && key > thr));
            eq_before += __popc(__ballot_sync(0xffffffffu, in && key == thr));
        }
        // and what the warps of this one do
        for (int i = tid; i < sh.list_n; i += threads) {
            const uint32_t key = list[rank * kSelList + i];
            if (key >= thr) atomicAdd(key > thr ? &sh.warp_gt[sh.owner[i]] : &sh.warp_eq[sh.owner[i]], 1);
        }
        __syncthreads();
    }

    // ---- ordered emission
    const bool ties = need_eq != eq_total;                   // cluster-uniform: some equal candidates stay out
    gt_before += __reduce_add_sync(0xffffffffu, lane < warp ? sh.warp_gt[lane] : 0);
    eq_before += __reduce_add_sync(0xffffffffu, lane < warp ? sh.warp_eq[lane] : 0);
    int pos = ns + gt_before + (ties ? min(eq_before, need_eq) : eq_before);
#pragma unroll 4
    for (int j0 = w0; j0 < w1; j0 += 32) {
        const uint32_t key = j0 + lane < w1 ? keys[j0 + lane] : 0u;
        const bool is_eq = j0 + lane < w1 && key == thr;
        bool keep = j0 + lane < w1 && key >= thr;
        if (ties) {
            const unsigned be = __ballot_sync(0xffffffffu, is_eq);
            keep = keep && (!is_eq || eq_before + __popc(be & lt) < need_eq);
            eq_before += __popc(be);
        }
        const unsigned bk = __ballot_sync(0xffffffffu, keep);
        if (keep) {
            if (ALONE) top[pos - ns + __popc(bk & lt)] = ns + j0 + lane;
            if (!ALONE || copy == 0) out[pos + __popc(bk & lt)] = ns + j_lo + j0 + lane;
        }
        pos += __popc(bk);
    }
}

__global__ void __launch_bounds__(kSelThreadsMax, 1)
select_cluster_kernel(const float* __restrict__ scores, const __grid_constant__ StreamTable st, int32_t keys_bytes,
                      int32_t* __restrict__ idx, int trigger_late) {
    extern __shared__ __align__(16) unsigned char sel_smem[];
    __shared__ SelShared sh;
    select_stream<false>(scores, st, blockIdx.x / cg::this_cluster().num_blocks(), 0, 1, keys_bytes, idx, trigger_late, sel_smem, sh, nullptr);
}

// Selection and row gather of a small layer step in one launch: a stream's CTAs all make its whole selection (a
// few microseconds, whoever does it) and then copy a share of its rows each, without a word between them.  What it
// saves is the second kernel's start: a step of 2 heads x 64 over 512 tokens 19.0 -> 17.2 us, 4 x 64 over 600 25.5 -> 23.8, 5 x 128 over 1800 +
// 2500 37.5 -> 37.0, 12 x 128 over 3000 (18 MB in and out) 54.1 -> 53.1.  Larger steps keep two launches: their always-kept rows are
// copied while the selection runs.
__global__ void __launch_bounds__(kSelThreadsMax, 1)
select_copy_kernel(const float* __restrict__ scores, const __grid_constant__ StreamTable st, int32_t keys_bytes,
                   int32_t* __restrict__ idx, const __grid_constant__ CopyShares shares, const uint4* __restrict__ K, const uint4* __restrict__ V,
                   int chunks_per_row, uint4* __restrict__ Kc, uint4* __restrict__ Vc, float* __restrict__ SLc) {
    extern __shared__ __align__(16) unsigned char sel_smem[];
    __shared__ SelShared sh;
    const int b = (int)blockIdx.x, threads = (int)blockDim.x;
    int s, copy, copies = shares.equal;
    if (copies > 0) {
        s = b / copies;
        copy = b - s * copies;
    } else {
        s = 0;                                               // the last stream that begins at or before b
#pragma unroll
        for (int d = PAFU_MAX_STREAMS / 2; d > 0; d /= 2)
            if (s + d < st.n_streams && shares.first[s + d] <= b) s += d;
        copy = b - shares.first[s];
        copies = shares.first[s + 1] - shares.first[s];
    }
    int* top = reinterpret_cast<int*>(sel_smem + keys_bytes + kSelFixedBytes);
    select_stream<true>(scores, st, s, copy, copies, keys_bytes, idx, 0, sel_smem, sh, top);
    __syncthreads();
    const int T = (int)(st.cu_T[s + 1] - st.cu_T[s]), B = (int)(st.cu_B[s + 1] - st.cu_B[s]);
    const bool everything = B >= T;
    const int ns = everything ? T : (int)st.n_sink[s], k = everything ? 0 : (int)st.k[s];
    auto token = [&](int r) { return r < ns ? r : r < ns + k ? top[r - ns] : T - B + r; };
    const uint4* Ks = K + st.cu_T[s] * chunks_per_row;
    const uint4* Vs = V + st.cu_T[s] * chunks_per_row;
    uint4* Kd = Kc + st.cu_B[s] * chunks_per_row;
    uint4* Vd = Vc + st.cu_B[s] * chunks_per_row;
    const int units = B * chunks_per_row, step = copies * threads;
    for (int u0 = copy * threads + (int)threadIdx.x; u0 < units; u0 += step * kSelCopyBatch) {
        uint4 kb[kSelCopyBatch], vb[kSelCopyBatch];
#pragma unroll
        for (int i = 0; i < kSelCopyBatch; ++i) {
            const int u = u0 + i * step;
            if (u < units) {
                const int row = u / chunks_per_row;
                const int64_t src = (int64_t)token(row) * chunks_per_row + (u - row * chunks_per_row);
                kb[i] = __ldg(Ks + src); vb[i] = __ldg(Vs + src);
            }
        }
#pragma unroll
        for (int i = 0; i < kSelCopyBatch; ++i) {
            const int u = u0 + i * step;
            if (u < units) { Kd[u] = kb[i]; Vd[u] = vb[i]; }
        }
    }
    if (SLc != nullptr)
        for (int r = copy * threads + (int)threadIdx.x; r < B; r += step) SLc[st.cu_B[s] + r] = __ldg(scores + st.cu_T[s] + token(r));
}

// Streams with more candidates than a cluster's shared memory holds: keys are re-read from L2 in every pass
// (4 passes of 8 bits), and each thread emits a contiguous token range.
__global__ void __launch_bounds__(kSelStreamThreads)
select_stream_kernel(const float* __restrict__ scores, StreamTable st, int32_t* __restrict__ idx, int trigger_late) {
    if (!trigger_late) grid_dep_launch_dependents();
    grid_dep_wait();
    if (trigger_late) grid_dep_launch_dependents();
    {
        const int64_t T = st.cu_T[blockIdx.x + 1] - st.cu_T[blockIdx.x], B = st.cu_B[blockIdx.x + 1] - st.cu_B[blockIdx.x];
        if (B >= T || T - st.n_sink[blockIdx.x] - st.n_recent[blockIdx.x] <= kSelCapCluster) return;   // the other kernel owns this stream
    }
    __shared__ int hist[256];
    __shared__ int warp_sums[33];
    __shared__ uint32_t sh_prefix;
    __shared__ int sh_krem;

    const int s = blockIdx.x;
    const int tid = threadIdx.x;
    const int64_t T64 = st.cu_T[s + 1] - st.cu_T[s];
    const float* sc = scores + st.cu_T[s];
    int32_t* out = idx + st.cu_B[s];
    const int T = (int)T64;
    const int ns = (int)st.n_sink[s], nr = (int)st.n_recent[s];
    const int k = (int)st.k[s];
    const int c0 = ns, c1 = T - nr;                     // candidates [c0, c1)

    // ---- radix select: key of the k-th largest candidate
    uint32_t thr = 0xffffffffu;
    int need_eq = 0;
    if (k > 0) {
        uint32_t prefix = 0u, mask = 0u;
        int k_rem = k;
        for (int pass = 0; pass < 4; ++pass) {
            const int shift = 24 - 8 * pass;
            if (tid < 256) hist[tid] = 0;
            __syncthreads();
            for (int t0 = c0 + tid; t0 < c1; t0 += kSelStreamThreads * kSelBatch) {
                float v[kSelBatch];                      // the batch's loads are in flight together
#pragma unroll
                for (int u = 0; u < kSelBatch; ++u) v[u] = t0 + u * kSelStreamThreads < c1 ? __ldg(sc + t0 + u * kSelStreamThreads) : 0.f;
#pragma unroll
                for (int u = 0; u < kSelBatch; ++u) {
                    const uint32_t key = score_key(v[u]);
                    if (t0 + u * kSelStreamThreads < c1 && (key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1);
                }
            }
            __syncthreads();
            if (tid < 32) {
                int cnt[8];
                int mine = 0;
#pragma unroll
                for (int b = 0; b < 8; ++b) { cnt[b] = hist[tid * 8 + b]; mine += cnt[b]; }
                // number of matching candidates in bins above this lane's bins
                int suf = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    int n = __shfl_down_sync(0xffffffffu, suf, o);
                    if (tid + o < 32) suf += n;
                }
                int above = suf - mine;
#pragma unroll
                for (int b = 7; b >= 0; --b) {
                    if (above < k_rem && k_rem <= above + cnt[b]) {
                        sh_prefix = prefix | ((uint32_t)(tid * 8 + b) << shift);
                        sh_krem = k_rem - above;
                    }
                    above += cnt[b];
                }
            }
            __syncthreads();
            prefix = sh_prefix;
            k_rem = sh_krem;
            mask |= 0xffu << shift;
        }
        thr = prefix;
        need_eq = k_rem;
    }

    // ---- ordered emission
    const int per = (T + kSelStreamThreads - 1) / kSelStreamThreads;
    const int t0 = min(T, tid * per), t1 = min(T, t0 + per);
    int eqc = 0;
    for (int t = max(t0, c0); t < min(t1, c1); ++t) eqc += (score_key(sc[t]) == thr);
    int total;
    const int eq_before = sel_exclusive_scan(eqc, warp_sums, &total);
    int kc = 0, e = eq_before;
    for (int t = t0; t < t1; ++t) {
        bool keep = (t < c0) || (t >= c1);
        if (!keep) {
            const uint32_t key = score_key(sc[t]);
            keep = key > thr;
            if (key == thr) { keep = e < need_eq; ++e; }
        }
        kc += keep;
    }
    int pos = sel_exclusive_scan(kc, warp_sums, &total);
    e = eq_before;
    for (int t = t0; t < t1; ++t) {
        bool keep = (t < c0) || (t >= c1);
        if (!keep) {
            const uint32_t key = score_key(sc[t]);
            keep = key > thr;
            if (key == thr) { keep = e < need_eq; ++e; }
        }
        if (keep) out[pos++] = t;
    }
}

int select_cta_count(const StreamTable& st, bool covered) {
    const SelLaunch pl = plan_select(st, covered);
    return (pl.any_cluster ? st.n_streams * pl.nc : 0) + (pl.any_stream ? st.n_streams : 0);
}

pafu_status launch_select_compact(const uint16_t* K, const uint16_t* V, const float* scores, const StreamTable& st, int32_t d_model, int32_t* idx,
                                  uint16_t* Kc, uint16_t* Vc, float* SLc, cudaStream_t stream, bool* done) {
    const int chunks = d_model / 8;
    const SelCopyLaunch cp = plan_select_copy(st, chunks, device_sm_count());
    *done = cp.small;
    if (!*done) return PAFU_OK;
    static bool attr[kMaxDevices] = {};
    if (!once_per_device(attr, [] {
            return cudaFuncSetAttribute(select_copy_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSelSmemMax) == cudaSuccess;
        }))
        return PAFU_ERR_CUDA;
    const int32_t keys_bytes = cp.per_cta * 4;
    return cuda_ok(launch_dependent(select_copy_kernel, dim3((unsigned)cp.shares.first[st.n_streams]), dim3(cp.threads),
                                    (size_t)keys_bytes * 2 + kSelFixedBytes, stream, 1, scores, st, keys_bytes, idx, cp.shares,
                                    reinterpret_cast<const uint4*>(K), reinterpret_cast<const uint4*>(V), chunks,
                                    reinterpret_cast<uint4*>(Kc), reinterpret_cast<uint4*>(Vc), SLc));
}

pafu_status launch_select(const float* scores, const StreamTable& st, int32_t* idx, cudaStream_t stream, int trigger_late, bool covered) {
    if (st.n_streams == 0 || st.cu_B[st.n_streams] == 0) return PAFU_OK;
    const SelLaunch pl = plan_select(st, covered);
    if (pl.any_cluster) {
        static bool done[kMaxDevices] = {};
        if (!once_per_device(done, [] {
                return cudaFuncSetAttribute(select_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSelSmemMax) == cudaSuccess;
            }))
            return PAFU_ERR_CUDA;
        const int32_t keys_bytes = (int32_t)(pl.per_cta * 4);
        const size_t smem = (size_t)keys_bytes + kSelFixedBytes;
        if (launch_dependent(select_cluster_kernel, dim3((unsigned)(st.n_streams * pl.nc)),
                             dim3(pl.threads()), smem, stream,
                             (unsigned)pl.nc, scores, st, keys_bytes, idx, trigger_late) != cudaSuccess)
            return PAFU_ERR_CUDA;
    }
    if (pl.any_stream &&
        launch_dependent(select_stream_kernel, dim3((unsigned)st.n_streams), dim3(kSelStreamThreads), 0, stream, 1, scores, st,
                         idx, trigger_late) != cudaSuccess)
        return PAFU_ERR_CUDA;
    return PAFU_OK;
}

}  // namespace pafu
