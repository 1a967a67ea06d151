// KV <- Select(KV; ids), SL <- Select(SL; ids) (Algorithm 2): row gather of the kept tokens.
//
// HBM-bound copy.  One warp moves one kept token: its K row and its V row (d_model bf16 each)
// in 16-byte pieces, all loads of a batch issued before the first store so that each warp
// keeps up to 12 x 512 B in flight.  Rows are contiguous, so every access is fully coalesced;
// the only indirection is one int32 index per row.
#include "select_plan.cuh"

namespace pafu {

constexpr int kCompactWarpsPerBlock = 8;
constexpr int kCompactUnroll = 6;   // 6 x 32 lanes x 16 B = one 3072-byte row (d_model 1536)

__device__ __forceinline__ uint4 ld_nc_v4(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// One warp copies row src_row of K and V (and the salience entry) to row dst_row of Kc and Vc.
__device__ __forceinline__ void copy_kv_row(const uint4* __restrict__ K, const uint4* __restrict__ V,
                                            const float* __restrict__ SL, int64_t src_row, int64_t dst_row,
                                            int chunks_per_row, uint4* __restrict__ Kc, uint4* __restrict__ Vc,
                                            float* __restrict__ SLc, int lane) {
    const uint4* ks = K + src_row * chunks_per_row;
    const uint4* vs = V + src_row * chunks_per_row;
    uint4* kd = Kc + dst_row * chunks_per_row;
    uint4* vd = Vc + dst_row * chunks_per_row;
    for (int c0 = 0; c0 < chunks_per_row; c0 += 32 * kCompactUnroll) {
        uint4 kb[kCompactUnroll], vb[kCompactUnroll];
#pragma unroll
        for (int u = 0; u < kCompactUnroll; ++u) {
            const int c = c0 + u * 32 + lane;
            if (c < chunks_per_row) { kb[u] = ld_nc_v4(ks + c); vb[u] = ld_nc_v4(vs + c); }
        }
#pragma unroll
        for (int u = 0; u < kCompactUnroll; ++u) {
            const int c = c0 + u * 32 + lane;
            if (c < chunks_per_row) { kd[c] = kb[u]; vd[c] = vb[u]; }
        }
    }
    if (SLc != nullptr && lane == 0) SLc[dst_row] = __ldg(SL + src_row);
}

// The same for `count` rows that are narrower than what a warp keeps in flight, laid end to end: lane l < count knows row l's
// source and destination, and unit u = i * 32 + lane of the stretch, which belongs to row u / chunks_per_row (bits 5 i .. 5 i + 4 of
// `row_of`), takes them from that lane.  (K, V, Kc and Vc hold less than 2^32 units each: the host sees to it.)
__device__ __forceinline__ uint32_t rows_of_units(int chunks_per_row, int lane) {
    uint32_t r = 0;
#pragma unroll
    for (int i = 0; i < kCompactUnroll; ++i) r |= (uint32_t)min((i * 32 + lane) / chunks_per_row, 31) << (5 * i);
    return r;
}
__device__ __forceinline__ void copy_kv_rows(const uint4* __restrict__ K, const uint4* __restrict__ V,
                                             const float* __restrict__ SL, int64_t src_row, int64_t dst_row, int count,
                                             int chunks_per_row, uint4* __restrict__ Kc, uint4* __restrict__ Vc,
                                             float* __restrict__ SLc, int lane, uint32_t row_of) {
    static_assert(kCompactUnroll <= 6, "row_of holds six rows");
    const int units = count * chunks_per_row;
    const uint32_t src = (uint32_t)(src_row - lane) * chunks_per_row + lane, dst = (uint32_t)(dst_row - lane) * chunks_per_row + lane;
    uint4 kb[kCompactUnroll], vb[kCompactUnroll];
#pragma unroll
    for (int i = 0; i < kCompactUnroll; ++i) {
        const int from = (row_of >> (5 * i)) & 31;
        const uint32_t s = __shfl_sync(0xffffffffu, src, from) - from + lane + i * 32;
        if (i * 32 + lane < units) { kb[i] = ld_nc_v4(K + s); vb[i] = ld_nc_v4(V + s); }
    }
#pragma unroll
    for (int i = 0; i < kCompactUnroll; ++i) {
        const int from = (row_of >> (5 * i)) & 31;
        const uint32_t d = __shfl_sync(0xffffffffu, dst, from) - from + lane + i * 32;
        if (i * 32 + lane < units) { Kc[d] = kb[i]; Vc[d] = vb[i]; }
    }
    if (SLc != nullptr && lane < count) SLc[dst_row] = __ldg(SL + src_row);
}

// always_first = 0: wait for the preceding kernel, then copy every kept row through the index list.
// always_first = 1 (inside a layer step, directly behind the selection kernels, which let their
// dependents start at once): the rows that are kept whatever the scores say - sink and recent
// tokens, and all tokens of a stream that keeps everything - are copied first, while the
// selection still runs on its few SMs; only then does the kernel wait for the indices and copy
// the top-k rows.  K and V are not written by the step's earlier kernels, and the outputs are
// not read by them, so the early part touches nothing the predecessor produces.  (SL is the
// score array in a step: all of its entries are copied after the wait.)
// When the selection occupies more than kStaticSelect SMs, rows are handed out through two counters in the
// workspace header (`work`: early rows, late rows, finished blocks), a row or a group per claim with the
// next claim under way during the copy: the blocks that only get an SM when the selection's CTAs
// leave simply find less work left, instead of starting a fixed share late (that tail cost 40 us
// at the batch-4 size); the last block to finish puts the counters back to zero.  With a selection
// of one cluster the grid leaves its SMs out and every block takes a fixed share (early_static;
// selection and gather of the 28 080-token cache, selected by eight CTAs, 39.6 us with claiming, 31.4 with shares; of the
// 93 600-token one 33.5 and 29.3; four streams, 32 CTAs: no difference).
// A claim in two halves: lane 0 issues the add; its result is fetched (and shared with the warp)
// only when the rows are needed, so the trip to L2 overlaps the copying in between.
__device__ __forceinline__ int claim_issue(int* counter, int group, int lane) {
    return lane == 0 ? atomicAdd(counter, group) : 0;
}
__device__ __forceinline__ int64_t claim_get(int pending) { return __shfl_sync(0xffffffffu, pending, 0); }

// GROUPS: a warp copies `rows_at_once` narrow rows at a time.  A narrow row alone leaves most of a warp's batch empty: 48 000 rows
// of 256 bytes, selected from 76 000 in four streams, selection and gather together 56 us, in groups of 12 rows 29.4; 24 000
// rows of 1280 bytes 45.7 and 39.6.  (At the 80 registers of three blocks an SM the instantiation in groups spills 28 bytes; the other one nothing.)
template <bool GROUPS>
__global__ void __launch_bounds__(kCompactWarpsPerBlock * 32, 3)
compact_rows_kernel(const uint4* __restrict__ K, const uint4* __restrict__ V,
                    const float* __restrict__ SL, const int32_t* idx,
                    const __grid_constant__ StreamTable st, int32_t chunks_per_row,
                    uint4* __restrict__ Kc, uint4* __restrict__ Vc, float* __restrict__ SLc,
                    int64_t n_rows, int* __restrict__ work, int early_static, int rows_at_once) {
    const int group = GROUPS ? rows_at_once : 1;
    const int lane = threadIdx.x & 31;
    const uint32_t row_of = GROUPS ? rows_of_units(chunks_per_row, lane) : 0u;
    const int64_t warp0 = (int64_t)blockIdx.x * kCompactWarpsPerBlock + (threadIdx.x >> 5);
    const int64_t n_warps = (int64_t)gridDim.x * kCompactWarpsPerBlock;
    // rows [base, base + group) of n: `where` says where row i comes from and goes to
    auto copy = [&](int64_t base, int64_t n, auto where, const float* from, float* to) {
        int64_t src, dst;
        if constexpr (!GROUPS) {
            where(base, src, dst);
            copy_kv_row(K, V, from, src, dst, chunks_per_row, Kc, Vc, to, lane);
        } else {
            const int count = (int)(n - base < group ? n - base : group);
            where(base + (lane < count ? lane : 0), src, dst);
            copy_kv_rows(K, V, from, src, dst, count, chunks_per_row, Kc, Vc, to, lane, row_of);
        }
    };
    if (work == nullptr) {
        grid_dep_wait();
        auto kept = [&](int64_t r, int64_t& src, int64_t& dst) {
            int s = 0;
            while (s + 1 < st.n_streams && r >= st.cu_B[s + 1]) ++s;
            src = st.cu_T[s] + (int64_t)ld_index(idx + r); dst = r;
        };
        for (int64_t r = warp0 * group; r < n_rows; r += n_warps * group) copy(r, n_rows, kept, SL, SLc);
        return;
    }
    // part 1: always-kept rows, enumerated stream by stream (A_s = n_sink + n_recent of them, or all T)
    int64_t n_always = 0;
    for (int s = 0; s < st.n_streams; ++s) {
        const int64_t T = st.cu_T[s + 1] - st.cu_T[s], B = st.cu_B[s + 1] - st.cu_B[s];
        n_always += B >= T ? T : st.n_sink[s] + st.n_recent[s];
    }
    auto always = [&](int64_t a, int64_t& src, int64_t& dst) {
        int s = 0;
        int64_t p = a;
        for (;; ++s) {
            const int64_t T = st.cu_T[s + 1] - st.cu_T[s], B = st.cu_B[s + 1] - st.cu_B[s];
            const int64_t A = B >= T ? T : st.n_sink[s] + st.n_recent[s];
            if (p < A) break;
            p -= A;
        }
        const int64_t T = st.cu_T[s + 1] - st.cu_T[s], B = st.cu_B[s + 1] - st.cu_B[s];
        const int64_t ns = B >= T ? T : st.n_sink[s], k = B >= T ? 0 : st.k[s], A = B >= T ? T : ns + st.n_recent[s];
        // position p < ns is token p; position ns + k + i is token T - n_recent + i
        src = st.cu_T[s] + (p < ns ? p : T - A + p); dst = st.cu_B[s] + (p < ns ? p : p + k);
    };
    auto top = [&](int64_t q, int64_t& src, int64_t& dst) {
        int s = 0;
        int64_t p = q;
        for (; p >= st.k[s]; ++s) p -= st.k[s];
        dst = st.cu_B[s] + st.n_sink[s] + p;
        src = st.cu_T[s] + (int64_t)ld_index(idx + dst);
    };
    int64_t n_top = 0;
    for (int s = 0; s < st.n_streams; ++s) n_top += st.k[s];
    auto fill_always_sl = [&]() {
        if (SLc == nullptr) return;
        for (int64_t a = warp0 * 32 + lane; a < n_rows; a += n_warps * 32) {
            int s = 0;
            while (s + 1 < st.n_streams && a >= st.cu_B[s + 1]) ++s;
            const int64_t ns = st.n_sink[s], k = st.k[s], p = a - st.cu_B[s];
            if (k == 0 || p < ns || p >= ns + k) SLc[a] = __ldg(SL + st.cu_T[s] + ld_index(idx + a));
        }
    };
    if (early_static) {
        // every block is resident from the start (the launcher sized the grid for it): fixed shares
        for (int64_t a = warp0 * group; a < n_always; a += n_warps * group) copy(a, n_always, always, nullptr, nullptr);
        grid_dep_wait();
        fill_always_sl();
        for (int64_t q = warp0 * group; q < n_top; q += n_warps * group) copy(q, n_top, top, SL, SLc);
        return;
    }
    int pending = claim_issue(work + 0, group, lane);
    for (int64_t base = claim_get(pending); base < n_always; base = claim_get(pending)) {
        pending = claim_issue(work + 0, group, lane);
        copy(base, n_always, always, nullptr, nullptr);
    }
    // part 2: the selection's result
    grid_dep_wait();
    fill_always_sl();
    pending = claim_issue(work + 1, group, lane);
    for (int64_t base = claim_get(pending); base < n_top; base = claim_get(pending)) {
        pending = claim_issue(work + 1, group, lane);
        copy(base, n_top, top, SL, SLc);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(work + 2, 1) == (int)gridDim.x - 1) {      // every block is past its last claim
            work[0] = 0; work[1] = 0; work[2] = 0;
        }
    }
}

// The same gather for several layers' caches at once: the paper takes the Top-k at the final
// layer only and applies those indices to every layer (Sec. 3.3), so one index list serves
// n_layers K/V pairs.  One warp moves one (layer, kept token) pair of rows; the layer is the
// slowest index, so a warp's accesses stay contiguous and the index list is re-read from L2.
// (Bound by memory: 30 layers x 14 040 rows of 3072 bytes 798 us, 6.5 TB/s.  The row's copy is written out here: called
// as copy_kv_row it compiles to fewer registers and takes 948 us.)
struct LayerPtrs {
    const uint4* K[PAFU_MAX_LAYERS];
    const uint4* V[PAFU_MAX_LAYERS];
    uint4* Kc[PAFU_MAX_LAYERS];
    uint4* Vc[PAFU_MAX_LAYERS];
};

__global__ void __launch_bounds__(kCompactWarpsPerBlock * 32)
compact_layers_kernel(const __grid_constant__ LayerPtrs lp, int32_t n_layers,
                      const float* __restrict__ SL, const int32_t* idx,
                      const __grid_constant__ StreamTable st, int32_t chunks_per_row,
                      float* __restrict__ SLc, int64_t n_rows) {
    grid_dep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (int64_t)blockIdx.x * kCompactWarpsPerBlock + (threadIdx.x >> 5);
    const int64_t n_warps = (int64_t)gridDim.x * kCompactWarpsPerBlock;
    for (int64_t w = warp0; w < n_rows * n_layers; w += n_warps) {
        const int layer = (int)(w / n_rows);
        const int64_t r = w - (int64_t)layer * n_rows;
        int s = 0;
        while (s + 1 < st.n_streams && r >= st.cu_B[s + 1]) ++s;
        const int64_t src_row = st.cu_T[s] + (int64_t)ld_index(idx + r);
        const uint4* ks = lp.K[layer] + src_row * chunks_per_row;
        const uint4* vs = lp.V[layer] + src_row * chunks_per_row;
        uint4* kd = lp.Kc[layer] + r * chunks_per_row;
        uint4* vd = lp.Vc[layer] + r * chunks_per_row;
        for (int c0 = 0; c0 < chunks_per_row; c0 += 32 * kCompactUnroll) {
            uint4 kb[kCompactUnroll], vb[kCompactUnroll];
#pragma unroll
            for (int u = 0; u < kCompactUnroll; ++u) {
                const int c = c0 + u * 32 + lane;
                if (c < chunks_per_row) { kb[u] = ld_nc_v4(ks + c); vb[u] = ld_nc_v4(vs + c); }
            }
#pragma unroll
            for (int u = 0; u < kCompactUnroll; ++u) {
                const int c = c0 + u * 32 + lane;
                if (c < chunks_per_row) { kd[c] = kb[u]; vd[c] = vb[u]; }
            }
        }
        if (layer == 0 && SLc != nullptr && lane == 0) SLc[r] = __ldg(SL + src_row);
    }
}

static LayerPtrs layer_ptrs(const uint16_t* const* K, const uint16_t* const* V, uint16_t* const* Kc, uint16_t* const* Vc, int32_t n_layers) {
    LayerPtrs lp;
    for (int l = 0; l < PAFU_MAX_LAYERS; ++l) {
        const int i = l < n_layers ? l : 0;
        lp.K[l] = reinterpret_cast<const uint4*>(K[i]); lp.V[l] = reinterpret_cast<const uint4*>(V[i]);
        lp.Kc[l] = reinterpret_cast<uint4*>(Kc[i]); lp.Vc[l] = reinterpret_cast<uint4*>(Vc[i]);
    }
    return lp;
}

pafu_status launch_compact_layers(const uint16_t* const* K, const uint16_t* const* V, int32_t n_layers,
                                  const float* SL, const int32_t* idx, const StreamTable& st, int32_t d_model,
                                  uint16_t* const* Kc, uint16_t* const* Vc, float* SLc, cudaStream_t stream) {
    const int64_t n_rows = st.cu_B[st.n_streams];
    if (n_rows == 0 || n_layers == 0) return PAFU_OK;
    int64_t blocks = (n_rows * n_layers + kCompactWarpsPerBlock - 1) / kCompactWarpsPerBlock;
    const int64_t max_blocks = 148 * 8 * 4;
    if (blocks > max_blocks) blocks = max_blocks;
    return cuda_ok(launch_dependent(compact_layers_kernel, dim3((unsigned)blocks), dim3(kCompactWarpsPerBlock * 32), 0, stream, 1,
                                    layer_ptrs(K, V, Kc, Vc, n_layers), n_layers, SL, idx, st, d_model / 8, SLc, n_rows));
}

// A rolling-cache update's copies: the chunk's new rows of every layer, then the kept rows through the
// index list.  The new rows need nothing that the selection ahead produces, so they are copied while
// it runs; and the kernel lets the one behind it start at once: that is the salience head of the chunk,
// tensor-bound work on one CTA an SM, which this kernel leaves registers for (one block of 256 threads an SM), and where head_shares_sms()
// says so shared memory too.  (Without that the head starts on an SM only when its block has ended.  Tried for long copies: the head on 13, 19 or
// 37 SMs of its own, 30 layers of 12 heads 586 -> 610, 601 and 593 us, since the copies miss those SMs and slow the head's weight reads down;
// all of the L1 but 28 KB given to the head's block 677.)
//
// Bound by memory.  What one block an SM reaches is set by its bytes in flight, so a warp's batch is a stretch of
// kCompactUnroll x 32 sixteen-byte units of a layer's rows laid end to end, whatever the row width, and the
// batch's indices are fetched one batch ahead.  (With a row at a time a warp had only that row in flight: 30
// layers, 4680 kept and 4680 new rows of 256, 512, 1536, 3072 and 4096 bytes took 219, 243, 375, 590 and 828 us, now 71,
// 117, 305, 588 and 781; as select, gather, head and append one after the other, many blocks an SM, 140, 164, 324,
// 612 and 807.  With the indices fetched before the batch's loads instead of behind them 618 at 3072 bytes.)
constexpr int kCacheSeg = kCompactUnroll * 32;     // units of a warp's batch
constexpr int kCacheCarveout = kHeadSmemBeside * 100 / (228 * 1024);     // per cent, which the driver rounds up to the next split: of 72 % it makes 196 KB

// One batch: unit dst + 32 i comes from src[i]; `between` runs while its loads are under way.
template <typename Between>
__device__ __forceinline__ void copy_units(const uint4* K, const uint4* V, const uint32_t (&src)[kCompactUnroll], uint4* Kd, uint4* Vd,
                                           uint32_t dst, uint32_t end, Between between) {
    uint4 kb[kCompactUnroll], vb[kCompactUnroll];
#pragma unroll
    for (int i = 0; i < kCompactUnroll; ++i)
        if (dst + i * 32 < end) { kb[i] = ld_nc_v4(K + src[i]); vb[i] = ld_nc_v4(V + src[i]); }
    between();
#pragma unroll
    for (int i = 0; i < kCompactUnroll; ++i)
        if (dst + i * 32 < end) { Kd[dst + i * 32] = kb[i]; Vd[dst + i * 32] = vb[i]; }
}

// (A layer's buffer holds less than 2^32 units: 64 GiB.)
__global__ void __launch_bounds__(kCompactWarpsPerBlock * 32)
cache_rows_kernel(const __grid_constant__ LayerPtrs add, const __grid_constant__ LayerPtrs keep, uint32_t n_layers,
                  uint32_t n_new, int64_t dst0, const float* __restrict__ SL, const int32_t* idx, uint32_t n_keep,
                  uint32_t chunks_per_row, float* __restrict__ SLd, int behind_select) {
    if (!behind_select) grid_dep_wait();
    grid_dep_launch_dependents();     // everything ahead of the selection (or of this kernel) is complete here
    const int lane = threadIdx.x & 31;
    const uint32_t warp0 = blockIdx.x * kCompactWarpsPerBlock + (threadIdx.x >> 5);
    const uint32_t n_warps = gridDim.x * kCompactWarpsPerBlock;
    const uint32_t new_units = n_new * chunks_per_row, new_segs = (new_units + kCacheSeg - 1) / kCacheSeg;
    for (uint32_t w = warp0; w < new_segs * n_layers; w += n_warps) {
        const uint32_t layer = w / new_segs, u = (w - layer * new_segs) * kCacheSeg + lane;
        uint32_t src[kCompactUnroll];
#pragma unroll
        for (int i = 0; i < kCompactUnroll; ++i) src[i] = u + i * 32;
        copy_units(add.K[layer], add.V[layer], src, add.Kc[layer] + dst0 * chunks_per_row, add.Vc[layer] + dst0 * chunks_per_row, u, new_units,
                   [] {});
    }
    if (behind_select) grid_dep_wait();
    const uint32_t keep_units = n_keep * chunks_per_row, keep_segs = (keep_units + kCacheSeg - 1) / kCacheSeg;
    const uint32_t total = keep_segs * n_layers;
    auto fetch = [&](uint32_t w, uint32_t (&src)[kCompactUnroll]) {      // where batch w's units come from
        const uint32_t u = (w - w / keep_segs * keep_segs) * kCacheSeg + lane;
#pragma unroll
        for (int i = 0; i < kCompactUnroll; ++i) {
            const uint32_t row = (u + i * 32) / chunks_per_row;
            src[i] = 0;
            if (u + i * 32 < keep_units) src[i] = (uint32_t)ld_index(idx + row) * chunks_per_row + (u + i * 32 - row * chunks_per_row);
        }
    };
    uint32_t src[kCompactUnroll], ahead[kCompactUnroll];
    if (warp0 < total) fetch(warp0, src);
    for (uint32_t w = warp0; w < total; w += n_warps) {
        const uint32_t layer = w / keep_segs;
        copy_units(keep.K[layer], keep.V[layer], src, keep.Kc[layer], keep.Vc[layer], (w - layer * keep_segs) * kCacheSeg + lane,
                   keep_units, [&] { if (w + n_warps < total) fetch(w + n_warps, ahead); });
#pragma unroll
        for (int i = 0; i < kCompactUnroll; ++i) src[i] = ahead[i];
    }
    for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < n_keep; r += gridDim.x * blockDim.x) SLd[r] = __ldg(SL + ld_index(idx + r));
}

pafu_status launch_cache_rows(const uint16_t* const* Knew, const uint16_t* const* Vnew, int64_t n_new,
                              const uint16_t* const* Ks, const uint16_t* const* Vs, const float* SL, const int32_t* idx,
                              int64_t keep, int64_t dst0, uint16_t* const* Kd, uint16_t* const* Vd, float* SLd, int32_t n_layers,
                              int32_t d_model, int select_ctas, bool share_sms, cudaStream_t stream) {
    const int64_t cpr = d_model / 8;
    const int64_t segs = ((n_new * cpr + kCacheSeg - 1) / kCacheSeg + (keep * cpr + kCacheSeg - 1) / kCacheSeg) * n_layers;
    int64_t blocks = (segs + kCompactWarpsPerBlock - 1) / kCompactWarpsPerBlock;
    // one block an SM, in fixed shares; the selection's SMs are left out
    const int64_t most = device_sm_count() > select_ctas ? device_sm_count() - select_ctas : 1;
    if (blocks > most) blocks = most;
    return cuda_ok(launch_dependent_carveout(share_sms ? kCacheCarveout : -1, cache_rows_kernel, dim3((unsigned)blocks), dim3(kCompactWarpsPerBlock * 32), 0, stream, 1,
                                    layer_ptrs(Knew, Vnew, Kd, Vd, n_layers), layer_ptrs(Ks, Vs, Kd, Vd, n_layers), (uint32_t)n_layers,
                                    (uint32_t)n_new, dst0, SL, idx, (uint32_t)keep, (uint32_t)cpr, SLd, select_ctas > 0 ? 1 : 0));
}

// `work`: three zeroed 32-bit words of device memory (the step's workspace header) - then the
// always-kept rows are copied before the kernel waits for its predecessor, which must be
// launch_select of the same step and runs on `select_ctas` CTAs; nullptr: plain gather after the
// predecessor.
pafu_status launch_compact(const uint16_t* K, const uint16_t* V, const float* SL,
                           const int32_t* idx, const StreamTable& st, int32_t d_model,
                           uint16_t* Kc, uint16_t* Vc, float* SLc, cudaStream_t stream, int* work, int select_ctas) {
    const int64_t n_rows = st.cu_B[st.n_streams];
    if (n_rows == 0) return PAFU_OK;
    const int32_t chunks = d_model / 8;
    // A few resident waves, larger inputs loop.  With the early part the grid is what the device
    // holds at once (three blocks fit on an SM): a block must not queue behind blocks that are
    // waiting for the selection.  Fixed shares: the selection's SMs are left out of the count.
    const int early_static = work != nullptr && select_ctas <= kStaticSelect;
    int sms = device_sm_count() - (early_static ? select_ctas : 0);
    if (sms < 1) sms = 1;
    const int64_t max_blocks = work != nullptr ? (int64_t)sms * 3 : 148 * 8 * 4;
    // Rows a warp copies at once: as many as fill its batch, but no more than leave every warp some, and one where a warp has but one
    // or two (10 280 rows of 512 bytes in pairs: 48.5 us a step, one by one 47.7).
    const int64_t resident = (int64_t)device_sm_count() * 3 * kCompactWarpsPerBlock;
    int64_t group = kCompactUnroll * 32 / chunks;
    if (group > n_rows / resident) group = n_rows / resident;
    if (group > 32) group = 32;
    if (group < 1 || n_rows < 3 * resident || st.cu_T[st.n_streams] * chunks >= (int64_t)1 << 32) group = 1;   // (32-bit unit numbers in groups)
    int64_t blocks = (n_rows + kCompactWarpsPerBlock * group - 1) / (kCompactWarpsPerBlock * group);
    if (blocks > max_blocks) blocks = max_blocks;
    return cuda_ok(launch_dependent(group > 1 ? compact_rows_kernel<true> : compact_rows_kernel<false>, dim3((unsigned)blocks), dim3(kCompactWarpsPerBlock * 32), 0, stream, 1,
                                    reinterpret_cast<const uint4*>(K), reinterpret_cast<const uint4*>(V), SL, idx, st,
                                    chunks, reinterpret_cast<uint4*>(Kc), reinterpret_cast<uint4*>(Vc), SLc, n_rows, work,
                                    early_static, (int)group));
}

}  // namespace pafu
