// Chunk attention on the 5th-generation tensor cores (tcgen05 + TMEM + TMA), d_head = 128 (and 64:
// a second instantiation, see HeadDims; the text below gives the sizes for 128).
//
//   o_i = sum_j softmax_j(scale q_i.k_j) v_j,  j over [retained cache ; chunk tokens]
//   (Sec. 3.2 for the operator; Eq. 2 / Eq. 7 for the key range)
//
// Work decomposition.  An "item" is 256 query rows of one head of one stream, handled as two
// 128-row "slots" that share every K/V tile (each tile is fetched once per 256 rows).  The
// grid is persistent: one CTA per SM.  Items go out whole, round by round, while no CTA exceeds its
// even share of the work; the key tiles of the items that are left are laid end to end and cut
// into contiguous shares, one per CTA, so that every CTA ends with the same total whatever the item
// count (a tile with both slots live costs 8 units, with one slot 7: a lone slot has no partner to
// hide its softmax behind).  A CTA whose share covers only
// part of an item's keys writes an unnormalised partial (O, running max, row sum) to the
// workspace; a second small kernel merges the partials of each split item in key order, which
// keeps the result deterministic.
//
// Warp roles inside a CTA (384 threads):
//   warps 0-3  softmax of slot 0 (thread = query row = TMEM lane)
//   warps 4-7  softmax of slot 1
//   warps 8,10 MMA issuers, one per slot: S = Q K^T (both operands in shared memory) and
//              O += P V (P read from tensor memory, V from shared memory, MN-major).  The MMA
//              stream itself needs only one issuer (1238 clocks a tile pair either way), but each
//              tile also costs an issuer some 500 clocks of waits and commits, which a second one hides
//              (one warp for both slots: 2375 clocks a tile pair, two: 1634)
//   warp  9    TMA loader: Q tiles per item, 64-key K/V tiles through a 10-stage ring that
//              runs ahead across item boundaries
//   warp  11   idle (completes the third warpgroup so registers can be re-balanced)
// Tensor memory (512 columns): per slot two S buffers of 64 fp32 columns and one O accumulator
// of 128; the bf16 P tile overwrites the first 32 columns of its S buffer.  S is double
// buffered so that S(j+1) = Q K_{j+1}^T is already finished when the softmax of tile j ends:
// the softmax warps never wait for the tensor core in steady state, and the issuer's order
// "P(j) ready -> O += P(j) V_j -> S(j+2)" keeps the buffer reuse safe without extra barriers.
//
// Online softmax with lazy rescaling: the running maximum only moves when the new tile
// exceeds it by more than 2^8 in the exponent, so the O accumulator is rarely rescaled; when
// it is, the slot's own softmax warps do it after waiting for the previous P V product.  Small problems
// hand the tensor core P's rounding error as well (round_mode()).
//
// Every mbarrier wait is bounded.  A wait that runs out sets the status word, raises a CTA-wide
// abort flag, and all roles fall through to the common exit where TMEM is released.
#pragma once
#include <type_traits>

#include "attn_plan.cuh"
#include "common.cuh"
#include "sm100.cuh"

namespace pafu {
namespace attn_tc {

using namespace sm100;

constexpr int kStages = 10;         // K/V ring depth (each stage one 64 x 128 bf16 tile)
constexpr int kThreads = 384;       // 3 warpgroups: softmax 0, softmax 1, {2 MMA issuers, loader, 1 idle}
constexpr int kQBytes = kBM * kD * 2;         // 32 KiB: one slot's Q tile
constexpr int kQHalf = kQBytes / 2;           // one [128 rows x 64 cols] swizzled half
constexpr int kTileBytes = kBN * kD * 2;      // 16 KiB: one K or V tile
constexpr int kHalfBytes = kTileBytes / 2;    // one [64 rows x 64 cols] swizzled half
constexpr int kSmemBytes = 2 * kQBytes + kStages * kTileBytes + 1024 /*align*/ + 512 /*barriers*/;
constexpr float kRescaleThresholdLog2 = 8.0f;
constexpr float kSumTrigger = 65536.0f;   // a 64-key row sum this large means some p exceeded 2^10
// Register re-balancing.  With 384 threads the kernel launches with 168 registers per thread.
// setmaxnreg.inc blocks until the registers exist, so what the third warpgroup gives up must
// cover what the two softmax warpgroups take: (168 - kRegsLow) * 128 >= (kRegsHigh - 168) * 256.
constexpr int kRegsLaunch = 168, kRegsLow = 80, kRegsHigh = 208;
static_assert((kRegsLaunch - kRegsLow) * 128 >= (kRegsHigh - kRegsLaunch) * 256,
              "setmaxnreg.inc would wait forever");
// one partial: O [128][256] fp32 (column-major: a column's 256 rows together), then m [256], then l [256]
constexpr int kPieceFloats = 2 * kBM * kD + 2 * 2 * kBM;
constexpr size_t kPieceBytes = (size_t)kPieceFloats * 4;

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// packed fp32 pairs (two lanes per instruction on the FMA pipe)
__device__ __forceinline__ uint64_t pack2(uint32_t lo, uint32_t hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t fadd2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// what rounding (lo, hi) to the bf16 pair `rounded` left over, as a bf16 pair
__device__ __forceinline__ uint32_t pack_rest(float lo, float hi, uint32_t rounded) {
    return pack_bf16(lo - __uint_as_float(rounded << 16), hi - __uint_as_float(rounded & 0xffff0000u));
}

// The pieces of a tile's softmax that attn_stats_kernel shares, so that both form the same bits.
// Row sum of 2^(s * scale log2 e + mb) over 64 logits; `pk` (32 words), if given, receives the
// probabilities as bf16 pairs, and `lo` what that rounding leaves over.
__device__ __forceinline__ float tile_sum(const uint32_t (&sr)[64], uint64_t sl2_2, float mb, uint32_t* pk = nullptr, uint32_t* lo = nullptr) {
    const uint64_t mb_2 = pack2(__float_as_uint(mb), __float_as_uint(mb));
    uint64_t rs2[2] = {0ull, 0ull};
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        float e0, e1;
        unpack2(ffma2(pack2(sr[2 * c], sr[2 * c + 1]), sl2_2, mb_2), e0, e1);
        const float p0 = fast_exp2(e0), p1 = fast_exp2(e1);
        rs2[c & 1] = fadd2(rs2[c & 1], pack2(__float_as_uint(p0), __float_as_uint(p1)));
        if (pk != nullptr) pk[c] = pack_bf16(p0, p1);
        if (lo != nullptr) lo[c] = pack_rest(p0, p1, pk[c]);
    }
    float r0, r1, r2, r3;
    unpack2(rs2[0], r0, r1);
    unpack2(rs2[1], r2, r3);
    return (r0 + r1) + (r2 + r3);
}
__device__ __forceinline__ float tile_max(const uint32_t (&sr)[64]) {
    float mx4[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float m = fmaxf(__uint_as_float(sr[16 * q]), __uint_as_float(sr[16 * q + 1]));
#pragma unroll
        for (int c = 2; c < 16; c += 2)
            m = fmax3(m, __uint_as_float(sr[16 * q + c]), __uint_as_float(sr[16 * q + c + 1]));
        mx4[q] = m;
    }
    return fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
}
__device__ __forceinline__ float final_lse(float m, float scale, float l) {      // one rounding, the same bits wherever it is inlined
    return l > 0.f ? __fmaf_rn(m, scale, logf(l)) : -INFINITY;
}

// GATHER = false: the retained keys/values are the rows of a compacted cache (mKc, mVc are tiled
// maps of it).  GATHER = true: they are rows idx[.] of the uncompacted cache, fetched by the
// loader warps with 16-byte asynchronous copies, or tiled where a tile's rows follow one another (mKc, mVc are
// maps of that cache); everything downstream of the shared-memory ring is identical.
// Sizes that depend on the head width D (128, or 64: every tile is then a single 64-column
// swizzled block, S = Q K^T takes four slices and O has 64 columns).
template <int D>
struct HeadDims {
    static constexpr int kQBytes = kBM * D * 2;                  // one slot's Q tile
    static constexpr int kQHalf = kBM * 64 * 2;                  // one [128 rows x 64 cols] swizzled block of it
    static constexpr int kHalfBytes = kBN * 64 * 2;              // one [64 rows x 64 cols] swizzled block of a K or V tile
    static constexpr int kTileBytes = kBN * D * 2;
    static constexpr int kSmemBytes = 2 * kQBytes + kStages * kTileBytes + 1024 /*align*/ + 512 /*barriers*/;
    static constexpr int kPieceFloats = 2 * kBM * D + 2 * 2 * kBM;   // one partial: O [D][256], m [256], l [256]
};

template <bool GATHER, int D, int ROUND>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mKc,
               const __grid_constant__ CUtensorMap mVc, const __grid_constant__ CUtensorMap mKq,
               const __grid_constant__ CUtensorMap mVq, const __grid_constant__ Params p) {
    static_assert(D == 128 || (D == 64 && !GATHER), "head widths: 128, or 64 with a compacted cache");
    // this instantiation's sizes (they shadow the D = 128 constants of the namespace)
    constexpr int kD = D;
    constexpr int kQBytes = HeadDims<D>::kQBytes, kQHalf = HeadDims<D>::kQHalf;
    constexpr int kTileBytes = HeadDims<D>::kTileBytes, kHalfBytes = HeadDims<D>::kHalfBytes;
    constexpr int kPieceFloats = HeadDims<D>::kPieceFloats;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sQ = smem_u32(smem);                       // 2 slots x 32 KiB
    const uint32_t sKV = sQ + 2 * kQBytes;                    // ring
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + 2 * kQBytes + kStages * kTileBytes);
    const uint32_t bar0 = smem_u32(bars);
    auto q_full = [&](int s) { return bar0 + 8 * (0 + s); };
    auto q_empty = [&](int s) { return bar0 + 8 * (2 + s); };
    auto s_full = [&](int s, int b) { return bar0 + 8 * (4 + 2 * s + b); };
    // P-ready is per S buffer as well: the softmax may finish tile j+1 (whose S was computed
    // early) before the issuer has looked at tile j, and a single barrier would be lapped
    auto p_full = [&](int s, int b) { return bar0 + 8 * (8 + 2 * s + b); };
    auto pv_done = [&](int s) { return bar0 + 8 * (12 + s); };
    auto o_done = [&](int s) { return bar0 + 8 * (14 + s); };
    auto turn = [&](int s) { return bar0 + 8 * (16 + s); };
    auto kv_full = [&](int st) { return bar0 + 8 * (18 + st); };
    auto kv_empty = [&](int st) { return bar0 + 8 * (18 + kStages + st); };
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5;

    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(q_full(s), 1); mbar_init(q_empty(s), 1);
            mbar_init(s_full(s, 0), 1); mbar_init(s_full(s, 1), 1);
            mbar_init(p_full(s, 0), 4); mbar_init(p_full(s, 1), 4);   // one arrival per softmax warp
            mbar_init(pv_done(s), 1); mbar_init(o_done(s), 1);
            mbar_init(turn(s), 1);
        }
        for (int st = 0; st < kStages; ++st) {
            mbar_init(kv_full(st), GATHER ? 32 : 1);    // gather: every lane of the loader warp arrives
            mbar_init(kv_empty(st), 2);                 // both issuers release a stage
        }
        abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 8) { tmem_alloc(smem_u32(&tmem_base_sh), 512); tmem_relinquish(); }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_base_sh;
    grid_dep_wait();          // set-up above is local; everything below reads or writes global memory

    auto fail = [&](int code) {
        abort_flag = 1;
        atomicCAS(p.status, 0, code);
    };

    if (warp >= 8) {
    // register budget: this warpgroup gives registers up, the softmax warpgroups take them
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLow));
    if (warp == 11 && !GATHER) {
        // idle
    } else if (warp == 9 || warp == 11) {
        // ------------------------------------------------------------------ TMA loader
        if constexpr (GATHER) {
            // Two loader warps walk the runs together: warp 9 fills the K stages of the ring (and
            // loads Q), warp 11 the V stages.  Lane 0 issues the tiled loads (Q, the chunk's own
            // K/V).  A retained 64-key tile is fetched with 16-byte asynchronous copies: a lane owns
            // 16-byte pieces c and c + 4 of a row in both 64-column halves (4 lanes per row, 8 rows
            // per warp instruction, 4 x 8 instructions per tile) and writes them where the tiled load
            // would have put them (128-byte swizzle: piece c of row r goes to piece c ^ (r mod 8)),
            // so the operand layout is unchanged.  The tile's 64 rows sit
            // in two registers per lane, are handed round by shuffles and are fetched one tile
            // ahead of their use.  A tile whose rows follow one another in the cache (sink and recent tokens, runs of
            // kept ones) takes the tiled load instead: the layer step with 6240 of 7020 kept rows in two runs (12 heads x 4680
            // queries) 345 -> 333 us before the power cap acts, 382 -> 372 behind it.
            const int lane = tid & 31;
            const int kv = warp == 9 ? 0 : 1;
            const int r8 = lane >> 2, piece = lane & 3;           // row within a group of eight; pieces `piece` and `piece + 4`
            if (lane == 0) {
                if (kv == 0) prefetch_tmap(&mQ);
                prefetch_tmap(kv ? &mVc : &mKc);
                if (p.has_chunk) prefetch_tmap(kv ? &mVq : &mKq);
            }
            SegIter iter(p, blockIdx.x, gridDim.x);
            Seg g;
            uint32_t ring = (uint32_t)kv, qcnt0 = 0, qcnt1 = 0;     // this warp's stages: every other ring entry
            bool ok = true;
            auto wait_all = [&](uint32_t bar, uint32_t ph, int code) {
                const bool w = !abort_flag && mbar_wait(bar, ph);
                if (!__all_sync(0xffffffffu, w)) { if (lane == 0) fail(code); ok = false; }
            };
            const uint32_t row16 = (uint32_t)p.n_heads * (kD * 2 / 16);          // 16-byte units per token row
            // row = 8 it + r8, so row & 7 = r8: a lane's two swizzled positions never change
            const uint32_t dst_a = (uint32_t)(r8 * 128 + ((piece ^ r8) << 4));
            const uint32_t dst_b = (uint32_t)(r8 * 128 + (((piece + 4) ^ r8) << 4));
            while (ok && iter.next(p, g)) {
                if (kv == 0) {
                    const int qrow = (int)(p.st.cu_Lq[g.stream] + g.q0);
                    for (int s = 0; s < g.n_slots && ok; ++s) {
                        const uint32_t qc = s ? qcnt1 : qcnt0;
                        wait_all(q_empty(s), (qc & 1u) ^ 1u, 100);
                        if (!ok) break;
                        if (s) ++qcnt1; else ++qcnt0;
                        if (lane == 0) {
                            mbar_arrive_expect_tx(q_full(s), kQBytes);
                            tma_load_3d(sQ + s * kQBytes, &mQ, q_full(s), 0, g.head, qrow + s * kBM);
                            if constexpr (D == 128) tma_load_3d(sQ + s * kQBytes + kQHalf, &mQ, q_full(s), 64, g.head, qrow + s * kBM);
                        }
                    }
                }
                const int32_t* sidx = p.idx + p.st.cu_B[g.stream];
                const int row_base = (int)p.st.cu_T[g.stream];
                const uint8_t* base = reinterpret_cast<const uint8_t*>(kv ? p.Vraw : p.Kraw) +
                                      (size_t)g.head * (kD * 2) + piece * 16;
                // rows of a retained tile (rows past the segment's end repeat its last row:
                // their logits are masked, and their values must be finite)
                auto tile_rows = [&](int j, int& r0, int& r1) {
                    r0 = r1 = 0;
                    if (j < g.t1 && j < g.nt1) {
                        int64_t pos = (int64_t)j * kBN + lane;
                        r0 = row_base + ld_index(sidx + (pos < g.nB ? pos : g.nB - 1));
                        pos += 32;
                        r1 = row_base + ld_index(sidx + (pos < g.nB ? pos : g.nB - 1));
                    }
                };
                int r0, r1, n0, n1;
                tile_rows(g.t0, r0, r1);
                for (int j = g.t0; j < g.t1 && ok; ++j, ring += 2) {
                    const bool seg2 = j >= g.nt1;
                    const int st = ring % kStages;
                    tile_rows(j + 1, n0, n1);                        // the next tile's indices, one tile ahead
                    wait_all(kv_empty(st), ((ring / kStages) & 1u) ^ 1u, 101);
                    if (!ok) break;
                    const int first = __shfl_sync(0xffffffffu, r0, 0);
                    const bool run = __all_sync(0xffffffffu, r0 == first + lane && r1 == first + 32 + lane);
                    if (seg2 || run) {
                        if (lane == 0) {
                            const CUtensorMap* m = seg2 ? (kv ? &mVq : &mKq) : (kv ? &mVc : &mKc);
                            const int row = seg2 ? (int)(p.st.cu_Lq[g.stream] + (int64_t)(j - g.nt1) * kBN) : first;
                            mbar_arrive_expect_tx(kv_full(st), kTileBytes);
                            tma_load_3d(sKV + st * kTileBytes, m, kv_full(st), 0, g.head, row);
                            if constexpr (D == 128) tma_load_3d(sKV + st * kTileBytes + kHalfBytes, m, kv_full(st), 64, g.head, row);
                        } else {
                            mbar_arrive(kv_full(st));
                        }
                    } else {
                        const uint32_t dst0 = sKV + st * kTileBytes;
#pragma unroll
                        for (int it = 0; it < kBN / 8; ++it) {
                            const uint32_t off16 = (uint32_t)__shfl_sync(0xffffffffu, it < 4 ? r0 : r1, (8 * it + r8) & 31) * row16;
                            const uint8_t* src = base + (size_t)off16 * 16;
                            const uint32_t d = dst0 + it * 1024;
                            cp_async_16(d + dst_a, src);                                // columns 0..63
                            cp_async_16(d + dst_b, src + 64);
                            cp_async_16(d + dst_a + kHalfBytes, src + 128);             // columns 64..127
                            cp_async_16(d + dst_b + kHalfBytes, src + 192);
                        }
                        cp_async_mbar_arrive_noinc(kv_full(st));
                    }
                    r0 = n0; r1 = n1;
                }
            }
            if (!ok) {
                // let lane 0's copies already in flight land before the CTA exits
                for (uint32_t r = ring >= (uint32_t)kStages ? ring - kStages : (uint32_t)kv; r < ring; r += 2)
                    mbar_wait(kv_full(r % kStages), (r / kStages) & 1u);
                if (qcnt0 > 0) mbar_wait(q_full(0), (qcnt0 - 1) & 1u);
                if (qcnt1 > 0) mbar_wait(q_full(1), (qcnt1 - 1) & 1u);
            }
            cp_async_wait_all();
        } else if (elect_one() && p.status[kStatusWordStallLoader] == 0) {
            prefetch_tmap(&mQ); prefetch_tmap(&mKc); prefetch_tmap(&mVc);
            if (p.has_chunk) { prefetch_tmap(&mKq); prefetch_tmap(&mVq); }
            SegIter iter(p, blockIdx.x, gridDim.x);
            Seg g;
            uint32_t ring = 0, qcnt0 = 0, qcnt1 = 0;      // scalars: a runtime-indexed array would live in local memory
            bool ok = true;
            while (ok && iter.next(p, g)) {
                const int qrow = (int)(p.st.cu_Lq[g.stream] + g.q0);
                for (int s = 0; s < g.n_slots && ok; ++s) {
                    const uint32_t qc = s ? qcnt1 : qcnt0;
                    if (abort_flag || !mbar_wait(q_empty(s), (qc & 1u) ^ 1u)) { fail(100); ok = false; break; }
                    if (s) ++qcnt1; else ++qcnt0;
                    mbar_arrive_expect_tx(q_full(s), kQBytes);
                    tma_load_3d(sQ + s * kQBytes, &mQ, q_full(s), 0, g.head, qrow + s * kBM);
                    if constexpr (D == 128) tma_load_3d(sQ + s * kQBytes + kQHalf, &mQ, q_full(s), 64, g.head, qrow + s * kBM);
                }
                for (int j = g.t0; j < g.t1 && ok; ++j) {
                    const bool seg2 = j >= g.nt1;
                    const int row = seg2 ? (int)(p.st.cu_Lq[g.stream] + (int64_t)(j - g.nt1) * kBN)
                                         : (int)(p.st.cu_B[g.stream] + (int64_t)j * kBN);
                    for (int kv = 0; kv < 2; ++kv, ++ring) {
                        const int st = ring % kStages;
                        const uint32_t ph = (ring / kStages) & 1u;
                        if (abort_flag || !mbar_wait(kv_empty(st), ph ^ 1u)) { fail(101); ok = false; break; }
                        const CUtensorMap* m = seg2 ? (kv ? &mVq : &mKq) : (kv ? &mVc : &mKc);
                        mbar_arrive_expect_tx(kv_full(st), kTileBytes);
                        tma_load_3d(sKV + st * kTileBytes, m, kv_full(st), 0, g.head, row);
                        if constexpr (D == 128) tma_load_3d(sKV + st * kTileBytes + kHalfBytes, m, kv_full(st), 64, g.head, row);
                    }
                }
            }
            if (!ok) {
                // let copies already in flight land before the CTA exits
                for (uint32_t r = ring > (uint32_t)kStages ? ring - kStages : 0; r < ring; ++r)
                    mbar_wait(kv_full(r % kStages), (r / kStages) & 1u);
                if (qcnt0 > 0) mbar_wait(q_full(0), (qcnt0 - 1) & 1u);
                if (qcnt1 > 0) mbar_wait(q_full(1), (qcnt1 - 1) & 1u);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------- MMA issuers: warp 8 -> slot 0, warp 10 -> slot 1
        // The whole warp walks the loop and every value in it is warp-uniform (broadcasts and votes
        // tell the compiler so); only the tensor-core instructions are issued by one lane.  Their
        // descriptors and addresses then live in uniform registers: a loop run by a single elected
        // lane has to move six operands there for every MMA.
        {
            const bool leader = elect_one();
            const int slot = __shfl_sync(0xffffffffu, warp, 0) == 8 ? 0 : 1;
            const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
            const uint32_t idesc_qk = make_idesc_bf16(kBM, kBN, false, false);
            const uint32_t idesc_pv = make_idesc_bf16(kBM, kD, false, true);
            // Descriptors differ from tile to tile only in the 14-bit start-address field, so the
            // constant part is built once and the address (in 16-byte units) is added per MMA.
            const uint64_t desc_k = make_smem_desc_sw128(0, 16, 1024);             // K-major Q / K
            const uint64_t desc_v = make_smem_desc_sw128(0, kHalfBytes, 1024);     // MN-major V
            const uint32_t hi = (uint32_t)(desc_k >> 32);                          // the same for both
            const uint32_t lo_q = (uint32_t)desc_k + ((sQ + slot * kQBytes) >> 4);
            const uint32_t lo_k = (uint32_t)desc_k + (sKV >> 4), lo_v = (uint32_t)desc_v + (sKV >> 4);
            const uint32_t tSslot = tm + slot * 128;
            const uint32_t tOslot = tm + 256 + slot * kD;
            // d_head 128 issues in predicated series (12 heads x 18 720 keys 489 us, in a branch of the leader
            // 497); the short series of d_head 64 are the other way round (292 and 274 us at 13 680 keys).
            auto issue_qk = [&](int buf, int stage, bool pass) {     // S[buf] = Q K^T, N = 64 keys; `pass`: hand the turn on
                if constexpr (D == 64) {
                    if (leader) {
#pragma unroll
                        for (int kk = 0; kk < kD / 16; ++kk)
                            umma_ss(tSslot + buf * kBN, desc_k + ((sQ + slot * kQBytes) >> 4) + kk * 2,
                                    desc_k + ((sKV + stage * kTileBytes) >> 4) + kk * 2, idesc_qk, kk > 0);
                        umma_commit(s_full(slot, buf));
                        umma_commit(kv_empty(stage));
                    }
                    __syncwarp();
                    return;
                }
                if constexpr (GATHER) fence_proxy_async_smem();     // the tile came through the generic proxy
#pragma unroll
                for (int c = 0; c < kD / 64; ++c) {
                    if (c == kD / 64 - 1 && pass) elect_arrive(turn(slot ^ 1));
                    umma_ss_x4(tSslot + buf * kBN, lo_q + c * (kQHalf >> 4),
                               lo_k + stage * (kTileBytes >> 4) + c * (kHalfBytes >> 4), idesc_qk, hi, c > 0);
                }
                elect_commit(s_full(slot, buf));
                elect_commit(kv_empty(stage));
            };
            auto issue_pv = [&](int buf, int stage, bool first, auto split) {   // O += P[buf] V, K = 64 keys
                if constexpr (D == 64) {
                    if (leader) {
#pragma unroll
                        for (int kk = 0; kk < kBN / 16; ++kk)
                            umma_ts(tOslot, tSslot + buf * kBN + kk * 8, desc_v + ((sKV + stage * kTileBytes) >> 4) + kk * (2048 >> 4),
                                    idesc_pv, !(first && kk == 0));
                        if constexpr (decltype(split)::value) {
#pragma unroll
                            for (int kk = 0; kk < kBN / 16; ++kk)
                                umma_ts(tOslot, tSslot + buf * kBN + 32 + kk * 8, desc_v + ((sKV + stage * kTileBytes) >> 4) + kk * (2048 >> 4),
                                        idesc_pv, true);
                        }
                        umma_commit(kv_empty(stage));
                    }
                    __syncwarp();
                    return;
                }
                if constexpr (GATHER) fence_proxy_async_smem();
                umma_ts_x4(tOslot, tSslot + buf * kBN, lo_v + stage * (kTileBytes >> 4), idesc_pv, hi, !first);
                if constexpr (decltype(split)::value) umma_ts_x4(tOslot, tSslot + buf * kBN + 32, lo_v + stage * (kTileBytes >> 4), idesc_pv, hi, 1);
                elect_commit(kv_empty(stage));
            };
            bool ok = true;
            auto wait = [&](uint32_t bar, uint32_t ph, int code) {
                if (!mbar_wait_warp(bar, ph)) { if (leader) fail(code); ok = false; }
            };
            struct Cursor {                      // position of a ring entry: stage and phase bit
                uint32_t st, ph;
                __device__ __forceinline__ void step(uint32_t k) {
                    st += k;
                    if (st >= (uint32_t)kStages) { st -= kStages; ph ^= 1u; }
                }
            };
            SegIter iter(p, blockIdx.x, gridDim.x);
            Seg g;
            Cursor cur{0u, 0u};                  // first ring entry of the next run
            uint32_t qcnt = 0, tc = 0;           // tc: tiles this slot has processed so far
            uint32_t turns = 0;                  // turns this slot has taken
            while (ok && iter.next(p, g)) {
                const int n = __shfl_sync(0xffffffffu, g.t1 - g.t0, 0);
                // d_head 64 has half the tensor work and is bound by the exponentials: no turns (3 % faster)
                const bool two_slots = __shfl_sync(0xffffffffu, g.n_slots, 0) == 2, two = two_slots && D == 128;
                if (slot == 1 && !two_slots) {
                    // nothing to compute for this slot, but every K/V stage is released by both issuers
                    for (int e = 0; e < 2 * n && ok; ++e) {
                        wait(kv_full(cur.st), cur.ph, 206);
                        if (ok && leader) mbar_arrive(kv_empty(cur.st));
                        cur.step(1);
                    }
                    continue;
                }
                wait(q_full(slot), qcnt & 1u, 201);
                ++qcnt;
                // ring entries of this run: K_i at +2i, V_i at +2i+1
                Cursor ck = cur, cv = cur;
                cv.step(1);
                for (int i = 0; i < 2 && i < n && ok; ++i) {        // S(0), S(1)
                    wait(kv_full(ck.st), ck.ph, 202);
                    if (!ok) break;
                    tc_fence_after_sync();
                    issue_qk((tc + i) & 1, ck.st, false);
                    ck.step(2);
                }
                if (n == 1) ck.step(2);                              // keep ck two tiles ahead of cv
                // tiles [i0, i1) of the run; split: P is carried in two operands
                auto tiles = [&](int i0, int i1, auto split) {
#pragma unroll 1
                    for (int i = i0; i < i1 && ok; ++i) {
                        const int buf = (tc + i) & 1;
                        const bool more = i + 2 < n;
                        wait(kv_full(cv.st), cv.ph, 203);
                        if (!ok) break;
                        wait(p_full(slot, buf), ((tc + i) >> 1) & 1u, 205);
                        if (!ok) break;
                        // The slots take turns at the tensor core, a tile's P V and the next Q K^T at a time: left
                        // alone they fall into step, their MMAs interleave one by one and then both wait (some CTAs
                        // 690k clocks, most 800k; with turns 727k on all).  The turn is handed on before the
                        // last block of Q K^T so that the other slot's MMAs queue up behind it without a gap.
                        if (two) {
                            wait(turn(slot), (turns & 1u) ^ (slot == 0 ? 1u : 0u), 207);
                            if (!ok) break;
                            ++turns;
                        }
                        tc_fence_after_sync();
                        issue_pv(buf, cv.st, i == 0, split);
                        if (more) wait(kv_full(ck.st), ck.ph, 204);
                        if (!ok) break;
                        if (more) issue_qk(buf, ck.st, two);            // S(i+2) reuses the buffer P(i) was read from
                        else if (two) elect_arrive(turn(slot ^ 1));
                        if (i + 2 == n && leader) umma_commit(pv_done(slot));     // lets the last tile's softmax know O is at rest
                        if (i == n - 1 && leader) { umma_commit(o_done(slot)); umma_commit(q_empty(slot)); }
                        __syncwarp();
                        cv.step(2);
                        ck.step(2);
                    }
                };
                if constexpr (ROUND == kRoundOpening) {      // two loops, so that issue_pv knows its form
                    tiles(0, n < kOpeningTiles ? n : kOpeningTiles, std::true_type{});
                    tiles(kOpeningTiles, n, std::false_type{});
                } else {
                    tiles(0, n, std::integral_constant<bool, ROUND == kRoundSplit>{});
                }
                tc += (uint32_t)n;
                cur.step((2u * (uint32_t)n) % kStages);
                if (((2u * (uint32_t)n) / kStages) & 1u) cur.ph ^= 1u;
            }
        }
        __syncwarp();
    }
    } else {
        // ------------------------------------------------------------------ softmax warps
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsHigh));
        const int slot = warp >> 2;
        const int row_in_slot = tid & 127;
        const uint32_t lane_base = ((uint32_t)((warp & 3) * 32)) << 16;
        const uint32_t tSslot = tmem + slot * 128 + lane_base;
        const uint32_t tO = tmem + 256 + slot * kD + lane_base;
        const float sl2 = p.scale * 1.4426950408889634f;
        const uint64_t sl2_2 = pack2(__float_as_uint(sl2), __float_as_uint(sl2));
        SegIter iter(p, blockIdx.x, gridDim.x);
        Seg g;
        uint32_t tc = 0, ocnt = 0, pvcnt = 0;     // pvcnt: runs of two or more tiles so far
        bool ok = true;
        while (ok && iter.next(p, g)) {
            if (slot >= g.n_slots) continue;
            float m_used = -INFINITY, l_sum = 0.f;
            const int n = g.t1 - g.t0;
            uint32_t sr[64];
            bool loaded = false;                       // S(i) already requested from tensor memory
            for (int i = 0; i < n; ++i) {
                const int j = g.t0 + i;
                const int buf = (tc + i) & 1;
                const uint32_t tS = tSslot + buf * kBN;
                if (!loaded) {
                    const bool w = mbar_wait_spin(s_full(slot, buf), ((tc + i) >> 1) & 1u) && !abort_flag;
                    if (!__all_sync(0xffffffffu, w)) { fail(301); ok = false; break; }   // warp-uniform
                    tc_fence_after_sync();
                    PAFU_TMEM_LD_X32(tS, sr);
                    PAFU_TMEM_LD_X32(tS + 32, sr + 32);
                }
                loaded = false;
                tmem_wait_ld();
                const bool seg2 = j >= g.nt1;
                const int64_t left = (seg2 ? g.nC - (int64_t)(j - g.nt1) * kBN : g.nB - (int64_t)j * kBN);
                // Fast path (every tile but a run's first and a segment's ragged last): the
                // exponentials use the running maximum as it stands.  Only when the tile's row sum
                // shows that some logit outgrew that maximum by more than 2^10 does the tile take
                // the full pass below (true maximum, rescale of O and of the row sum).
                const bool opening = i < (ROUND == kRoundOpening ? kOpeningTiles : 1);
                bool full_pass = opening || (left < kBN);
                if (!full_pass) {
                    const float mbf = -m_used * sl2;
                    const uint64_t mb_2 = pack2(__float_as_uint(mbf), __float_as_uint(mbf));
                    uint64_t rs2[2] = {0ull, 0ull};
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t pk[16], lo[ROUND == kRoundSplit ? 16 : 1];
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            float e0, e1;
                            unpack2(ffma2(pack2(sr[32 * c + 2 * q], sr[32 * c + 2 * q + 1]), sl2_2, mb_2), e0, e1);
                            const float p0 = fast_exp2(e0), p1 = fast_exp2(e1);
                            rs2[q & 1] = fadd2(rs2[q & 1], pack2(__float_as_uint(p0), __float_as_uint(p1)));
                            pk[q] = pack_bf16(p0, p1);
                            if constexpr (ROUND == kRoundSplit) lo[q] = pack_rest(p0, p1, pk[q]);
                        }
                        PAFU_TMEM_ST_X16(tS + 16 * c, pk);
                        if constexpr (ROUND == kRoundSplit) PAFU_TMEM_ST_X16(tS + 32 + 16 * c, lo);
                    }
                    float r0, r1, r2, r3;
                    unpack2(rs2[0], r0, r1);
                    unpack2(rs2[1], r2, r3);
                    const float rs = (r0 + r1) + (r2 + r3);
                    full_pass = __any_sync(0xffffffffu, !(rs < kSumTrigger));    // also true for inf / NaN
                    if (!full_pass) l_sum += rs;
                } else if (left < kBN) {               // ragged end of a key segment
#pragma unroll
                    for (int c = 0; c < kBN; ++c)
                        if (c >= left) sr[c] = 0xff800000u;   // -inf
                }
                if (full_pass) {
                    if ((tid & 31) == 0) atomicAdd(p.status + ((opening || left < kBN) ? kStatusWordFullFirst : kStatusWordFullSum), 1);
                    const float mx = tile_max(sr);
                    if (i == 0) {
                        m_used = mx;
                    } else if (__any_sync(0xffffffffu, (mx - m_used) * sl2 > kRescaleThresholdLog2)) {
                        // The whole warp rescales together (TMEM accesses are warp-collective); rows
                        // whose maximum did not move get alpha = 1.  O must be at rest, i.e. the previous
                        // tile's P V product finished: S(i+1) being ready implies it (it was issued
                        // after that product); the run's last tile has a barrier of its own.
                        const bool w = (i + 1 < n ? mbar_wait(s_full(slot, buf ^ 1), ((tc + i + 1) >> 1) & 1u)
                                                  : mbar_wait(pv_done(slot), pvcnt & 1u)) && !abort_flag;
                        if (!__all_sync(0xffffffffu, w)) { fail(303); ok = false; break; }
                        tc_fence_after_sync();
                        if ((tid & 31) == 0) atomicAdd(p.status + kStatusWordRescale, 1);
                        const float m_new = fmaxf(m_used, mx);
                        const float alpha = fast_exp2((m_used - m_new) * sl2);
                        l_sum = __fmul_rn(l_sum, alpha);
                        m_used = m_new;
#pragma unroll
                        for (int c = 0; c < kD / 32; ++c) {
                            uint32_t orr[32];
                            PAFU_TMEM_LD_X32(tO + c * 32, orr);
                            tmem_wait_ld();
#pragma unroll
                            for (int q = 0; q < 32; ++q) orr[q] = __float_as_uint(__uint_as_float(orr[q]) * alpha);
                            PAFU_TMEM_ST_X32(tO + c * 32, orr);
                        }
                    }
                    uint32_t pk[32], lo[ROUND != kRoundPlain ? 32 : 1];
                    l_sum += tile_sum(sr, sl2_2, -m_used * sl2, pk, ROUND != kRoundPlain ? lo : nullptr);
                    PAFU_TMEM_ST_X32(tS, pk);
                    if constexpr (ROUND != kRoundPlain) PAFU_TMEM_ST_X32(tS + 32, lo);      // read only where issue_pv is told to
                }   // full_pass
                if (i + 1 < n && __all_sync(0xffffffffu, mbar_test_wait(s_full(slot, buf ^ 1), ((tc + i + 1) >> 1) & 1u))) {
                    // S(i+1) is already complete: request it now, so that its trip from tensor
                    // memory overlaps the hand-over of P(i)
                    tc_fence_after_sync();
                    PAFU_TMEM_LD_X32(tSslot + (buf ^ 1) * kBN, sr);
                    PAFU_TMEM_LD_X32(tSslot + (buf ^ 1) * kBN + 32, sr + 32);
                    loaded = true;
                }
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                if ((tid & 31) == 0) mbar_arrive(p_full(slot, buf));
            }
            if (!ok) break;
            tc += (uint32_t)n;
            if (n >= 2) ++pvcnt;
            {
                const bool w = mbar_wait(o_done(slot), ocnt & 1u) && !abort_flag;
                if (!__all_sync(0xffffffffu, w)) { fail(302); ok = false; break; }
                ++ocnt;
            }
            tc_fence_after_sync();
            const int64_t row = g.q0 + slot * kBM + row_in_slot;
            if (g.piece < 0) {
                // whole item: normalise and store bf16
                const float inv = (l_sum > 0.f) ? 1.0f / l_sum : 0.f;
                uint16_t* dst = p.O + ((p.st.cu_Lq[g.stream] + row) * p.n_heads + g.head) * kD;
#pragma unroll
                for (int c = 0; c < kD / 32; ++c) {
                    uint32_t orr[32];
                    PAFU_TMEM_LD_X32(tO + c * 32, orr);
                    tmem_wait_ld();
                    if (row < g.Lq) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            uint4 v;
                            v.x = pack_bf16(__uint_as_float(orr[8 * q + 0]) * inv, __uint_as_float(orr[8 * q + 1]) * inv);
                            v.y = pack_bf16(__uint_as_float(orr[8 * q + 2]) * inv, __uint_as_float(orr[8 * q + 3]) * inv);
                            v.z = pack_bf16(__uint_as_float(orr[8 * q + 4]) * inv, __uint_as_float(orr[8 * q + 5]) * inv);
                            v.w = pack_bf16(__uint_as_float(orr[8 * q + 6]) * inv, __uint_as_float(orr[8 * q + 7]) * inv);
                            *reinterpret_cast<uint4*>(dst + c * 32 + q * 8) = v;
                        }
                    }
                }
                if (p.LSE != nullptr && row < g.Lq)
                    p.LSE[(int64_t)g.head * p.total_Lq + p.st.cu_Lq[g.stream] + row] =
                        final_lse(m_used, p.scale, l_sum);
            } else {
                // part of an item: unnormalised fp32 partial for the merge kernel
                float* piece = p.pieces + ((size_t)blockIdx.x * 2 + g.piece) * kPieceFloats;
                const int prow = slot * kBM + row_in_slot;
                // column by column, so that a warp's 32 rows are 128 contiguous bytes (row by row the
                // two partials of a CTA took 10 us to write)
                float* dst = piece + prow;
#pragma unroll
                for (int c = 0; c < kD / 32; ++c) {
                    uint32_t orr[32];
                    PAFU_TMEM_LD_X32(tO + c * 32, orr);
                    tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < 32; ++q) dst[(c * 32 + q) * (2 * kBM)] = __uint_as_float(orr[q]);
                }
                piece[2 * kBM * kD + prow] = m_used;
                piece[2 * kBM * kD + 2 * kBM + prow] = l_sum;
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tmem, 512);
}

// Merges the partials of every item that was split across CTAs.  The host walks the CTAs'
// shares once per launch and passes the work as a table: item i was begun by CTA cta[first]
// (its last run, stored as that CTA's piece 1) and continued by the following entries (each
// CTA's first run, piece 0), in key order.  Sums are formed in a fixed order, which keeps the result
// deterministic.  Bound by the pieces' way through L2: two kernels, by how many pieces the longest item has.
constexpr int kMergeThreads = 256;
constexpr int kMergeWarps = kMergeThreads / 32;
__device__ __forceinline__ const float* merge_piece(const MergeTable& tb, const MergeItem& it, const float* pieces, int i, int piece_floats) {
    return pieces + ((size_t)tb.cta[it.first + i] * 2 + (i == 0 ? 1 : 0)) * piece_floats;
}
__device__ __forceinline__ float4 ld_f4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 fmax4(float4 a, float4 b) {
    return make_float4(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z), fmaxf(a.w, b.w));
}
__device__ __forceinline__ float4 merge_weights(float4 m, float4 M, float sl2) {
    return make_float4(fast_exp2((m.x - M.x) * sl2), fast_exp2((m.y - M.y) * sl2), fast_exp2((m.z - M.z) * sl2), fast_exp2((m.w - M.w) * sl2));
}
__device__ __forceinline__ void fma4(float4& acc, float4 w, float4 v) {
    acc.x = __fmaf_rn(w.x, v.x, acc.x); acc.y = __fmaf_rn(w.y, v.y, acc.y); acc.z = __fmaf_rn(w.z, v.z, acc.z); acc.w = __fmaf_rn(w.w, v.w, acc.w);
}

// Few pieces: such a problem has so many items that their rows alone fill the GPU.  A block takes 32 rows, a warp an eighth of
// the columns, a lane four rows of every fourth of those, so that a column's rows are read as whole 128-byte
// lines; the pieces follow one another.  (Groups of eight rows, 32 bytes of a line at a time, pieces shared out between two
// warps: 12 heads x 1764 queries x 2595 keys, 84 items of two or three pieces,
// 15.6 us, now 8.6; 4 streams x 40 heads of the 14B-class layer 19.8 and 10.5.  With up to 20 pieces here 12 heads x 4680 keys x
// 256 queries, 12 pieces an item, take 13.0 us instead of 7.2.)
// OUT = false: only the log-sum-exps are merged (attn_stats_kernel's pieces hold nothing else).
constexpr int kFewPieces = 8;
constexpr int kFewRows = 32;
template <int D, bool OUT>
__global__ void __launch_bounds__(kMergeThreads)
attn_tc_merge_few_kernel(const __grid_constant__ MergeTable tb, const float* pieces, float scale,
                         int n_heads, int64_t total_Lq, uint16_t* O, float* LSE) {
    constexpr int kPieceFloats = HeadDims<D>::kPieceFloats;
    constexpr int kCols = D / kMergeWarps / 4;                         // columns of a lane
    __shared__ float part[OUT ? kFewRows : 1][OUT ? D + 1 : 1];        // odd pitch: the lanes' four rows and columns hit 32 banks
    grid_dep_wait();
    constexpr int kBlocks = 2 * kBM / kFewRows;
    const MergeItem& it = tb.item[blockIdx.x / kBlocks];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b0 = (blockIdx.x % kBlocks) * kFewRows;                  // rows of the item (slot * 128 + row of the slot)
    if (b0 >= it.rows) return;                                         // block-uniform
    const int n_pieces = it.n_pieces;
    const float sl2 = scale * 1.4426950408889634f;
    const int rs = (lane & 7) * 4, col = warp * (D / kMergeWarps) + (lane >> 3);
    float4 M = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
#pragma unroll 4
    for (int i = 0; i < n_pieces; ++i) M = fmax4(M, ld_f4(merge_piece(tb, it, pieces, i, kPieceFloats) + 2 * kBM * D + b0 + rs));
    float4 L = make_float4(0.f, 0.f, 0.f, 0.f), acc[OUT ? kCols : 1];
#pragma unroll
    for (int k = 0; k < (OUT ? kCols : 1); ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
    for (int i = 0; i < n_pieces; ++i) {
        const float* piece = merge_piece(tb, it, pieces, i, kPieceFloats) + b0 + rs;
        float4 v[OUT ? kCols : 1];
        if (OUT) {
#pragma unroll
            for (int k = 0; k < kCols; ++k) v[k] = ld_f4(piece + (size_t)(col + 4 * k) * (2 * kBM));
        }
        const float4 w = merge_weights(ld_f4(piece + 2 * kBM * D), M, sl2);
        fma4(L, w, ld_f4(piece + 2 * kBM * D + 2 * kBM));
        if (OUT) {
#pragma unroll
            for (int k = 0; k < kCols; ++k) fma4(acc[k], w, v[k]);
        }
    }
    const float Mr[4] = {M.x, M.y, M.z, M.w}, Lr[4] = {L.x, L.y, L.z, L.w};
    if (OUT) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float inv = (Lr[q] > 0.f) ? 1.0f / Lr[q] : 0.f;
#pragma unroll
            for (int k = 0; k < kCols; ++k)
                part[rs + q][col + 4 * k] = (q == 0 ? acc[k].x : q == 1 ? acc[k].y : q == 2 ? acc[k].z : acc[k].w) * inv;
        }
    }
    if (LSE != nullptr && warp == 0 && lane < 8) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (b0 + rs + q < it.rows) LSE[(int64_t)it.head * total_Lq + it.o_row + b0 + rs + q] = final_lse(Mr[q], scale, Lr[q]);
    }
    if (OUT) {
        __syncthreads();
        for (int r = warp; r < kFewRows && b0 + r < it.rows; r += kMergeWarps) {
            uint32_t* dst = reinterpret_cast<uint32_t*>(O + (((int64_t)it.o_row + b0 + r) * n_heads + it.head) * D);
#pragma unroll
            for (int h = 0; h < D / 64; ++h) dst[h * 32 + lane] = pack_bf16(part[r][h * 64 + 2 * lane], part[r][h * 64 + 2 * lane + 1]);
        }
    }
}

// Many pieces: a few items cut up over dozens of CTAs.  A block takes eight rows, each of its eight warps every eighth
// piece of them, and the warps' sums are added in warp order: the pieces come from L2, a trip of about a microsecond, so
// they are fetched side by side (with a warp walking all pieces of its rows one after the other an item of 37 pieces took
// 67 us).  Four blocks an SM fit with d_head 64 without spills (7.4 -> 6.2 us at 11 pieces); with 128 they cost one (7.2 -> 8.4).
constexpr int kMergeRows = 8;
static_assert(kMergeRows == kMergeWarps, "each warp finishes one row");
template <int D, bool OUT>
__global__ void __launch_bounds__(kMergeThreads, D == 64 ? 4 : 3)
attn_tc_merge_kernel(const __grid_constant__ MergeTable tb, const float* pieces, float scale,
                     int n_heads, int64_t total_Lq, uint16_t* O, float* LSE) {
    constexpr int kPieceFloats = HeadDims<D>::kPieceFloats;
    constexpr int kVec = D / 4;                                        // float4 per row of the output
    constexpr int kPitch = OUT ? D + 4 : 4;                            // floats: 16-byte rows, four of them half the banks apart
    __shared__ __align__(16) float part[kMergeWarps][kMergeRows][kPitch];
    __shared__ float part_l[kMergeWarps][kMergeRows];
    grid_dep_wait();
    constexpr int kBlocks = 2 * kBM / kMergeRows;
    const MergeItem& it = tb.item[blockIdx.x / kBlocks];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b0 = (blockIdx.x % kBlocks) * kMergeRows;                // rows of the item (slot * 128 + row of the slot)
    if (b0 >= it.rows) return;                                         // block-uniform
    const int n_pieces = it.n_pieces;
    const float sl2 = scale * 1.4426950408889634f;
    const int rs = (lane & 1) * 4, d0 = lane >> 1;                     // this lane's four rows, and its columns d0 + 16 k
    // the rows' maxima over all pieces (every warp for itself, a lane pair per piece)
    float4 M = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    for (int i = d0; i < n_pieces; i += 16) M = fmax4(M, ld_f4(merge_piece(tb, it, pieces, i, kPieceFloats) + 2 * kBM * D + b0 + rs));
#pragma unroll
    for (int o = 16; o > 1; o >>= 1)
        M = fmax4(M, make_float4(__shfl_xor_sync(0xffffffffu, M.x, o), __shfl_xor_sync(0xffffffffu, M.y, o),
                                 __shfl_xor_sync(0xffffffffu, M.z, o), __shfl_xor_sync(0xffffffffu, M.w, o)));
    // this warp's pieces
    float4 L = make_float4(0.f, 0.f, 0.f, 0.f), acc[OUT ? D / 16 : 1];
#pragma unroll
    for (int k = 0; k < (OUT ? D / 16 : 1); ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = warp; i < n_pieces; i += kMergeWarps) {
        const float* piece = merge_piece(tb, it, pieces, i, kPieceFloats) + b0 + rs;
        const float4 m = ld_f4(piece + 2 * kBM * D), l = ld_f4(piece + 2 * kBM * D + 2 * kBM);
        float4 v[OUT ? D / 16 : 1];
        if (OUT) {
#pragma unroll
            for (int k = 0; k < D / 16; ++k) v[k] = ld_f4(piece + (size_t)(k * 16 + d0) * (2 * kBM));
        }
        const float4 w = merge_weights(m, M, sl2);
        fma4(L, w, l);
        if (OUT) {
#pragma unroll
            for (int k = 0; k < D / 16; ++k) fma4(acc[k], w, v[k]);
        }
    }
    if (OUT) {
#pragma unroll
        for (int k = 0; k < D / 16; ++k) {
            part[warp][rs + 0][k * 16 + d0] = acc[k].x; part[warp][rs + 1][k * 16 + d0] = acc[k].y;
            part[warp][rs + 2][k * 16 + d0] = acc[k].z; part[warp][rs + 3][k * 16 + d0] = acc[k].w;
        }
    }
    if (d0 == 0) { part_l[warp][rs + 0] = L.x; part_l[warp][rs + 1] = L.y; part_l[warp][rs + 2] = L.z; part_l[warp][rs + 3] = L.w; }
    __syncthreads();
    // each warp finishes one row
    const int row = b0 + warp;
    if (row >= it.rows) return;
    const int q = warp & 3;
    const float Mr = __shfl_sync(0xffffffffu, q == 0 ? M.x : q == 1 ? M.y : q == 2 ? M.z : M.w, warp >> 2);   // lane 0 holds rows 0..3, lane 1 4..7
    const int n_sum = n_pieces < kMergeWarps ? n_pieces : kMergeWarps;
    float Ls = 0.f;
    float4 o4 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int w = 0; w < n_sum; ++w) {
        Ls += part_l[w][warp];
        if (OUT && lane < kVec) {
            const float4 x = ld_f4(&part[w][warp][lane * 4]);
            o4.x += x.x; o4.y += x.y; o4.z += x.z; o4.w += x.w;
        }
    }
    if (OUT && lane < kVec) {
        const float inv = (Ls > 0.f) ? 1.0f / Ls : 0.f;
        uint2 o;
        o.x = pack_bf16(o4.x * inv, o4.y * inv);
        o.y = pack_bf16(o4.z * inv, o4.w * inv);
        *reinterpret_cast<uint2*>(O + (((int64_t)it.o_row + row) * n_heads + it.head) * D + lane * 4) = o;
    }
    if (LSE != nullptr && lane == 0) LSE[(int64_t)it.head * total_Lq + it.o_row + row] = final_lse(Mr, scale, Ls);
}

template <int D, bool OUT>
inline pafu_status launch_merge(const Params& p, int grid, int32_t n_heads, cudaStream_t stream) {
    if (grid <= 1) return PAFU_OK;
    MergeTable tb;
    build_merge_table(p, grid, tb);
    if (tb.n_items == 0) return PAFU_OK;
    const bool few = tb.longest <= kFewPieces;
    return cuda_ok(launch_dependent(few ? attn_tc_merge_few_kernel<D, OUT> : attn_tc_merge_kernel<D, OUT>,
                                    dim3(tb.n_items * (2 * kBM / (few ? kFewRows : kMergeRows))), dim3(kMergeThreads), 0, stream, 1,
                                    tb, (const float*)p.pieces, p.scale, (int)n_heads, p.total_Lq, p.O, p.LSE));
}

// True when every stream with queries has at least one key (the cost line has no entry for a
// key-less item).
inline bool supports(const StreamTable& st, bool has_chunk) {
    for (int s = 0; s < st.n_streams; ++s) {
        const int64_t lq = st.cu_Lq[s + 1] - st.cu_Lq[s], nB = st.cu_B[s + 1] - st.cu_B[s];
        if (lq > 0 && nB == 0 && !has_chunk) return false;
    }
    return true;
}

// Scratch for the partials: one pair per CTA.
inline size_t workspace_bytes() { return (size_t)sm_count() * 2 * kPieceBytes; }

// Tensor maps are rebuilt per call (a few microseconds of host work); nothing is cached, so
// the library stays stateless.  D: head width (128; 64 with a compacted cache only).
template <int D>
inline pafu_status launch_d(const uint16_t* Q, const uint16_t* Kc, const uint16_t* Vc,
                            const uint16_t* Kq, const uint16_t* Vq, const StreamTable& st,
                            int32_t n_heads, float scale, uint16_t* O, float* LSE, int* status,
                            float* pieces, cudaStream_t stream, int max_ctas, const int32_t* idx) {
    constexpr int kSmem = HeadDims<D>::kSmemBytes;
    const int n = st.n_streams;
    const int64_t nQ = st.cu_Lq[n], nB = st.cu_B[n];
    const int has_chunk = Kq != nullptr;
    const int64_t cost = total_cost(st, n_heads, has_chunk);
    if (cost == 0) return PAFU_OK;
    CUtensorMap mQ, mKc, mVc, mKq, mVq;
    if (!TmapEncoder::token_tensor(&mQ, Q, (uint64_t)nQ, n_heads, D, kBM)) return PAFU_ERR_CUDA;
    const bool gather = idx != nullptr;      // Kc, Vc are then the uncompacted cache
    if (gather && D != 128) return PAFU_ERR_UNSUPPORTED_SHAPE;
    if (nB > 0 && gather) {                // the uncompacted cache, for runs of neighbouring rows
        if (!TmapEncoder::token_tensor(&mKc, Kc, (uint64_t)st.cu_T[n], n_heads, D, kBN) ||
            !TmapEncoder::token_tensor(&mVc, Vc, (uint64_t)st.cu_T[n], n_heads, D, kBN)) return PAFU_ERR_CUDA;
    } else if (nB > 0) {
        if (!TmapEncoder::token_tensor(&mKc, Kc, (uint64_t)nB, n_heads, D, kBN) ||
            !TmapEncoder::token_tensor(&mVc, Vc, (uint64_t)nB, n_heads, D, kBN)) return PAFU_ERR_CUDA;
    } else { mKc = mQ; mVc = mQ; }
    if (has_chunk) {
        if (!TmapEncoder::token_tensor(&mKq, Kq, (uint64_t)nQ, n_heads, D, kBN) ||
            !TmapEncoder::token_tensor(&mVq, Vq, (uint64_t)nQ, n_heads, D, kBN)) return PAFU_ERR_CUDA;
    } else { mKq = mQ; mVq = mQ; }
    Params p;
    p.st = st; p.n_heads = n_heads; p.has_chunk = has_chunk; p.scale = scale;
    p.O = O; p.LSE = LSE; p.status = status; p.pieces = pieces; p.idx = idx; p.Kraw = gather ? Kc : nullptr; p.Vraw = gather ? Vc : nullptr; p.total_Lq = nQ;
    static bool attr_set[kMaxDevices] = {};
    if (!once_per_device(attr_set, [] {
            auto opt_in = [](auto* kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) == cudaSuccess; };
            if (!opt_in(attn_tc_kernel<false, D, kRoundPlain>) || !opt_in(attn_tc_kernel<false, D, kRoundSplit>) ||
                !opt_in(attn_tc_kernel<false, D, kRoundOpening>)) return false;
            if constexpr (D == 128)
                return opt_in(attn_tc_kernel<true, 128, kRoundPlain>) && opt_in(attn_tc_kernel<true, 128, kRoundSplit>) &&
                       opt_in(attn_tc_kernel<true, 128, kRoundOpening>);
            return true;
        }))
        return PAFU_ERR_CUDA;
    bool whole;
    const int grid = grid_for(st, n_heads, has_chunk, cost, max_ctas, whole);
    plan_shares(p, grid, cost, whole);
    const int mode = round_mode(st, has_chunk, cost, max_ctas, whole);
    auto go = [&](auto* kernel) { return launch_dependent(kernel, dim3(grid), dim3(kThreads), kSmem, stream, 1, mQ, mKc, mVc, mKq, mVq, p); };
    cudaError_t le = cudaSuccess;
    if constexpr (D == 128) {
        if (gather) le = mode == kRoundPlain ? go(attn_tc_kernel<true, 128, kRoundPlain>) : mode == kRoundSplit ? go(attn_tc_kernel<true, 128, kRoundSplit>)
                                                                                                             : go(attn_tc_kernel<true, 128, kRoundOpening>);
    }
    if (!gather) le = mode == kRoundPlain ? go(attn_tc_kernel<false, D, kRoundPlain>) : mode == kRoundSplit ? go(attn_tc_kernel<false, D, kRoundSplit>)
                                                                                                        : go(attn_tc_kernel<false, D, kRoundOpening>);
    if (le != cudaSuccess) return PAFU_ERR_CUDA;
    return launch_merge<D, true>(p, grid, n_heads, stream);
}

inline pafu_status launch(const uint16_t* Q, const uint16_t* Kc, const uint16_t* Vc,
                          const uint16_t* Kq, const uint16_t* Vq, const StreamTable& st,
                          int32_t n_heads, float scale, uint16_t* O, float* LSE, int* status,
                          float* pieces, cudaStream_t stream, int max_ctas = 0,
                          const int32_t* idx = nullptr, int d_head = kD) {
    if (d_head == 64)
        return launch_d<64>(Q, Kc, Vc, Kq, Vq, st, n_heads, scale, O, LSE, status, pieces, stream, max_ctas, idx);
    return launch_d<128>(Q, Kc, Vc, Kq, Vq, st, n_heads, scale, O, LSE, status, pieces, stream, max_ctas, idx);
}

}  // namespace attn_tc
}  // namespace pafu
