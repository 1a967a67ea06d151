// Row log-sum-exps of the attention over one key segment, without its output (d_head = 128):
//   LSE[n, i] = log sum_j exp(scale q_i . k_j),  j over all kept keys of the stream
// - the row statistics that the salience target (Sec. 3.2, Eq. 4) subtracts in the exponent.
//
// The result is bit-identical to the LSE that attn_tc_kernel writes: same items, shares, 64-key
// tiles, running maximum per 32-row group and order of the sums, and the same merge.  What falls
// away is the P V half of the tensor work, the V tiles, P's conversion and its way through tensor
// memory.  Without the output accumulators each slot has four S buffers, handed back as soon as
// their logits are in registers, so Q K^T runs ahead and the exponentials set the pace (128 of them
// per scheduler and tile pair are 1024 clocks; Q K^T takes 768).
//
// Warp roles (384 threads): 0-3 and 4-7 exponentials and sums of slot 0 and 1 (thread = query
// row), 8 and 10 issue the MMAs of slot 0 and 1, 9 loads Q and 64-key K tiles, 11 idle.
// Every mbarrier wait is bounded.
#pragma once
#include "attn_tc.cuh"

namespace pafu {
namespace attn_tc {

constexpr int kStatsBufs = 4;
constexpr int kStatsStages = 9;
constexpr int kStatsSmemBytes = 2 * kQBytes + kStatsStages * kTileBytes + 1024 /*align*/ + 512 /*barriers*/;

__global__ void __launch_bounds__(kThreads, 1)
attn_stats_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK, const __grid_constant__ Params p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sQ = smem_u32(smem);                       // 2 slots x 32 KiB
    const uint32_t sK = sQ + 2 * kQBytes;                     // ring
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + 2 * kQBytes + kStatsStages * kTileBytes);
    const uint32_t bar0 = smem_u32(bars);
    auto q_full = [&](int s) { return bar0 + 8 * (0 + s); };
    auto q_empty = [&](int s) { return bar0 + 8 * (2 + s); };
    auto s_full = [&](int s, int b) { return bar0 + 8 * (4 + kStatsBufs * s + b); };
    auto s_empty = [&](int s, int b) { return bar0 + 8 * (4 + 2 * kStatsBufs + kStatsBufs * s + b); };
    auto k_full = [&](int st) { return bar0 + 8 * (4 + 4 * kStatsBufs + st); };
    auto k_empty = [&](int st) { return bar0 + 8 * (4 + 4 * kStatsBufs + kStatsStages + st); };
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(q_full(s), 1); mbar_init(q_empty(s), 1);
            for (int b = 0; b < kStatsBufs; ++b) { mbar_init(s_full(s, b), 1); mbar_init(s_empty(s, b), 4); }
        }
        for (int st = 0; st < kStatsStages; ++st) { mbar_init(k_full(st), 1); mbar_init(k_empty(st), 2); }
        abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 8) { tmem_alloc(smem_u32(&tmem_base_sh), 512); tmem_relinquish(); }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base_sh, 0);
    grid_dep_wait();

    auto fail = [&](int code) {
        abort_flag = 1;
        atomicCAS(p.status, 0, code);
    };

    if (warp == 9) {
        // ---------------------------------------------------------------------- TMA loader
        if (elect_one() && p.status[kStatusWordStallLoader] == 0) {
            prefetch_tmap(&mQ); prefetch_tmap(&mK);
            SegIter iter(p, blockIdx.x, gridDim.x);
            Seg g;
            uint32_t ring = 0, qc0 = 0, qc1 = 0;
            bool ok = true;
            while (ok && iter.next(p, g)) {
                const int qrow = (int)(p.st.cu_Lq[g.stream] + g.q0);
                for (int s = 0; s < g.n_slots && ok; ++s) {
                    const uint32_t qc = s ? qc1 : qc0;
                    if (abort_flag || !mbar_wait(q_empty(s), (qc & 1u) ^ 1u)) { fail(700); ok = false; break; }
                    if (s) ++qc1; else ++qc0;
                    mbar_arrive_expect_tx(q_full(s), kQBytes);
                    tma_load_3d(sQ + s * kQBytes, &mQ, q_full(s), 0, g.head, qrow + s * kBM);
                    tma_load_3d(sQ + s * kQBytes + kQHalf, &mQ, q_full(s), 64, g.head, qrow + s * kBM);
                }
                for (int j = g.t0; j < g.t1 && ok; ++j, ++ring) {
                    const int st = ring % kStatsStages, row = (int)(p.st.cu_B[g.stream] + (int64_t)j * kBN);
                    if (abort_flag || !mbar_wait(k_empty(st), ((ring / kStatsStages) & 1u) ^ 1u)) { fail(701); ok = false; break; }
                    mbar_arrive_expect_tx(k_full(st), kTileBytes);
                    tma_load_3d(sK + st * kTileBytes, &mK, k_full(st), 0, g.head, row);
                    tma_load_3d(sK + st * kTileBytes + kHalfBytes, &mK, k_full(st), 64, g.head, row);
                }
            }
            if (!ok) {     // let copies already in flight land before the CTA exits
                for (uint32_t r = ring > (uint32_t)kStatsStages ? ring - kStatsStages : 0; r < ring; ++r)
                    mbar_wait(k_full(r % kStatsStages), (r / kStatsStages) & 1u);
                if (qc0 > 0) mbar_wait(q_full(0), (qc0 - 1) & 1u);
                if (qc1 > 0) mbar_wait(q_full(1), (qc1 - 1) & 1u);
            }
        }
        __syncwarp();
    } else if (warp == 8 || warp == 10) {
        // -------------------------------------------------------- MMA issuers (warp-uniform loops)
        const int slot = warp == 8 ? 0 : 1;
        const uint32_t idesc = make_idesc_bf16(kBM, kBN, false, false);
        const uint64_t desc = make_smem_desc_sw128(0, 16, 1024);
        const uint32_t hi = (uint32_t)(desc >> 32), lo_q = (uint32_t)desc + ((sQ + slot * kQBytes) >> 4), lo_k = (uint32_t)desc + (sK >> 4);
        uint32_t st = 0, ph = 0, qcnt = 0, tc = 0;                // tc: tiles this slot has processed so far
        bool ok = true;
        auto wait = [&](uint32_t bar, uint32_t parity, int code) {
            if (ok && !mbar_wait_warp(bar, parity)) { if (lane == 0) fail(code); ok = false; }
        };
        SegIter iter(p, blockIdx.x, gridDim.x);
        Seg g;
        while (ok && iter.next(p, g)) {
            const int n = __shfl_sync(0xffffffffu, g.t1 - g.t0, 0);
            const bool live = slot < __shfl_sync(0xffffffffu, g.n_slots, 0);
            if (live) wait(q_full(slot), qcnt++ & 1u, 711);
#pragma unroll 1
            for (int i = 0; i < n && ok; ++i) {
                wait(k_full(st), ph, 712);
                if (live) {
                    const int buf = tc % kStatsBufs;
                    wait(s_empty(slot, buf), ((tc / kStatsBufs) & 1u) ^ 1u, 713);
                    if (!ok) break;
                    ++tc;
                    tc_fence_after_sync();
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        umma_ss_x4(tmem + (slot * kStatsBufs + buf) * kBN, lo_q + c * (kQHalf >> 4),
                                   lo_k + ((st * kTileBytes + c * kHalfBytes) >> 4), idesc, hi, c);
                    elect_commit(s_full(slot, buf));
                    elect_commit(k_empty(st));
                } else if (ok) {
                    elect_arrive(k_empty(st));               // a stage is released by both issuers
                }
                if (++st == (uint32_t)kStatsStages) { st = 0; ph ^= 1u; }
            }
            if (ok && live) elect_commit(q_empty(slot));
        }
    } else if (warp < 8) {
        // --------------------------------------------- exponentials and sums, as attn_tc_kernel forms them
        const int slot = warp >> 2;
        const uint32_t tSslot = tmem + slot * (kStatsBufs * kBN) + (((uint32_t)((warp & 3) * 32)) << 16);
        const float sl2 = p.scale * 1.4426950408889634f;
        const uint64_t sl2_2 = pack2(__float_as_uint(sl2), __float_as_uint(sl2));
        SegIter iter(p, blockIdx.x, gridDim.x);
        Seg g;
        uint32_t tc = 0;
        bool ok = true;
        while (ok && iter.next(p, g)) {
            if (slot >= g.n_slots) continue;
            float m_used = -INFINITY, l_sum = 0.f;
            const int n = g.t1 - g.t0;
            const int rag = (g.nB % kBN) != 0 ? g.nt - 1 - g.t0 : -1, lim = (int)(g.nB % kBN);   // the segment's ragged last tile
#pragma unroll 1
            for (int i = 0; i < n; ++i, ++tc) {
                const int buf = tc % kStatsBufs;
                const uint32_t tS = tSslot + buf * kBN;
                if (!mbar_wait_warp(s_full(slot, buf), (tc / kStatsBufs) & 1u)) { if (lane == 0) fail(721); ok = false; break; }
                tc_fence_after_sync();
                uint32_t sr[64];
                PAFU_TMEM_LD_X32(tS, sr);
                PAFU_TMEM_LD_X32(tS + 32, sr + 32);
                tmem_wait_ld();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(s_empty(slot, buf));
                const int left = i == rag ? lim : kBN;
                bool full_pass = (i == 0) || (left < kBN);
                if (!full_pass) {
                    const float rs = tile_sum(sr, sl2_2, -m_used * sl2);
                    full_pass = __any_sync(0xffffffffu, !(rs < kSumTrigger));    // also true for inf / NaN
                    if (!full_pass) l_sum += rs;
                } else if (left < kBN) {
#pragma unroll
                    for (int c = 0; c < kBN; ++c)
                        if (c >= left) sr[c] = 0xff800000u;   // -inf
                }
                if (full_pass) {
                    const float mx = tile_max(sr);
                    if (i == 0) {
                        m_used = mx;
                    } else if (__any_sync(0xffffffffu, (mx - m_used) * sl2 > kRescaleThresholdLog2)) {
                        const float m_new = fmaxf(m_used, mx);
                        l_sum = __fmul_rn(l_sum, fast_exp2((m_used - m_new) * sl2));
                        m_used = m_new;
                    }
                    l_sum += tile_sum(sr, sl2_2, -m_used * sl2);
                }
            }
            if (!ok) break;
            const int64_t row = g.q0 + slot * kBM + (tid & 127);
            if (g.piece < 0) {
                if (row < g.Lq)
                    p.LSE[(int64_t)g.head * p.total_Lq + p.st.cu_Lq[g.stream] + row] = final_lse(m_used, p.scale, l_sum);
            } else {
                float* piece = p.pieces + ((size_t)blockIdx.x * 2 + g.piece) * kPieceFloats;
                const int prow = slot * kBM + (tid & 127);
                piece[2 * kBM * kD + prow] = m_used;
                piece[2 * kBM * kD + 2 * kBM + prow] = l_sum;
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tmem, 512);
}

// Q [cu_Lq], K [cu_B] tokens; `pieces` as for the attention kernel.
inline pafu_status launch_stats(const uint16_t* Q, const uint16_t* K, const StreamTable& st, int32_t n_heads, float scale,
                                float* LSE, int* status, float* pieces, cudaStream_t stream) {
    const int n = st.n_streams;
    const int64_t cost = total_cost(st, n_heads, 0);
    if (cost == 0) return PAFU_OK;
    CUtensorMap mQ, mK;
    if (!TmapEncoder::token_tensor(&mQ, Q, (uint64_t)st.cu_Lq[n], n_heads, kD, kBM) ||
        !TmapEncoder::token_tensor(&mK, K, (uint64_t)st.cu_B[n], n_heads, kD, kBN)) return PAFU_ERR_CUDA;
    Params p = {};
    p.st = st; p.n_heads = n_heads; p.scale = scale; p.LSE = LSE; p.status = status; p.pieces = pieces; p.total_Lq = st.cu_Lq[n];
    static bool attr_set[kMaxDevices] = {};
    if (!once_per_device(attr_set, [] {
            return cudaFuncSetAttribute(attn_stats_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kStatsSmemBytes) == cudaSuccess;
        }))
        return PAFU_ERR_CUDA;
    bool whole;
    const int grid = grid_for(st, n_heads, 0, cost, 0, whole);
    plan_shares(p, grid, cost, whole);
    if (launch_dependent(attn_stats_kernel, dim3(grid), dim3(kThreads), kStatsSmemBytes, stream, 1, mQ, mK, p) != cudaSuccess)
        return PAFU_ERR_CUDA;
    return launch_merge<kD, false>(p, grid, n_heads, stream);
}

}  // namespace attn_tc
}  // namespace pafu
