// Internal declarations shared by the kernels' launchers and the C ABI layer.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include "../../include/pafu.h"

namespace pafu {

// Per-stream prefix offsets and retention parameters, passed to kernels by value.
struct StreamTable {
    int32_t n_streams;
    int64_t cu_T[PAFU_MAX_STREAMS + 1];   // cache tokens
    int64_t cu_B[PAFU_MAX_STREAMS + 1];   // retained tokens
    int64_t cu_Lq[PAFU_MAX_STREAMS + 1];  // chunk tokens
    int64_t n_sink[PAFU_MAX_STREAMS];     // clamped sink length
    int64_t n_recent[PAFU_MAX_STREAMS];   // clamped recent length
    int64_t k[PAFU_MAX_STREAMS];          // candidates to take by salience
};

// Workspace layout: [0, 256) status header (int32 words), then per-step scratch.
constexpr size_t kWsHeaderBytes = 256;
constexpr int kStatusWordTimeout = 0;   // non-zero: a bounded wait ran out
// Diagnostic counters of the tcgen05 attention kernel, one count per (softmax warp, key tile):
constexpr int kStatusWordFullFirst = 8;    // exact pass on a run's first tile or a segment's ragged last tile
constexpr int kStatusWordFullSum = 9;      // exact pass forced by a row sum that outgrew the running maximum
constexpr int kStatusWordRescale = 10;     // output accumulator and row sum rescaled in tensor memory
// Test hook: while this word is non-zero the attention kernel's loader role issues no copies, so
// every consumer's bounded wait runs out and the kernel unwinds with PAFU_ERR_TIMEOUT.
constexpr int kStatusWordStallLoader = 32;
// Work counters of the row gather inside a layer step (three words; back to zero when it ends).
constexpr int kStatusWordGatherWork = 16;

inline pafu_status cuda_ok(cudaError_t e) { return e == cudaSuccess ? PAFU_OK : PAFU_ERR_CUDA; }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// SM count of the current device (148 when no device is visible, e.g. sizing queries on a
// build host); capped so per-CTA tables stay small.
constexpr int kMaxPersistentGrid = 256;
constexpr int kMaxDevices = 64;       // per-device caches below are indexed by the CUDA device ordinal
inline int current_device() {
    int dev = 0;
    return (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices) ? dev : -1;
}
inline int device_sm_count() {
    static int n[kMaxDevices] = {};
    const int dev = current_device();
    if (dev < 0) return 148;
    if (n[dev] == 0) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
            n[dev] = v < kMaxPersistentGrid ? v : kMaxPersistentGrid;
        else
            return 148;
    }
    return n[dev];
}
// Runs `set` (the cudaFuncSetAttribute calls of one kernel family) once per device; `done` is
// that family's per-device record.  Function attributes belong to the device's context, so a
// process that uses several GPUs has to opt in on each of them.
template <typename Set>
inline bool once_per_device(bool (&done)[kMaxDevices], Set set) {
    const int dev = current_device();
    if (dev < 0) return false;
    if (!done[dev]) {
        if (!set()) return false;
        done[dev] = true;
    }
    return true;
}

// Every kernel of this library is launched with programmatic stream serialization: its CTAs
// may be scheduled, and run their local set-up, as soon as the preceding kernel's CTAs have
// left the SMs, without waiting for that kernel's completion to be processed first.  In return
// each kernel executes grid_dep_wait() before its first access to global memory; that wait
// returns only when the preceding kernel has completed and its writes are visible.  Only the
// selection and the rolling cache's row copies let their dependents start early (see there): CTAs of a following kernel that sat on the SMs while a
// bandwidth-bound kernel was still in its last wave cost more than the earlier start gained.
#ifdef __CUDACC__
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the kernel launched behind this one (as a programmatic dependent) start now; that kernel
// still sees this one's results only after its own grid_dep_wait().
__device__ __forceinline__ void grid_dep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// An index written by the kernel ahead while this one may already be running: read after
// grid_dep_wait(), and not through the read-only path (__ldg, const __restrict__), which may be used - and moved
// above the wait - only for what nothing writes during the kernel's whole lifetime.
__device__ __forceinline__ int32_t ld_index(const int32_t* p) {
    int32_t v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
#endif
// carveout >= 0: that share (per cent) of an SM's L1 and shared memory is to be shared memory while the kernel runs, so that a kernel
// with dynamic shared memory can join it.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_dependent_carveout(int carveout, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                             cudaStream_t stream, unsigned cluster_x, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[3];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 1;
    if (cluster_x > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = cluster_x;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    if (carveout >= 0) {
        attr[cfg.numAttrs].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
        attr[cfg.numAttrs].val.sharedMemCarveout = (unsigned)carveout;
        ++cfg.numAttrs;
    }
    cfg.attrs = attr;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, unsigned cluster_x, Args... args) {
    return launch_dependent_carveout(-1, kernel, grid, block, smem, stream, cluster_x, args...);
}

// Shared memory of an SM that row copies leave to a salience head beside them, a split that the hardware has; 92 KB of L1 stay.
constexpr int kHeadSmemBeside = 164 * 1024;

// Launchers (each enqueues on `stream` and returns the launch status).
// beside_predecessor = 1: the kernel runs beside the one launched before it, which must be
// launch_cache_rows (that kernel lets it start only once everything before it is complete), and ends after it.
// 2: the same, with shared memory that lets it join that kernel's blocks (launched with share_sms).
pafu_status launch_score(const pafu_head& head, const uint16_t* const* X, int n_parts, int64_t n_tokens, int64_t ldx,
                         float* scores, void* ws, size_t ws_bytes, cudaStream_t stream, int beside_predecessor = 0);
// trigger_late = 1: the kernel behind it may start early, but not before everything ahead of the
// selection is complete.  covered: work beside the selection takes longer than it, on the SMs that it leaves
pafu_status launch_select(const float* scores, const StreamTable& st, int32_t* idx,
                          cudaStream_t stream, int trigger_late = 0, bool covered = false);
// Selection and row gather of a small step in one launch; *done = false: the step is not small, nothing was launched.
pafu_status launch_select_compact(const uint16_t* K, const uint16_t* V, const float* scores, const StreamTable& st, int32_t d_model, int32_t* idx,
                                  uint16_t* Kc, uint16_t* Vc, float* SLc, cudaStream_t stream, bool* done);
int select_cta_count(const StreamTable& st, bool covered = false);      // CTAs launch_select's kernels occupy for this geometry
// work != nullptr (three zeroed words of the workspace header): the rows that are kept whatever
// the scores say are copied before the kernel waits for its predecessor (only valid when that
// predecessor is launch_select of the same step)
pafu_status launch_compact(const uint16_t* K, const uint16_t* V, const float* SL,
                           const int32_t* idx, const StreamTable& st, int32_t d_model,
                           uint16_t* Kc, uint16_t* Vc, float* SLc, cudaStream_t stream, int* work = nullptr,
                           int select_ctas = 0);
pafu_status launch_compact_layers(const uint16_t* const* K, const uint16_t* const* V, int32_t n_layers,
                                  const float* SL, const int32_t* idx, const StreamTable& st, int32_t d_model,
                                  uint16_t* const* Kc, uint16_t* const* Vc, float* SLc, cudaStream_t stream);
// The row copies of a rolling-cache update, all layers in one launch: n_new rows of Knew/Vnew to row `dst0` on of
// Kd/Vd, and rows idx[0 .. keep) of Ks/Vs (and SL) to the front of Kd/Vd (and SLd).
// select_ctas > 0: launched directly behind launch_select(.., trigger_late = 1), which occupies that many
// CTAs; 0: after what is ahead (keep must be 0).  n_new or keep may be 0, not both.
pafu_status launch_cache_rows(const uint16_t* const* Knew, const uint16_t* const* Vnew, int64_t n_new,
                              const uint16_t* const* Ks, const uint16_t* const* Vs, const float* SL, const int32_t* idx,
                              int64_t keep, int64_t dst0, uint16_t* const* Kd, uint16_t* const* Vd, float* SLd, int32_t n_layers,
                              int32_t d_model, int select_ctas, bool share_sms, cudaStream_t stream);
// Whether the salience head of n_tokens should share the SMs with row copies that take about copy_us and leave select_ctas SMs to the selection.
bool head_shares_sms(const pafu_head& head, int64_t n_tokens, double copy_us, int select_ctas);
pafu_status launch_attn(const uint16_t* Q, const uint16_t* Kc, const uint16_t* Vc,
                        const uint16_t* Kq, const uint16_t* Vq, const StreamTable& st,
                        int32_t n_heads, int32_t d_head, float scale, uint16_t* O, float* LSE,
                        void* ws, size_t ws_bytes, cudaStream_t stream);
pafu_status launch_attn_indexed(const uint16_t* Q, const uint16_t* K, const uint16_t* V, const int32_t* idx,
                                const uint16_t* Kq, const uint16_t* Vq, const StreamTable& st,
                                int32_t n_heads, float scale, uint16_t* O, float* LSE,
                                void* ws, size_t ws_bytes, cudaStream_t stream);
pafu_status launch_attn_stats(const uint16_t* Q, const uint16_t* K, const StreamTable& st, int32_t n_heads, float scale,
                              float* LSE, void* ws, cudaStream_t stream);
bool attn_indexed_supported(const StreamTable& st, int32_t d_head, bool has_chunk);
size_t attn_workspace_bytes(const StreamTable& st, int32_t n_heads, int32_t d_head);
size_t score_workspace_bytes(const pafu_head& head);

}  // namespace pafu
