// Salience head launcher (the kernel is in score_tc.cuh).
#include "common.cuh"
#include "score_tc.cuh"

namespace pafu {

size_t score_workspace_bytes(const pafu_head&) { return 0; }

pafu_status launch_score(const pafu_head& head, const uint16_t* const* X, int n_parts, int64_t n_tokens, int64_t ldx,
                         float* scores, void* ws, size_t, cudaStream_t stream, int beside_predecessor) {
    if (n_tokens == 0) return PAFU_OK;
    return score_tc::launch(head, X, n_parts, n_tokens, ldx, scores,
                            reinterpret_cast<int*>(ws) + kStatusWordTimeout, device_sm_count(), stream, beside_predecessor);
}

// Row copies leave the head no room: they run with the largest L1, and an SM's split changes only when it is idle, so
// the head starts where they end.  With 164 KB of shared memory set aside it joins them, but their bytes in flight pass
// through what is left of the L1, and long copies lose more (up to a twentieth) than the head takes.  So they share while the copies
// take at most kSharePerSlice us for each of the head's reduction slices, of which it needs 0.45 to 1.1 us: 11 layers of 16 heads,
// 2300 + 700 tokens 126.7 -> 97.3 us; 10 x 12, 4000 + 2000 148.7 -> 127.6; 8 x 12, 4680 + 4680 209.9 -> 198.4; 30 x 6, 2500 + 1500 135.4 -> 124.4.
// Beyond: 15 x 12, 4680 + 4680 329.6 and 328; 20 x 12 415 and 420; 30 x 12 587 and 607; 25 x 12, 13 000 + 1000 676 and 716.  (With 196 KB set aside,
// which a share of 72 % gives, the first four took 99.9, 131.7, 201 and 128.3.)  Heads of few slices do not share; that line was drawn with
// 196 KB, 10 layers of 2 heads, 5000 + 4000 56.1 us and 58.7; with 164 KB it is 46.4 and 37.7.
// A head of few CTAs runs on the SMs that the copies leave to the selection: 128 tokens, 16 hidden units (one CTA) beside 20 layers of 12
// heads, 4000 tokens, 173 us sharing, 159 so; four CTAs beside 6 layers, 12 000 tokens, 162.6 and 151.3.
bool head_shares_sms(const pafu_head& head, int64_t n_tokens, double copy_us, int select_ctas) {
    constexpr double kSharePerSlice = 3.5;
    constexpr int kShareSlices = 24;
    const int slices = head.d_in / score_tc::kBK;
    if (score_tc::plan(head, n_tokens, device_sm_count()).grid <= select_ctas) return false;
    return slices >= kShareSlices && copy_us <= kSharePerSlice * slices;
}

}  // namespace pafu
