// Host harness for the attention kernels' schedule: plans one problem as the launcher does and writes down what every
// CTA would walk and what the merge would be told.  Built by test_attn_plan.py with a plain host compiler.
#include <string.h>

#include "../paper_2601_21896_b200/csrc/attn_plan.cuh"

using namespace pafu;
using namespace pafu::attn_tc;

// out: [grid, whole, n_waves, mode, n_items, longest], then per run {cta, stream, head, q0, slots, t0, t1, nt, piece} after its
// count, then per merged item {o_row, rows, head, n_pieces, cta...} after their count.  Returns the words written, or -1.
extern "C" int64_t attn_plan(int n, const int64_t* cu_B, const int64_t* cu_Lq, int heads, int has_chunk, int max_ctas, int64_t* out,
                             int64_t cap) {
    static Params p;
    static MergeTable tb;
    p = Params();
    p.st.n_streams = n;
    p.n_heads = heads;
    p.has_chunk = has_chunk;
    for (int s = 0; s <= n; ++s) { p.st.cu_B[s] = cu_B[s]; p.st.cu_Lq[s] = cu_Lq[s]; }
    const int64_t cost = total_cost(p.st, heads, has_chunk);
    bool whole;
    const int grid = grid_for(p.st, heads, has_chunk, cost, max_ctas, whole);
    plan_shares(p, grid, cost, whole);
    memset(&tb, 0, sizeof tb);
    if (grid > 1) build_merge_table(p, grid, tb);
    int64_t w = 0;
    auto put = [&](int64_t v) { if (w < cap) out[w] = v; ++w; };
    put(grid); put(whole); put(p.n_waves); put(round_mode(p.st, has_chunk, cost, max_ctas, whole)); put(tb.n_items); put(tb.longest);
    const int64_t at = w;
    put(0);
    int64_t runs = 0;
    for (int c = 0; c < grid; ++c) {
        SegIter it(p, c, grid);
        Seg g;
        while (it.next(p, g)) {
            for (int64_t v : {(int64_t)c, (int64_t)g.stream, (int64_t)g.head, g.q0, (int64_t)g.n_slots, (int64_t)g.t0, (int64_t)g.t1, (int64_t)g.nt, (int64_t)g.piece}) put(v);
            ++runs;
        }
    }
    if (at < cap) out[at] = runs;
    put(tb.n_items);
    for (int i = 0; i < tb.n_items; ++i) {
        const MergeItem& m = tb.item[i];
        put(m.o_row); put(m.rows); put(m.head); put(m.n_pieces);
        for (int j = 0; j < m.n_pieces; ++j) put(tb.cta[m.first + j]);
    }
    return w <= cap ? w : -1;
}
