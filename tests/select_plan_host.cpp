// Host harness for the selection's launch rules: plans one problem as the launchers do.  Built by test_select_plan.py with a plain
// host compiler.
#include <string.h>

#include "../paper_2601_21896_b200/csrc/select_plan.cuh"

using namespace pafu;

static StreamTable table(int n, const int64_t* T, const int64_t* B, int64_t sink, int64_t recent) {
    StreamTable st;
    memset(&st, 0, sizeof st);
    st.n_streams = n;
    for (int s = 0; s < n; ++s) {
        const int64_t b = B[s] < T[s] ? B[s] : T[s];
        st.n_recent[s] = recent < b ? recent : b;
        st.n_sink[s] = sink < b - st.n_recent[s] ? sink : b - st.n_recent[s];
        st.k[s] = b - st.n_sink[s] - st.n_recent[s];
        st.cu_T[s + 1] = st.cu_T[s] + T[s];
        st.cu_B[s + 1] = st.cu_B[s] + b;
    }
    return st;
}

// out: [small, threads, per_cta, first[0 .. n]]
extern "C" void plan_copy(int n, const int64_t* T, const int64_t* B, int64_t sink, int64_t recent, int64_t chunks, int sms, int64_t* out) {
    const SelCopyLaunch cp = plan_select_copy(table(n, T, B, sink, recent), chunks, sms);
    out[0] = cp.small; out[1] = cp.threads; out[2] = cp.per_cta;
    for (int s = 0; cp.small && s <= n; ++s) out[3 + s] = cp.shares.first[s];
}

// out: [CTAs a stream, candidates a CTA, streaming kernel too]
extern "C" void plan_selection(int n, const int64_t* T, const int64_t* B, int64_t sink, int64_t recent, int covered, int64_t* out) {
    const SelLaunch pl = plan_select(table(n, T, B, sink, recent), covered != 0);
    out[0] = pl.nc; out[1] = pl.per_cta; out[2] = pl.any_stream;
}
