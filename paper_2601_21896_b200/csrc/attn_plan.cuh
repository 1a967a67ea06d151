// How an attention problem is handed to the CTAs: items, shares, the CTAs' walk over them, the list of split items
// for the merge, and how P is rounded.  Plain arithmetic on the host and in the kernels, without device code, so that a
// host compiler can check it.  attn_tc.cuh describes the kernel.
#pragma once
#include "common.cuh"

namespace pafu {
namespace attn_tc {

constexpr int kD = 128;
constexpr int kBM = 128;            // query rows per slot
constexpr int kBN = 64;             // keys per tile
constexpr int kMaxGrid = kMaxPersistentGrid;

struct Params {
    StreamTable st;
    int n_heads;
    int has_chunk;
    float scale;
    uint16_t* O;
    float* LSE;
    int* status;        // workspace status word (device)
    float* pieces;      // [gridDim][2][kPieceFloats]
    const int32_t* idx; // gather variant: retained token indices, stream-local, [cu_B[n_streams]]
    const uint16_t* Kraw;   // gather variant: the uncompacted cache [cu_T[n_streams], n_heads, 128]
    const uint16_t* Vraw;
    int64_t total_Lq;
    int n_waves;                       // whole-item rounds: CTA c takes items c, c + grid, ... (n_waves of them)
    int64_t rest0;                     // position of item n_waves * grid on the cost line
    int64_t share[kMaxGrid + 1];       // CTA c's share of the rest of the cost line: [rest0 + share[c], rest0 + share[c + 1])
};

// A contiguous run of key tiles [t0, t1) of one item, as seen by one CTA.
struct Seg {
    int stream, head, n_slots;
    int64_t q0;          // first query row (stream-local)
    int64_t Lq, nB, nC;  // stream's query rows, retained keys, chunk keys
    int nt1, nt, t0, t1; // tiles in the retained segment, tiles in total, this run
    int piece;           // -1: whole item (final output); 0: continues an item begun by an
                         // earlier CTA; 1: begins an item that a later CTA continues
};

constexpr int kCost2 = 8, kCost1 = 7;   // cost of one key tile with two / one live slots (with 6 the CTAs that got a
                                        // one-slot item ended 20 to 30 us after the others)

struct StreamCost {
    int64_t nqp, nt, head_cost;
    int tail_slots;
};

__host__ __device__ inline StreamCost stream_cost(const StreamTable& st, int s, int has_chunk) {
    StreamCost c;
    const int64_t lq = st.cu_Lq[s + 1] - st.cu_Lq[s];
    const int64_t nB = st.cu_B[s + 1] - st.cu_B[s];
    c.nqp = (lq + 2 * kBM - 1) / (2 * kBM);
    c.tail_slots = (lq - (c.nqp - 1) * 2 * kBM > kBM) ? 2 : 1;
    c.nt = (nB + kBN - 1) / kBN + (has_chunk ? (lq + kBN - 1) / kBN : 0);
    c.head_cost = (lq > 0) ? c.nt * (kCost2 * (c.nqp - 1) + (c.tail_slots == 2 ? kCost2 : kCost1)) : 0;
    return c;
}

__host__ __device__ inline int64_t total_cost(const StreamTable& st, int n_heads, int has_chunk) {
    int64_t t = 0;
    for (int s = 0; s < st.n_streams; ++s) t += stream_cost(st, s, has_chunk).head_cost * n_heads;
    return t;
}

// Walks the runs of one CTA: its whole items (one per round, n_waves rounds), then its share of the
// rest of the cost line.  Only the first run of that share can start inside an item (t0 > 0) and only
// its last run can stop inside one (t1 < nt).
struct SegIter {
    int64_t cur, c1;       // position on the cost line, end of the share
    int64_t item, step;    // next whole item
    int waves;             // whole items left
    __host__ __device__ SegIter(const Params& p, int cta, int n_cta, bool rest_only = false) {
        cur = p.rest0 + p.share[cta];
        c1 = p.rest0 + p.share[cta + 1];
        item = cta;
        step = n_cta;
        waves = rest_only ? 0 : p.n_waves;
    }
    __host__ __device__ static void fill(const Params& p, Seg& g, int s, const StreamCost& sc, int64_t qp) {
        g.stream = s;
        g.n_slots = qp < sc.nqp - 1 ? 2 : sc.tail_slots;
        g.q0 = qp * 2 * kBM;
        g.Lq = p.st.cu_Lq[s + 1] - p.st.cu_Lq[s];
        g.nB = p.st.cu_B[s + 1] - p.st.cu_B[s];
        g.nC = p.has_chunk ? g.Lq : 0;
        g.nt1 = (int)((g.nB + kBN - 1) / kBN);
        g.nt = (int)sc.nt;
    }
    __host__ __device__ bool next(const Params& p, Seg& g) {
        if (waves > 0) {
            int64_t i = item;
            int s = 0;
            StreamCost sc;
            for (;; ++s) {
                sc = stream_cost(p.st, s, p.has_chunk);
                const int64_t n = sc.head_cost > 0 ? sc.nqp * p.n_heads : 0;
                if (i < n) break;
                i -= n;
            }
            g.head = (int)(i / sc.nqp);
            fill(p, g, s, sc, i % sc.nqp);
            g.t0 = 0; g.t1 = g.nt; g.piece = -1;
            item += step;
            --waves;
            return true;
        }
        while (cur < c1) {
            int64_t c = cur;
            int s = 0;
            StreamCost sc;
            for (;; ++s) {
                sc = stream_cost(p.st, s, p.has_chunk);
                const int64_t tot = sc.head_cost * p.n_heads;
                if (c < tot) break;
                c -= tot;
            }
            g.head = (int)(c / sc.head_cost);
            const int64_t r = c % sc.head_cost;
            const int64_t full = sc.nt * kCost2 * (sc.nqp - 1);
            int64_t qp, rr;
            if (r < full) { qp = r / (kCost2 * sc.nt); rr = r % (kCost2 * sc.nt); }
            else { qp = sc.nqp - 1; rr = r - full; }
            fill(p, g, s, sc, qp);
            const int unit = g.n_slots == 2 ? kCost2 : kCost1;
            const int64_t item_start = cur - rr, item_end = item_start + sc.nt * unit;
            g.t0 = (int)(rr / unit);
            if (c1 >= item_end) { g.t1 = g.nt; cur = item_end; }
            else { g.t1 = (int)((c1 - item_start) / unit); cur = c1; }
            if (g.t1 > g.t0) {
                g.piece = (g.t0 == 0 && g.t1 == g.nt) ? -1 : (g.t0 > 0 ? 0 : 1);
                return true;
            }
        }
        return false;
    }
};

// Host side of the schedule.  Items go out whole, round by round, as long as no CTA exceeds its even
// share of the work: the CTAs then work on neighbouring items - a few heads - at any one time and
// their K/V tiles come from L2 instead of DRAM.  (With every CTA walking its own contiguous piece of
// the cost line, 148 different heads are read at once, far more than L2 holds: 40 heads x 4 streams
// of the 14B-class layer 6.24 -> 5.09 ms a launch, 12 heads x 18 720 keys 559 -> 530 us.)  What is left
// of the line is cut so that all CTAs end with the same total.
inline void plan_shares(Params& p, int grid, int64_t total, bool whole) {
    if (whole) {                                     // one round of whole items and nothing left
        p.n_waves = 1;
        p.rest0 = total;
        for (int b = 0; b <= grid; ++b) p.share[b] = 0;
        return;
    }
    const int64_t even = total / grid;
    int64_t done[kMaxGrid] = {}, next[kMaxGrid];
    p.n_waves = 0;
    p.rest0 = 0;
    int64_t pos = 0;
    int c = 0;
    bool fits = true;
    for (int s = 0; s < p.st.n_streams && fits; ++s) {
        const StreamCost sc = stream_cost(p.st, s, p.has_chunk);
        if (sc.head_cost == 0) continue;
        const int64_t full = sc.nt * kCost2, tail = sc.nt * (sc.tail_slots == 2 ? kCost2 : kCost1);
        for (int64_t i = 0, qp = 0; i < sc.nqp * p.n_heads; ++i) {
            const int64_t cost = qp < sc.nqp - 1 ? full : tail;
            if (++qp == sc.nqp) qp = 0;
            next[c] = done[c] + cost;
            if (next[c] > even) { fits = false; break; }
            pos += cost;
            if (++c == grid) {                       // a whole round fits
                for (int b = 0; b < grid; ++b) done[b] = next[b];
                c = 0;
                ++p.n_waves;
                p.rest0 = pos;
            }
        }
    }
    int64_t before = 0;
    for (int b = 0; b <= grid; ++b) {
        p.share[b] = total / grid * b + total % grid * b / grid - before;
        if (b < grid) before += done[b];
    }
}

struct MergeItem {
    int32_t o_row;        // row of O (and LSE column) of the item's first query
    int32_t rows;         // valid query rows of the item (<= 256)
    int16_t head, n_slots;
    int16_t first, n_pieces;   // entries [first, first + n_pieces) of MergeTable::cta
};
struct MergeTable {
    int32_t n_items;
    int32_t longest;           // most pieces of an item
    MergeItem item[kMaxGrid];
    int16_t cta[2 * kMaxGrid];
};

// ROUND: how P's rounding is kept small where that matters (round_mode() decides).
//   kRoundPlain    P as one bf16 operand, relative to the lazy running maximum
//   kRoundSplit    P as two, its rounded value and what rounding left over (the second half of the S buffer, whose
//                  logits are in registers by then)
//   kRoundOpening  as two in the tiles that open a run
constexpr int kRoundPlain = 0, kRoundSplit = 1, kRoundOpening = 2;
constexpr int kOpeningTiles = 2;

// Host side of the merge: which CTAs hold the pieces of which item.
inline void build_merge_table(const Params& p, int n_cta, MergeTable& tb) {
    tb.n_items = 0;
    tb.longest = 0;
    int n_list = 0;
    Seg g, last;
    for (int b = 0; b < n_cta; ++b) {
        bool have = false;
        {
            SegIter iter(p, b, n_cta, true);
            while (iter.next(p, g)) { last = g; have = true; }
        }
        if (!have || last.piece != 1) continue;
        MergeItem& it = tb.item[tb.n_items++];
        it.o_row = (int32_t)(p.st.cu_Lq[last.stream] + last.q0);
        const int64_t left = last.Lq - last.q0;
        it.rows = (int32_t)(left < 2 * kBM ? left : 2 * kBM);
        it.head = (int16_t)last.head;
        it.n_slots = (int16_t)last.n_slots;
        it.first = (int16_t)n_list;
        tb.cta[n_list++] = (int16_t)b;
        int t = last.t1;
        for (int c = b + 1; c < n_cta && t < last.nt; ++c) {
            SegIter iter(p, c, n_cta, true);
            if (!iter.next(p, g)) continue;    // an empty share holds no piece
            t = g.t1;
            tb.cta[n_list++] = (int16_t)c;
        }
        it.n_pieces = (int16_t)(n_list - it.first);
        if (it.n_pieces > tb.longest) tb.longest = it.n_pieces;
    }
}

inline int sm_count() { return device_sm_count(); }

// CTAs for a problem, and whether each takes one whole item (`whole`) instead of a share.
// Splitting shortens the longest CTA to its share but adds the partials' way through memory and the merge, 6 to
// 8 us together.  So a problem whose items fit on the GPU at once and whose longest item is at most three
// 64-key tiles longer than a share is not split (seven: 2 to 4 us faster on some problems of 8 to 15 tiles an item, slower on
// others), and no share is made smaller than one tile.  Before (shares down to a fraction of a tile, a
// serial merge): 2 heads x 120 queries x 8023 keys 80 us, now 20; three ragged streams of 2 heads 31.7 and 16.7;
// 2 heads x 600 queries x 2000 keys 44 and 18.
constexpr int kMergeTiles = 3, kMinShareTiles = 1;
inline int cta_limit(int max_ctas) {                         // max_ctas > 0: the caller's scratch holds fewer partials
    const int sms = sm_count();
    return max_ctas > 0 && sms > max_ctas ? max_ctas : sms;
}
inline int longest_item(const StreamTable& st, int has_chunk) {
    int64_t longest = 0;
    for (int s = 0; s < st.n_streams; ++s) {
        const StreamCost sc = stream_cost(st, s, has_chunk);
        if (sc.head_cost > 0 && sc.nt > longest) longest = sc.nt;
    }
    return (int)longest;
}
inline int grid_for(const StreamTable& st, int n_heads, int has_chunk, int64_t cost, int max_ctas, bool& whole) {
    const int sms = cta_limit(max_ctas);
    int64_t items = 0;
    for (int s = 0; s < st.n_streams; ++s) {
        const StreamCost sc = stream_cost(st, s, has_chunk);
        if (sc.head_cost > 0) items += sc.nqp * n_heads;
    }
    int64_t share = cost / ((int64_t)kCost2 * sms);
    if (share < kMinShareTiles) share = kMinShareTiles;
    whole = items <= sms && longest_item(st, has_chunk) <= share + kMergeTiles;
    if (whole) return (int)items;
    const int64_t g = (cost + kCost2 * kMinShareTiles - 1) / (kCost2 * kMinShareTiles);
    return (int)(g < sms ? g : sms);
}

// How P is rounded.  Relative to its run's running maximum a probability is rounded to bf16, a relative error of 2^-9; only
// the maximum itself is exact (1).  A problem cut into single tiles has an exact one in each, which shows on peaked
// rows (logits twice as wide as normal: error 1.76e-3 in single tiles, 2.2e-3 and more in long runs; 1.66e-3 is the output's own
// rounding).  So that leaving items whole, and shares a little longer, costs no precision, P's rounding error is carried along
//   - in every tile below kSplitShare tiles a share: 2 heads x 600 queries x 2000 keys 1.97e-3 in pieces of a tile or two, 1.66e-3;
//     18.7 us, 18.9 without it;
//   - in the two tiles that open a run below kOpeningShare, and in whole items of up to kOpeningItem tiles, where carrying it
//     everywhere would cost up to a quarter: 140 heads x 256 queries x 704 keys 2.25e-3 in pieces, 2.30e-3 whole, 2.24e-3 like this;
//     19.8 us, 18.9 without it, 40.8 in pieces.
// Longer runs show no difference: a piece more or less is a few exact probabilities among hundreds.
constexpr int kSplitShare = 5, kOpeningShare = 8, kOpeningItem = 64;
inline int round_mode(const StreamTable& st, int has_chunk, int64_t cost, int max_ctas, bool whole) {
    const int64_t tile = (int64_t)kCost2 * cta_limit(max_ctas);     // cost of a share of one tile
    if (cost < kSplitShare * tile) return kRoundSplit;
    return cost < kOpeningShare * tile || (whole && longest_item(st, has_chunk) <= kOpeningItem) ? kRoundOpening : kRoundPlain;
}

}  // namespace attn_tc
}  // namespace pafu
