// Plans of the attention kernels: how the key range of a (frame, head, query tile) is cut into items.  Arithmetic on sizes
// alone, for the host and the kernels (and for a plain C++ compiler).
#pragma once
#include <stdint.h>
#ifdef __CUDACC__
#define NFD_HD __host__ __device__ __forceinline__
#else
#define NFD_HD inline
#endif

// Division by a number that is fixed at launch, as a multiplication: exact for n < 2^32 / d.  An integer division
// costs over a hundred clocks and takes the special-function unit.
struct FastDiv {
    unsigned int d = 1, m = 0;       // m = ceil(2^32 / d); d = 1: m = 0
    void set(unsigned int v) { d = v, m = v > 1 ? (unsigned int)((0x100000000ull + v - 1) / v) : 0; }
    NFD_HD int div(int n) const {
#ifdef __CUDA_ARCH__
        return m ? (int)__umulhi((unsigned int)n, m) : n;
#else
        return m ? (int)(((uint64_t)(unsigned int)n * m) >> 32) : n;
#endif
    }
};

#define ATTN_CTA_ITEMS 2048      // items of a CTA, at most: each has a byte of shared memory (see attn_finish)
struct AttnPlan {
    int KB = 0;          // keys per block
    int BPF = 0;         // blocks per frame page
    int QT = 0;          // 128-row query tiles per frame
    int CH = 0;          // key blocks per split
    int MAXSPLIT = 0;    // splits of the longest window
    int WH = 0;          // (head, query tile) pairs of a frame whose key range is not split: the first ones
    int SP = 0;          // those whose key range is
    int NB = 0;          // key blocks of the longest window (with WH)
    FastDiv split_div, qt_div, wh_div, sp_div, ch_div, bpf_div;      // by MAXSPLIT, QT, WH, SP, CH, BPF
    // of a launch (attn_deal)
    int grid = 0, n_items = 0;       // CTAs, items
    int whole = 0, pieces = 0;       // items that are not split, and that are
    int wq = 0, wr = 0;              // whole / grid, whole % grid
    int first = 0, fq = 0, fr = 0;   // pieces that the CTAs from wr on get before all get some; that by grid - wr, and what is left
    int rq = 0, rr = 0;              // the other pieces by grid, and what is left
    NFD_HD bool dealt() const { return whole > 0; }
};

// An item of a launch: one of the `whole` ones, (frame, head, query tile) that are not split, and behind them the pieces,
// (frame, head, query tile, split).  Without whole ones CTA c takes the items c, c + grid, ...  With both, a CTA takes its
// whole ones in turn; then the pieces go first to the CTAs that have a whole item fewer than others, about as many as take the time
// of one (a piece six blocks more than it has, where several follow one another), then to all in turn.  (Dealt on in turn behind the
// whole ones, pieces went to CTAs that had one while others stood idle.  A context for 8 streams of 16 heads x 3 query tiles behind 32
// frames, 4 layers, us of a pass with whole windows, with pieces in turn, as it is: two streams 470, 530, 465; three 505, 584,
// 583; five 890, 1011, 923; six 1017, 1133, 1091; eight 1460, 1407, 1379.)
static inline void attn_deal(AttnPlan &pl, int frames, int n_sm) {
    pl.whole = frames * pl.WH, pl.pieces = frames * pl.SP * pl.MAXSPLIT;
    pl.n_items = pl.whole + pl.pieces;
    pl.grid = pl.n_items < n_sm ? pl.n_items : n_sm;
    pl.wq = pl.whole / pl.grid, pl.wr = pl.whole % pl.grid;
    const int behind = pl.grid - pl.wr, each = pl.whole ? (pl.NB + 1) / (pl.CH + 6) : 0;
    pl.first = pl.pieces < each * behind ? pl.pieces : each * behind;
    pl.fq = pl.first / behind, pl.fr = pl.first % behind;
    pl.rq = (pl.pieces - pl.first) / pl.grid, pl.rr = (pl.pieces - pl.first) % pl.grid;
}
// Item n of CTA c, and their number.
NFD_HD int attn_dealt(int c, int n, const AttnPlan &pl) {
    const int m = n - pl.wq - (c < pl.wr);
    if (m < 0) return c + n * pl.grid;
    const int b = pl.grid - pl.wr, o = c < pl.wr ? c + b : c - pl.wr;      // place of the CTA in a round of pieces
    const int own = c < pl.wr ? 0 : pl.fq + (o < pl.fr);
    return pl.whole + (m < own ? o + m * b : pl.first + o + (m - own) * pl.grid);
}
NFD_HD int attn_dealt_count(int c, const AttnPlan &pl) {
    const int o = c < pl.wr ? c + pl.grid - pl.wr : c - pl.wr;
    return pl.wq + (c < pl.wr) + (c < pl.wr ? 0 : pl.fq + (o < pl.fr)) + pl.rq + (o < pl.rr);
}
// What an item is: frame j of the pass, (head, query tile) t of it, split; number of its query tile among those that are split.
struct AttnPlace {
    int j, t, split, tile;
    bool whole;
};
template <bool DEALT> NFD_HD AttnPlace attn_place(int item, const AttnPlan &pl) {
    AttnPlace p;
    p.whole = DEALT && item < pl.whole;
    if (p.whole) {
        p.j = pl.wh_div.div(item), p.t = item - p.j * pl.WH;
        p.split = p.tile = 0;
    } else {
        if (DEALT) item -= pl.whole;
        p.tile = pl.split_div.div(item), p.split = item - p.tile * pl.MAXSPLIT;
        p.j = pl.sp_div.div(p.tile), p.t = p.tile - p.j * pl.SP;
        if (DEALT) p.t += pl.WH;
    }
    return p;
}

// Key block, blocks per page and query tiles for pages of T tokens: the block that walks a page in the least time, a
// block costing its columns (padded ones included) plus a fixed part of about 24 columns (barriers and hand-overs).
static void attn_blocks(AttnPlan &pl, int T) {
    const int kbs[4] = {128, 112, 96, 64};
    for (int kb : kbs) {
        const int bpf = (T + kb - 1) / kb;
        if (!pl.KB || bpf * (kb + 24) < pl.BPF * (pl.KB + 24)) pl.KB = kb, pl.BPF = bpf;
    }
    pl.QT = (T + 127) / 128;
}
// The plan's divisors; false where a dividend is too large for them (n * d has to stay below 2^32) or a CTA would get more
// items than it keeps account of.
static bool attn_divisors(AttnPlan &pl, int n_frames, int W, int n_sm) {
    pl.split_div.set(pl.MAXSPLIT), pl.qt_div.set(pl.QT), pl.ch_div.set(pl.CH), pl.bpf_div.set(pl.BPF);
    pl.wh_div.set(pl.WH > 0 ? pl.WH : 1), pl.sp_div.set(pl.SP > 0 ? pl.SP : 1);
    const long long nb = ((long long)W + 1) * pl.BPF + pl.CH, big = 0x100000000ll;
    const long long n_items = n_frames * (pl.WH + (long long)pl.SP * pl.MAXSPLIT);
    const int tiles = pl.WH + pl.SP, d_item = tiles > pl.MAXSPLIT ? tiles : pl.MAXSPLIT;
    // (with whole items and pieces a CTA may get ten items more than its share: attn_deal)
    const int cta_items = pl.WH > 0 ? ATTN_CTA_ITEMS - 16 : ATTN_CTA_ITEMS;
    return n_items <= (long long)cta_items * n_sm && n_items * d_item < big && nb < 0x7fffffffll && nb * (pl.CH > pl.BPF ? pl.CH : pl.BPF) < big;
}
// Pieces of the key range of a call on the caller's pages: as many as pay (as in attn_split_plan; starting a cluster and the merge
// through distributed shared memory take 2 us and 0.2 per piece) and as clusters of that size fit the machine at once.  Head
// dimension 64, us of whole windows and in pieces, on the device: 30 heads x 40 tokens, 8 blocks of 64 keys 10.8, 11.3, 12 blocks
// 12.6, 11.8; 8 x 96 tokens, 6 blocks of 96 10.7, 11.2, 10 blocks 12.7, 11.9; 8 x 336, 12 blocks of 112 15.3, 13.1.
// clusters(k): clusters of k CTAs that the machine holds.  (Clusters of 1 to 8 are 148, 74, 45, 33, 26, 22, 15, 15 on a 148-SM B200,
// which no formula gives: by SMs / k - 4 there would be 17 of seven, and 2 heads x 64, 8 x 40 queries behind 32 frames, 16 query
// tiles, took 25.3 -> 27.2 us in two rounds of them.)
template <typename F> static void attn_own_plan(AttnPlan &pl, int tiles, int n_blocks, F clusters) {
    float best = 1e30f;
    int best_k = 1;
    for (int k = 1; k <= 8 && k <= n_blocks; ++k) {
        const int ch = (n_blocks + k - 1) / k;
        if (k > 1 && ((n_blocks + ch - 1) / ch != k || tiles > clusters(k))) continue;
        const float t = ch * 0.65f * (pl.KB + 24) / 136.f + (k > 1 ? 2.0f + 0.2f * k : 0.f);
        if (t < best) best = t, best_k = k;
    }
    pl.CH = (n_blocks + best_k - 1) / best_k, pl.MAXSPLIT = best_k;
}
// How the key ranges of a frame's `tiles` (head, query tile) pairs are split.  By the configuration alone (the longest
// window, as many frames as there are streams), never by the pass: the order of the sums must not depend on it.
//   One stream: all of them, into at most as many pieces as fill the SMs once, and no more than pay: a block takes about 0.65 us
// (of 112 keys; its columns and 24 count), publishing and counting 2.5, the merge 0.25 per piece.  (A frame of a model of 2 layers,
// 4 heads, 64 tokens: behind four frames five pieces of a block 286 us, one of five 270; behind 30 frames 31 pieces 443, eight 300.)
//   Several: whole windows, dealt out to the CTAs, may leave a last round in which most SMs idle (16 heads
// x 3 query tiles x 8 streams = 384 items on 148 SMs: two rounds and six tenths of one, at the price of three).  Splitting all
// of them finely costs a state of 33 KB each; so the first WH are left whole and the others split, for the least blocks on the
// busiest CTA of a pass with a frame of every stream, a whole item counted a block more than it has and a piece two and a half (start,
// publication, merge).  Eight pieces to a window are looked at; where that is the best, of all windows, half of the SMs idle all the
// same and a piece has more than sixteen blocks, as long as starting and merging it take, the rule for one stream holds (two streams of
// 4 heads x 32 behind 1000 frames, eight pieces a tile 766 us a frame step, eighteen 619).
//   A pass with fewer frames than streams may take longer than with whole windows (see attn_deal for both sides): a plan that
// did not let it would be another order of the sums.
static void attn_split_plan(AttnPlan &pl, int tiles, int n_streams, int n_blocks, int n_sm) {
    auto pieces = [&](int k) { pl.CH = (n_blocks + k - 1) / k, pl.MAXSPLIT = (n_blocks + pl.CH - 1) / pl.CH; };
    pl.WH = 0, pl.SP = tiles, pl.NB = n_blocks;
    const long long items = (long long)n_streams * tiles;
    float best = 1e30f;
    int best_k = 1, best_wh = 0;
    for (int k = 1; n_streams > 1 && k <= 8 && k <= n_blocks; ++k) {
        pieces(k);
        for (int wh = k == 1 ? tiles : 0; wh <= (k == 1 ? tiles : tiles - 1); ++wh) {
            const int nw = n_streams * wh, n = nw + n_streams * (tiles - wh) * pl.MAXSPLIT, grid = n < n_sm ? n : n_sm;
            // the CTAs before, between and behind those with a whole item and with an item more than others
            float most = 0.f;
            const int at[3] = {0, nw % grid, n % grid};
            for (int c : at) {
                const int w = nw / grid + (c < nw % grid), all = n / grid + (c < n % grid);
                const float t = w * (n_blocks + 1.f) + (all - w) * (pl.CH + 2.5f);
                if (t > most) most = t;
            }
            if (most < best) best = most, best_k = k, best_wh = k == 1 ? 0 : wh;      // (none is split: MAXSPLIT 1)
        }
    }
    if (n_streams == 1 || (best_k == 8 && best_wh == 0 && 16 * items <= n_sm && n_blocks > 128)) {
        best = 1e30f;
        for (int k = n_streams == 1 ? 1 : 8; k <= n_blocks && (k == 1 || k * items <= n_sm); ++k) {
            pieces(k);
            const float t = pl.CH * 0.65f * (pl.KB + 24) / 136.f + (k > 1 ? 2.5f + 0.25f * k : 0.f);
            if (t < best) best = t, best_k = k;
        }
    }
    pieces(best_k);
    pl.WH = best_wh, pl.SP = tiles - best_wh;
}
