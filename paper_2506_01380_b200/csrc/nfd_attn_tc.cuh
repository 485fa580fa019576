// Block-wise causal flash attention on tcgen05 / TMEM (bf16, head_dim 64, or 32 padded with zeros by TMA).
//
// Work item = (frame of the pass, head, 128-row query tile, split of the key
// range).  The keys of a query frame are the frame pages win_first..frame of the
// ring cache, walked in blocks of KB keys; a block never straddles a page (the
// last block of a page is masked where KB does not divide the tokens per frame),
// so the frame-granular mask is a page range and needs no test per element.  Per block:
//     S  = Q K^T          UMMA 128 x KB x 64, operands in shared memory (TMA),
//                         accumulator in tensor memory
//     P  = exp2(S*c - m)  one thread per query row: TMEM -> registers, running
//                         sum, P written back to tensor memory as the sum of two
//                         bf16 numbers, over the S columns it came from
//     O += P V            two UMMAs 128 x 64 x KB, P read from tensor memory, V used
//                         straight from its page (MN-major B operand in shared
//                         memory), accumulated in tensor memory
// The second number of P keeps what rounding to bf16 leaves (2^-17 of P at most is lost), so that the error of the result
// is that of its own rounding to bf16: 1.66e-3 (2-norm) for normal data, as with fp32 probabilities.  With the first
// number alone it was 2.33e-3 whatever the data; the product doubles and a block takes about 200 clocks more (16 heads
// x 64, 336 tokens: one frame 23.0 -> 25.0 us, two 37.3 -> 40.9, four 64.2 -> 70.7, eight streams 181 -> 210).
// The reference m of a row is the largest of the first 16 scores of the item and is never changed: a probability is
// exact to the same number of bits whatever its size, so that m only has to keep exp2 in range.  With no maximum to take
// there is no state to rescale, and all softmax groups share one m and one O accumulator.  Should a block's sum of a
// row pass 2^100 (scores rising by more than 69 nats over the first ones), all of its first scores be -inf, or O leave fp32,
// the item is walked twice more when the CTA is through with its items: once for the true maxima of its rows and once with
// these as m (attn_again).  No data takes more than three times as long, and no wait is any longer.
// No barrier joins the groups at the end of an item: m, found by the group of the first block, and the sums go through shared
// memory and barriers of their own, two items deep, and the group of an item's last block reads O and finishes the item while
// the others go on (groups 0 and 1 share a CTA's last item).
//
// Warps 0 and 3 = TMA producers (K, V), warp 1 = issuer of all products (and loader of Q), warps 4-15 = three softmax
// groups of four warps; group g takes the CTA's blocks n with
// n % 3 == g.  A softmax warp is a chain of tensor-memory loads, FMAs, exponentials and conversions: with two groups the
// schedulers issued in 42 % of the clocks.
// S has NS accumulators in tensor memory, the CTA's n-th block using number n % NS (and a "P is stored" barrier of its
// own: a warp of a group may be a whole block ahead of another).  S(n + NS) is issued right behind P V(n), which reads P(n)
// from that accumulator: the tensor pipe takes one thread's instructions in order.  (With an issuer for each product
// S(n + NS) had to wait for the completion of P V(n): 1000 clocks a block, four accumulators against 2050 clocks of
// softmax and 1900 of hand-overs.)  A group finds its next S ready when it comes back for it.  K blocks go through a
// ring of NS stages (free again when S(n) is complete, which the barrier of accumulator n % NS tells), V blocks through
// one of NS (free when P V is complete); V(n) and K(n + NS), which the issuer needs at the same time, arrive on one barrier.
//
// What bounds it: the turn of an accumulator, S -> softmax -> P V, and in it the softmax warps (exponentials: 896 clocks per
// 128 x 112 block on the special-function unit) and the one issuer (18 products, 29 to 60 clocks each, and their barriers); a
// block takes about 1300 clocks.  Registers and code size count: spilled registers are cold local memory, about 1 us on the
// path of a short item, and a cold code path costs as much.
// Measured, 16 heads x 64 on one B200 (events around a launch), one, two and four frames of 336 tokens behind 16: 25.0, 39.3,
// 65.6 us (25.0, 40.8, 71.8 with pieces merged as their items end).  How it came there, with P rounded to bf16 and a quarter of
// the exponentials by a polynomial on the FMA pipe: one frame 28.4 with one thread for all loads, one for all products and a
// maximum pass over S; 25.0 with the threads split and no maximum pass; 23.0 with three groups; 22.5 with items that overlap
// and the issuer's loop in one copy (then 35.2, 61 and, eight streams behind 32 frames, 165 for the others).  The polynomial's range reduction saturated,
// which gave the score NaN a probability of nought; with every exponential the special-function unit's 23.0, 37.3, 64.2, 181.
// With P as two numbers the polynomial gains nothing (24.9, 39.4, 69.5, 210 with an eighth of the exponentials, 25.0, 39.9,
// 70.2, 207 without).  Pages of 220 tokens behind nine frames: 17 us (plain kernel: 800).
// Tried and worse: sixteen softmax warps with half a row each (178 -> 201: the fixed part of a block doubles); four epilogue
// warps beside the groups (96 registers a thread: four frames 60, but 2 us more on every short launch).
//
// The grid is persistent: a CTA takes items blockIdx.x, + gridDim.x, ..., or those that attn_deal gives it; producers and
// issuer run ahead into the next item.  A key range
// longer than CH blocks is split over several items; each publishes its
// unnormalised (O, m, l) state in global memory, stored so that a warp writes and reads
// whole lines.  When a CTA is through with all its items, one warp counts it in at each of
// them (a counter per query tile) and all its warps merge, in split order, those for which
// it is the last (attn_merge).  CH depends only on the configuration, so
// a frame's result does not depend on which other frames share its pass.  In a context of
// several streams some (head, query tile) pairs are not split: attn_split_plan.
#pragma once
#include "nfd_sm100.cuh"

// A published state: [16 groups of 4 columns][128 rows] float4, then [2 halves of O][128 rows] (m, l).
#define ATTN_STATE_BYTES (128 * 64 * 4 + 2 * 128 * 8)
// Flags that are read when all roles are through: an item is marked, a wait has run out.  (In registers, with a vote at the
// end, they cost two frames 39.6 -> 41.5 us.)
#define ATTN_MARKED 1u
#define ATTN_EXPIRED 2u

template <int KB> struct AttnCfg {
    static constexpr int NS = KB <= 112 ? 4 : 3;           // S accumulators = stages of the K and the V ring
    static constexpr int NGRP = 3;                         // softmax groups
    static constexpr int Q_BYTES = 128 * 128;              // two of them
    static constexpr int KV_BYTES = KB * 128;              // one K (or V) block
    static constexpr int ML_BYTES = (2 * (1 + NGRP) + 1) * 128 * 4;   // m of every row, l of every row and group, two items; maxima
    static constexpr int SMEM = 2 * Q_BYTES + 2 * NS * KV_BYTES + ML_BYTES + 8 + ATTN_CTA_ITEMS + 256 + 1024;
    // behind the rest, from the 1024-byte boundary that AttnShared starts at: the CTA's state (k_attn_own), or its items
    static constexpr int STATE_AT = (SMEM - 1024 + 127) / 128 * 128, OWN_SMEM = 1024 + STATE_AT + ATTN_STATE_BYTES,
                         DEALT_SMEM = 1024 + STATE_AT + 4 * ATTN_CTA_ITEMS;
    static constexpr int TMEM_COLS = 512;
    static constexpr int S_STRIDE = KB <= 112 ? 112 : 128; // S accumulators from column 0, O at column 448
    static constexpr int TM_O = 448;
    static constexpr int SM_WARP0 = 4;                     // first softmax warp
    static constexpr int THREADS = 32 * (SM_WARP0 + 4 * NGRP);
    static_assert(THREADS == 512, "attn_merge: a warp per quarter of the columns and quadrant of the rows");
    static_assert(KB % 16 == 0 && KB <= 128 && NS * S_STRIDE <= TM_O, "key block");
    static_assert(SMEM <= 232448 && OWN_SMEM <= 232448 && DEALT_SMEM <= 232448, "shared memory of a CTA");
    static_assert(STATE_AT % 16 == 0 && ATTN_STATE_BYTES % 16 == 0, "states are read and written in 16-byte words");
};

__host__ __device__ constexpr uint32_t umma_idesc_bf16_bmn(int M, int N) {
    return umma_idesc_bf16(M, N) | (1u << 16);             // B operand MN-major
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// p as a sum of two bf16 numbers: hi = p rounded, lo = what that leaves, rounded (2^-17 of p at most is lost), as
// packed pairs.  The subtraction takes hi as it is packed (fma with a bf16 factor).
__device__ __forceinline__ void bf16_split2(float2 p, uint32_t &hi, uint32_t &lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(p.x, p.y);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    float2 d;
    asm("{\n"
        ".reg .b16 a, b, m1;\n"
        "mov.b32 {a, b}, %2;\n"
        "mov.b16 m1, 0xBF80;\n"                            // -1
        "fma.rn.f32.bf16 %0, a, m1, %3;\n"
        "fma.rn.f32.bf16 %1, b, m1, %4;\n"
        "}\n"
        : "=f"(d.x), "=f"(d.y)
        : "r"(hi), "f"(p.x), "f"(p.y));
    const __nv_bfloat162 l = __floats2bfloat162_rn(d.x, d.y);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}
// add 1 with release and acquire semantics at device scope
__device__ __forceinline__ unsigned int atomic_inc_acq_rel(unsigned int *p) {
    unsigned int v;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// One item of the grid.  A CTA's items are numbered from attn_first<DEALT>() on in steps of attn_step<DEALT>(): by themselves, or, in a
// launch that deals them out, by their places in a table of the CTA's.
template <bool DEALT> __device__ __forceinline__ int attn_first() { return DEALT ? 0 : blockIdx.x; }
template <bool DEALT> __device__ __forceinline__ int attn_step() { return DEALT ? 1 : gridDim.x; }
struct AttnItem {
    int j, h, qt, split;     // frame of the pass, head, query tile, split
    int tile;                // number of the query tile among those that are split
    int b0, nb, nsplit;      // key blocks of this split (nb = 0: the frame's window has no such split)
    FrameDesc fr;
    template <bool DEALT> __device__ __forceinline__ bool place(int item, const AttnPlan &pl) {
        const AttnPlace p = attn_place<DEALT>(item, pl);
        j = p.j, split = p.split, tile = p.tile;
        h = pl.qt_div.div(p.t), qt = p.t - h * pl.QT;
        return p.whole;
    }
    template <bool DEALT> __device__ __forceinline__ void set(int item, const StepParams *sp, const Dims &D, const AttnPlan &pl) {
        const bool whole = place<DEALT>(item, pl);
        fr = sp->fr[j];
        const int nbt = (fr.frame - fr.win_first + 1) * pl.BPF;      // key blocks of this frame's window
        if (whole) {
            nsplit = 1, b0 = 0, nb = nbt;
        } else {
            nsplit = pl.ch_div.div(nbt + pl.CH - 1);
            b0 = split * pl.CH;
            nb = min(nbt, b0 + pl.CH) - b0;
        }
        if (nb < 0) nb = 0;
    }
    // the first item at or after `num` (in steps) that has blocks; `end` or more: there is none
    template <bool DEALT>
    __device__ __forceinline__ int find(int num, int end, const int *tab, const StepParams *sp, const Dims &D, const AttnPlan &pl) {
        for (; num < end; num += attn_step<DEALT>()) {
            set<DEALT>(DEALT ? tab[num] : num, sp, D, pl);
            if (nb > 0) break;
        }
        return num;
    }
};

// Offsets in a published state of row `trow`: columns 4 g .. 4 g + 3, (m, l) as the warp with half p of the columns wrote it.
__device__ __forceinline__ uint32_t attn_o_at(int g, int trow) { return (uint32_t)(g * 128 + trow) * 16; }
__device__ __forceinline__ uint32_t attn_ml_at(int p, int trow) { return 128 * 64 * 4 + (uint32_t)(p * 128 + trow) * 8; }
// n (a multiple of 8) columns of a result row from column e0 on
template <int n>
__device__ __forceinline__ void attn_write(const AttnItem &w, int row, int e0, const float *O, float l, const Dims &D, bf16 *out) {
    if (row >= D.T || e0 >= D.dh) return;
    const float inv = 1.0f / l;
    bf16 *o = out + (size_t)(w.j * D.T + row) * D.d + w.h * D.dh + e0;
#pragma unroll
    for (int e = 0; e < n; e += 8) {
        float t[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) t[u] = O[e + u] * inv;
        *reinterpret_cast<uint4 *>(o + e) = pack_bf16x8(t);
    }
}

// The end of an item for one warp: halves p0 .. p0 + np - 1 (32 columns each) of the 32 rows of its quadrant are read from
// tensor memory and written out, or published (attn_merge).
// m, l: reference and sum of this thread's row.  With `redo` (see AttnShared; a byte per item, a bit per half and
// quadrant; this is item `num`) a half whose l or O has left fp32 is left alone and marked there; without it, `mask` tells
// which halves to take.
template <bool OWN>
static __device__ __forceinline__ void attn_finish(const AttnItem &w, int p0, int np, int mask, uint32_t tO, uint32_t o_free,
                                                   int trow, float m, float l, const Dims &D, const AttnPlan &pl, bf16 *out,
                                                   float *part_o, uint32_t *redo, int num) {
    const int lane = threadIdx.x & 31, row = w.qt * 128 + trow;
    // OWN: the state goes to the CTA's own shared memory, for its cluster
    uint8_t *state = reinterpret_cast<uint8_t *>(part_o) + (OWN ? 0 : ((size_t)w.tile * pl.MAXSPLIT + w.split) * ATTN_STATE_BYTES);
#pragma unroll 1
    for (int p = p0; p < p0 + np; ++p) {
        float O[32];
        tmem_ld32(tO + 32 * p, reinterpret_cast<uint32_t *>(O));
        tmem_ld_wait();
        if (redo) {
            float2 x = make_float2(0.f, 0.f);              // NaN if an element of O is infinite or NaN
#pragma unroll
            for (int e = 0; e < 32; e += 2) x = ffma2(make_float2(O[e], O[e + 1]), make_float2(0.f, 0.f), x);
            // (rows beyond the frame's are another frame's or nothing, and not looked at)
            if (__any_sync(0xffffffffu, row < D.T && (l == INFINITY || x.x != x.x || x.y != x.y))) {
                mask &= ~(1 << p);
                if (lane == 0) {
                    atomicOr(redo, ATTN_MARKED);
                    atomicOr(redo + 2 + (num >> 2), 1u << (8 * (num & 3) + 4 * p + (trow >> 5)));
                }
            }
        }
        if (!((mask >> p) & 1)) continue;
        if (w.nsplit == 1) {
            attn_write<32>(w, row, 32 * p, O, l, D, out);
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                *reinterpret_cast<float4 *>(state + attn_o_at(8 * p + e, trow)) = make_float4(O[4 * e], O[4 * e + 1], O[4 * e + 2], O[4 * e + 3]);
            *reinterpret_cast<float2 *>(state + attn_ml_at(p, trow)) = make_float2(m, l);
        }
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0 && o_free) mbar_arrive(o_free);
}

// When a CTA is through with its items: one warp counts it in for each of those that are pieces of a split key range, a lane
// for an item, and all merge, in split order, those for which it is the last, a warp a quarter of the columns of a quadrant's
// rows.  Done as each item ended, the fence, the counter and the merge kept one of the softmax groups, and with it the order
// of the products, for 3.5 us an item (310M class, four frames behind 16: 70.7 -> 65.6 us a launch; one frame, an item to a CTA, 25.0
// both ways).  What the merge needs of an item comes through shared memory: read from the descriptor
// once more, behind the barrier, it cost launches of one item to a CTA 0.2 to 0.5 us.  Three states in flight and no more: with four the kernel's spilled registers
// doubled, on the path of every item (5407, 13880, 4142).
// The counter of the lane's item, if it has one; `all`: its pieces.
template <bool DEALT>
static __device__ __forceinline__ unsigned int *attn_counter(int num, int end, const int *tab, const StepParams *sp, const Dims &D,
                                                             const AttnPlan &pl, unsigned int *counters, unsigned int &all) {
    if (num >= end) return nullptr;
    AttnItem w;
    w.set<DEALT>(DEALT ? tab[num] : num, sp, D, pl);
    all = w.nsplit;
    return w.nb > 0 && w.nsplit > 1 ? counters + w.tile : nullptr;
}
// Bit i: this CTA is the last of the tile of lane i's item.  (One warp; a barrier has ordered the CTA's states before.)
static __device__ __forceinline__ uint32_t attn_count(unsigned int *cnt, unsigned int all) {
    bool last = false;
    if (cnt) {
        last = atomic_inc_acq_rel(cnt) == all - 1;
        if (last) *cnt = 0;                                // ready for the next launch
    }
    return __ballot_sync(0xffffffffu, last);
}
// i0: item of bit 0; pieces: of the tile of each bit's item
template <bool DEALT>
static __device__ __forceinline__ void attn_merge(uint32_t last, int i0, const int *tab, const uint32_t *pieces, const Dims &D,
                                                  const AttnPlan &pl, bf16 *out, const float *part_o) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cq = warp >> 2, trow = (warp & 3) * 32 + lane;
    if (16 * cq >= D.dh) return;
    AttnItem w;
#pragma unroll 1
    for (; last; last &= last - 1) {
        const int bit = __ffs(last) - 1;
        const int num = i0 + bit * attn_step<DEALT>();
        w.place<DEALT>(DEALT ? tab[num] : num, pl);
        w.nsplit = pieces[bit];
        const uint8_t *st = reinterpret_cast<const uint8_t *>(part_o) + (size_t)w.tile * pl.MAXSPLIT * ATTN_STATE_BYTES;
        float O[16], lt = 0.f, mx = -INFINITY;
#pragma unroll
        for (int e = 0; e < 16; ++e) O[e] = 0.f;
        // three states at a time, their loads in flight together
#pragma unroll 1
        for (int s0 = 0; s0 < w.nsplit; s0 += 3, st += 3 * ATTN_STATE_BYTES) {
            float2 ml[3];
            float4 v[3][4];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                ml[i] = make_float2(-INFINITY, 0.f);
#pragma unroll
                for (int e = 0; e < 4; ++e) v[i][e] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (s0 + i < w.nsplit) {
                    ml[i] = __ldcg(reinterpret_cast<const float2 *>(st + i * ATTN_STATE_BYTES + attn_ml_at(cq >> 1, trow)));
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        v[i][e] = __ldcg(reinterpret_cast<const float4 *>(st + i * ATTN_STATE_BYTES + attn_o_at(4 * cq + e, trow)));
                }
            }
            // every rounding is spelled out: the bits must not depend on which CTA merges
            const float mb = fmaxf(fmaxf(mx, ml[0].x), fmaxf(ml[1].x, ml[2].x));
            const float fo = mx == mb ? 1.0f : ex2_approx(mx - mb);
            mx = mb, lt = __fmul_rn(lt, fo);
#pragma unroll
            for (int e = 0; e < 16; ++e) O[e] = __fmul_rn(O[e], fo);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                // (a state with nothing but scores of -inf has m = -inf and counts for nothing)
                const float wgt = ml[i].x == -INFINITY ? 0.f : ex2_approx(ml[i].x - mb);
                lt = fmaf(ml[i].y, wgt, lt);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    O[4 * e] = fmaf(v[i][e].x, wgt, O[4 * e]);
                    O[4 * e + 1] = fmaf(v[i][e].y, wgt, O[4 * e + 1]);
                    O[4 * e + 2] = fmaf(v[i][e].z, wgt, O[4 * e + 2]);
                    O[4 * e + 3] = fmaf(v[i][e].w, wgt, O[4 * e + 3]);
                }
            }
        }
        attn_write<16>(w, w.qt * 128 + trow, 16 * cq, O, lt, D, out);
    }
}

// The shared memory of a CTA, and its tensor memory.
template <int KB> struct AttnShared {
    using A = AttnCfg<KB>;
    uint8_t *base;           // 1024-byte boundary
    uint32_t q, kv, bars, tmem;
    float *m, *l, *mx;       // [item parity][128], [item parity][group][128], [128] true maxima (times c)
    int *tab;                // [ATTN_CTA_ITEMS] the CTA's items, where they are dealt out
    uint32_t *redo;          // flags (below), the items to merge, and a byte per item (see attn_finish)
    __device__ __forceinline__ uint32_t *tmem_slot() const { return redo + 2 + ATTN_CTA_ITEMS / 4 + 2 * (11 + 5 * A::NS); }
    __device__ __forceinline__ AttnShared(uint8_t *raw) {
        uint8_t *smem = base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
        q = smem_u32(smem), kv = q + 2 * A::Q_BYTES, tmem = 0;
        m = reinterpret_cast<float *>(smem + 2 * A::Q_BYTES + 2 * A::NS * A::KV_BYTES), l = m + 2 * 128;
        mx = l + 2 * A::NGRP * 128, redo = reinterpret_cast<uint32_t *>(mx + 128);
        bars = smem_u32(redo + 2 + ATTN_CTA_ITEMS / 4);
        tab = reinterpret_cast<int *>(smem + A::STATE_AT);
    }
    // barriers (K of blocks 0 .. NS-1 arrives on k_first, V(n) and K(n + NS) on kv_full)
    __device__ __forceinline__ uint32_t q_full() const { return bars; }
    __device__ __forceinline__ uint32_t q_empty() const { return bars + 16; }
    __device__ __forceinline__ uint32_t m_full() const { return bars + 32; }
    __device__ __forceinline__ uint32_t l_full() const { return bars + 48; }
    __device__ __forceinline__ uint32_t ml_empty() const { return bars + 64; }
    __device__ __forceinline__ uint32_t o_free() const { return bars + 80; }
    __device__ __forceinline__ uint32_t k_first() const { return bars + 88; }
    __device__ __forceinline__ uint32_t s_full() const { return k_first() + 8 * A::NS; }
    __device__ __forceinline__ uint32_t p_full() const { return s_full() + 8 * A::NS; }
    __device__ __forceinline__ uint32_t kv_full() const { return p_full() + 8 * A::NS; }
    __device__ __forceinline__ uint32_t v_empty() const { return kv_full() + 8 * A::NS; }
    __device__ __forceinline__ void init_bars() const {
        for (int s = 0; s < 2; ++s) {
            mbar_init(q_full() + 8 * s, 1);
            mbar_init(q_empty() + 8 * s, 1);
            mbar_init(m_full() + 8 * s, 4);                // one arrival per warp of the group that finds m
            mbar_init(l_full() + 8 * s, 4 * A::NGRP);      // one per softmax warp
            mbar_init(ml_empty() + 8 * s, 4);              // one per warp of the group that finishes the item
        }
        mbar_init(o_free(), 4);                            // one arrival per warp that has read O
        for (int s = 0; s < A::NS; ++s) {
            mbar_init(k_first() + 8 * s, 1);
            mbar_init(s_full() + 8 * s, 1);
            mbar_init(p_full() + 8 * s, 4);                // one arrival per softmax warp of the group
            mbar_init(kv_full() + 8 * s, 2);               // one arrival per producer
            mbar_init(v_empty() + 8 * s, 1);
        }
        fence_mbar_init();
    }
    __device__ __forceinline__ void inval_bars() const {
        for (int i = 0; i < 11 + 5 * A::NS; ++i) mbar_inval(bars + 8 * i);
    }
};

// What a walk through items is for: the results, with m from the first scores; the true maxima of an item's rows (S alone
// counts: P and O are not looked at); the results with these as m.
enum { RD_FIRST, RD_MAX, RD_AGAIN };

// The CTA's items from number `first` on, below end (w0 is the first one); `num`: number of the item in sh.redo, not for
// RD_FIRST.
template <int KB, bool OWN, bool DEALT>
__device__ __forceinline__ void attn_items(const AttnShared<KB> &sh, const CUtensorMap &tmQ, const CUtensorMap &tmK,
                                           const CUtensorMap &tmV, const StepParams *sp, const Dims &D, int layer, const AttnPlan &pl,
                                           const AttnItem &w0, int first, int end, int mode, int num, bf16 *out, float *part_o,
                                           int *status, int test_skip) {
    using A = AttnCfg<KB>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t q_full = sh.q_full(), q_empty = sh.q_empty(), o_free = sh.o_free(), k_first = sh.k_first(), s_full = sh.s_full(),
                   p_full = sh.p_full(), kv_full = sh.kv_full(), v_empty = sh.v_empty(), m_full = sh.m_full(), l_full = sh.l_full(),
                   ml_empty = sh.ml_empty(), tmem = sh.tmem;
    float *s_m = sh.m, *s_l = sh.l;
    bool ok = true;
    // Blocks are numbered through the items (n): ring stages, accumulators and barrier phases follow n.
    if (warp == 0 || warp == 3) {
        // ---------------- TMA producers: K (warp 0), V (warp 3) ----------------
        // The two loops are kept short and free of divisions: as one thread with a division per block they took
        // 900 clocks a load (instruction fetches and the special-function unit are what the softmax warps saturate),
        // and this thread, not the softmax, set the pace of the whole kernel.
        if (elect_one()) {
            const bool is_k = warp == 0;
            const uint32_t ring = sh.kv + (is_k ? 0 : A::NS * A::KV_BYTES);
            const CUtensorMap *tm = is_k ? &tmK : &tmV;
            const uint32_t empty = is_k ? s_full : v_empty;
            bool waited = false;
            if (is_k && test_skip) ok = false;             // test switch: no K comes, and every wait behind it runs out
            int st = 0, lap = 0;                           // ring stage of the next block, how often the ring was filled
            AttnItem w = w0;
            for (int item = first; item < end && ok; item += attn_step<DEALT>()) {
                if (item != first) w.set<DEALT>(DEALT ? sh.tab[item] : item, sp, D, pl);
                const int f = pl.bpf_div.div(w.b0);
                int kb = w.b0 - f * pl.BPF;
                int left = w.fr.first_new - (w.fr.win_first + f);      // frames until the pages that this pass writes
                int slot = w.fr.win_slot + f;
                if (slot >= D.R) slot -= D.R;
                int page = ((w.fr.stream * D.L + layer) * D.R + slot) * D.H + w.h;
                const int wrap = D.R * D.H;
                int to_wrap = D.R - slot;            // frames until the ring of this layer wraps
                for (int b = 0; b < w.nb; ++b) {
                    if (left <= 0 && !waited) {
                        pdl_wait();                  // from here on the predecessor's output is needed
                        waited = true;
                    }
                    if (lap > 0) ok = mbar_wait(empty + 8 * st, (lap - 1) & 1, status);
                    if (!ok) break;
                    const uint32_t bar = (is_k && lap == 0 ? k_first : kv_full) + 8 * st;
                    mbar_expect_tx(bar, A::KV_BYTES);
                    tma_load_3d(ring + st * A::KV_BYTES, tm, bar, 0, kb * KB, page);
                    if (++st == A::NS) st = 0, ++lap;
                    if (++kb == pl.BPF) {
                        kb = 0, --left, page += D.H;
                        if (--to_wrap == 0) page -= wrap, to_wrap = D.R;
                    }
                }
            }
            // the last V blocks have no K block NS further on
            if (is_k) {
                const int n = lap * A::NS + st;            // blocks of this CTA
                for (int i = n < A::NS ? n : A::NS; i > 0 && ok; --i) {
                    const int x = n - i;
                    ok = mbar_wait(s_full + 8 * (x % A::NS), (x / A::NS) & 1, status);
                    if (ok) mbar_arrive(kv_full + 8 * (x % A::NS));
                }
            }
            if (!ok) atomicOr(sh.redo, ATTN_EXPIRED);
        }
    } else if (warp == 1) {
        // ---------------- issuer of S = Q K^T and O += P V, loader of Q ----------------
        if (elect_one()) {
            pdl_launch();
            constexpr uint32_t idesc_s = umma_idesc_bf16(128, KB), idesc_pv = umma_idesc_bf16_bmn(128, 64);
            const uint32_t sQ = sh.q, sK = sh.kv, sV = sK + A::NS * A::KV_BYTES;
            // S runs NS blocks ahead of P V: items of their own for both.  (One copy of the code for both the first S and the
            // later ones: this thread's registers and instruction fetches are on every block's path.)
            AttnItem ws = w0, w = w0;
            int item_s = first, it_s = -1, left_s = 0;            // item whose Q was asked for last; items before S's; S to come
            int item = first - attn_step<DEALT>(), it = 0, left = 0;            // the same for P V
            int st_s = 0, lap_s = 0, st = 0, lap = 0;
            int ahead = A::NS;                             // S to issue before the first P V
            auto load_q = [&](int qs) {                    // Q of item ws
                mbar_expect_tx(q_full + 8 * qs, A::Q_BYTES);
                tma_load_3d(sQ + qs * A::Q_BYTES, &tmQ, q_full + 8 * qs, 0, ws.j * D.T + ws.qt * 128, ws.h);
            };
            pdl_wait();
            if (ws.nb == 0) item_s = ws.find<DEALT>(item_s + attn_step<DEALT>(), end, sh.tab, sp, D, pl);
            if (item_s < end) load_q(0);
            while (ok) {
                if (ahead > 0) {
                    --ahead;
                } else {
                    uint32_t acc = 1;
                    if (left == 0) {
                        item = w.find<DEALT>(item + attn_step<DEALT>(), end, sh.tab, sp, D, pl);
                        if (item >= end) break;
                        left = w.nb, acc = 0;
                        if (it > 0) ok = mbar_wait(o_free, (it - 1) & 1, status);          // O of the last item has been read
                        ++it;
                    }
                    ok = ok && mbar_wait(kv_full + 8 * st, lap & 1, status) && mbar_wait(p_full + 8 * st, lap & 1, status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t vd = umma_desc_k128(sV + st * A::KV_BYTES);
                    const uint32_t tP = tmem + A::S_STRIDE * st;
#pragma unroll
                    for (int i = 0; i < KB / 16; ++i) {
                        // P: 16 keys = 8 columns of packed bf16 pairs, and 8 of what they leave; V: MN-major, 16 keys = 2 KiB
                        const uint64_t vi = vd + (uint64_t)(i * (2048 >> 4));
                        umma_bf16_ts(tmem + A::TM_O, tP + 16 * i, vi, idesc_pv, i ? 1u : acc);
                        umma_bf16_ts(tmem + A::TM_O, tP + 16 * i + 8, vi, idesc_pv, 1u);
                    }
                    umma_commit(v_empty + 8 * st);         // P V(n) is complete: V's stage is free, O at rest
                    if (++st == A::NS) st = 0, ++lap;
                    --left;
                }
                // S of the next block, if there is one, into the accumulator that P V(n) reads
                if (left_s == 0) {
                    if (item_s >= end) continue;
                    ++it_s, left_s = ws.nb;
                    ok = mbar_wait(q_full + 8 * (it_s & 1), (it_s >> 1) & 1, status);
                    item_s = ws.find<DEALT>(item_s + attn_step<DEALT>(), end, sh.tab, sp, D, pl);
                    if (ok && item_s < end) {              // Q of the item after it
                        if (it_s >= 1) ok = ok && mbar_wait(q_empty + 8 * ((it_s + 1) & 1), ((it_s - 1) >> 1) & 1, status);
                        if (ok) load_q((it_s + 1) & 1);    // (no copy is begun after a wait has run out)
                    }
                }
                // (K of later blocks has arrived together with V of the block NS back)
                if (lap_s == 0) ok = ok && mbar_wait(k_first + 8 * st_s, 0, status);
                if (!ok) break;
                tc_fence_after();
                const uint64_t qd = umma_desc_k128(sQ + (it_s & 1) * A::Q_BYTES), kd = umma_desc_k128(sK + st_s * A::KV_BYTES);
#pragma unroll
                for (int k4 = 0; k4 < 4; ++k4)
                    umma_bf16_ss(tmem + A::S_STRIDE * st_s, qd + 2 * k4, kd + 2 * k4, idesc_s, k4 != 0);
                umma_commit(s_full + 8 * st_s);            // S is ready; K's stage is free
                if (++st_s == A::NS) st_s = 0, ++lap_s;
                if (--left_s == 0) umma_commit(q_empty + 8 * (it_s & 1));
            }
            // completions that nobody has waited for yet: none may arrive when the barriers are set up anew
            const int n = lap * A::NS + st;
            for (int x = n > A::NS ? n - A::NS : 0; x < n; ++x)
                ok = ok && mbar_wait(v_empty + 8 * (x % A::NS), (x / A::NS) & 1, status);
            for (int i = it_s > 0 ? it_s - 1 : 0; i <= it_s; ++i) ok = ok && mbar_wait(q_empty + 8 * (i & 1), (i >> 1) & 1, status);
            if (!ok) atomicOr(sh.redo, ATTN_EXPIRED);
        }
    } else if (warp == 2) {
        // no work of its own (the softmax warps start at a multiple of four: a warp reads tensor-memory lanes 32 (warp % 4) ..)
    } else {
        // ---------------- softmax: one thread per query row, three groups ----------------
        const int g = (warp - A::SM_WARP0) >> 2;           // group: blocks n with n % 3 == g
        const int quad = warp & 3;                         // tensor-memory lanes this warp may touch
        const int trow = quad * 32 + lane;
        const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
        const float c = (1.0f / sqrtf((float)D.dh)) * 1.4426950408889634f;   // softmax scale in the log2 domain
        int n0 = 0, n03 = 0, it = 0;                       // the item's first block, that modulo 3, items before it
        const uint32_t tO = tmem + A::TM_O + lane_off;
        AttnItem w = w0;
        int item = first;
        if (w.nb == 0) item = w.find<DEALT>(item + attn_step<DEALT>(), end, sh.tab, sp, D, pl);
        while (item < end) {
            const int ip = it & 1, iph = (it >> 1) & 1;    // item parity: which m and l, phase of their barriers
            const int r = g >= n03 ? g - n03 : g - n03 + A::NGRP;      // this group's blocks: b % 3 == r
            float m_run = 0.f, l_run = mode == RD_MAX ? -INFINITY : 0.f, l_top = 0.f;      // l_top: the largest sum of a block
            int kb = w.b0 + r;                             // block of the page, for the mask of its last block
            kb -= pl.bpf_div.div(kb) * pl.BPF;
            for (int b = r; b < w.nb || b == r; b += A::NGRP) {
                // (a group without a block still takes part in the hand-over of m and l)
                const bool some = b < w.nb;
                const int n = n0 + b, st = n % A::NS;
                const uint32_t tS = tmem + A::S_STRIDE * st + lane_off;
                if (some) {
                    const int nvalid = D.T - kb * KB;      // keys of this block (>= KB except at the end of a page)
                    kb += A::NGRP;
                    while (kb >= pl.BPF) kb -= pl.BPF;
                    // (a warp whose wait has run out goes on without waiting, on whatever the accumulators hold: it has to
                    // take part in the barriers below)
                    ok = ok && mbar_wait(s_full + 8 * st, (n / A::NS) & 1, status);
                    __syncwarp();
                    tc_fence_after();
                    if (nvalid < KB) {
                        // the last block of a page whose length KB does not divide: the columns beyond the page take -inf
                        int cm = nvalid & ~7;
                        if (nvalid & 7) {
                            uint32_t r[8];
                            tmem_ld8(tS + cm, r);
                            tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 8; ++e)
                                if (cm + e >= nvalid) r[e] = 0xff800000u;
                            tmem_st8(tS + cm, r);
                            cm += 8;
                        }
                        for (; cm < KB; cm += 8) {
                            uint32_t r[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) r[e] = 0xff800000u;
                            tmem_st8(tS + cm, r);
                        }
                        tmem_st_wait();
                    }
                }
                if (b == r) {
                    // m of the item: the largest of the first 16 scores of the row, found by the group of block 0 for all
                    if (r == 0) {
                        NFD_TRACE_MARK_T(TRK_OTHER + 11, 128);
                        if (it >= 2) ok = ok && mbar_wait(ml_empty + 8 * ip, iph ^ 1, status);   // item it - 2 is done with
                        __syncwarp();
                        uint32_t x[16];
                        tmem_ld16(tS, x);
                        tmem_ld_wait();
                        float mx = -INFINITY;
#pragma unroll
                        for (int e = 0; e < 16; ++e) mx = fmaxf(mx, __uint_as_float(x[e]));
                        m_run = mode == RD_AGAIN ? sh.mx[trow] : mx * c;
                        s_m[ip * 128 + trow] = m_run;
                        __syncwarp();
                        if (lane == 0) mbar_arrive(m_full + 8 * ip);
                    } else {
                        ok = ok && mbar_wait(m_full + 8 * ip, iph, status);
                        m_run = s_m[ip * 128 + trow];
                        __syncwarp();
                    }
                    if (!some) break;
                }
                if (mode == RD_MAX) {                      // l_run: the largest score
#pragma unroll 1
                    for (int cc = 0; cc < KB; cc += 16) {
                        uint32_t x[16];
                        tmem_ld16(tS + cc, x);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 16; ++e) l_run = fmaxf(l_run, __uint_as_float(x[e]));
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(p_full + 8 * st);
                    continue;
                }
                // One pass over S, 16 columns at a time with the next load in flight: p = exp2(S c - m), written as two packed
                // bf16 pairs over the columns it came from (keys k .. k+15: the first numbers go to columns k .. k+7).
                float2 ls2[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                uint32_t sa[16], sb[16];
                tmem_ld16(tS, sa);
#pragma unroll
                for (int cc = 0; cc < KB; cc += 16) {
                    uint32_t *cur = ((cc >> 4) & 1) ? sb : sa, *nxt = ((cc >> 4) & 1) ? sa : sb;
                    tmem_ld_wait();
                    if (cc + 16 < KB) tmem_ld16(tS + cc + 16, nxt);
                    uint32_t pk[16];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const float s0 = __uint_as_float(cur[2 * u]), s1 = __uint_as_float(cur[2 * u + 1]);
                        const float2 y = ffma2(make_float2(s0, s1), make_float2(c, c), make_float2(-m_run, -m_run));
                        const float2 p = make_float2(ex2_approx(y.x), ex2_approx(y.y));
                        ls2[u & 3] = fadd2(ls2[u & 3], p);
                        bf16_split2(p, pk[u], pk[8 + u]);
                    }
                    tmem_st16(tS + cc, pk);
                }
                const float ls = ((ls2[0].x + ls2[0].y) + (ls2[1].x + ls2[1].y)) + ((ls2[2].x + ls2[2].y) + (ls2[3].x + ls2[3].y));
                l_run += ls;
                l_top = fmaxf(l_top, ls);
                tmem_st_wait();                            // P is in tensor memory
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(p_full + 8 * st);
            }
            NFD_TRACE_MARK_T(TRK_OTHER + 12, 128);
            // the group's sum; infinite: the item's row is to be computed again
            s_l[(ip * A::NGRP + r) * 128 + trow] =
                mode == RD_FIRST && (l_top > 1.2676506e30f /* 2^100 */ || m_run == -INFINITY) ? INFINITY : l_run;
            __syncwarp();
            if (lane == 0) mbar_arrive(l_full + 8 * ip);
            const int bl = n0 + w.nb - 1;                  // the item's last block
            n0 += w.nb, ++it;
            const int gl = (n03 + w.nb - 1) % A::NGRP;     // the group of that block
            n03 = gl + 1 == A::NGRP ? 0 : gl + 1;
            AttnItem wn;
            int was = item;
            item = wn.find<DEALT>(item + attn_step<DEALT>(), end, sh.tab, sp, D, pl);
            // The group of the last block finishes the item while the others are on the next one; groups 0 and 1 share the
            // CTA's last item.
            const bool fin = item >= end;
            if (fin ? g < 2 : g == gl) {
                // (The item worked out again: kept through the loop it would cost registers that it needs.  Ahead of the waits:
                // behind them it held back the next item's products, 0.1 us an item.)
                asm volatile("" : "+r"(was));
                w.place<DEALT>(DEALT ? sh.tab[was] : was, pl);
                ok = ok && mbar_wait(l_full + 8 * ip, iph, status);
                const float *sl = s_l + ip * A::NGRP * 128 + trow;
                float l = (sl[0] + sl[128]) + sl[256];
                float m = s_m[ip * 128 + trow];
                // the maxima of the rows; a row without any counts from 0 (and its sum is 0)
                if (mode == RD_MAX && g == 0) {
                    const float mx = fmaxf(fmaxf(sl[0], sl[128]), sl[256]) * c;
                    sh.mx[trow] = mx == -INFINITY ? 0.f : mx;
                }
                __syncwarp();
                if (!fin && lane == 0) mbar_arrive(ml_empty + 8 * ip);
                ok = ok && mbar_wait(v_empty + 8 * (bl % A::NS), (bl / A::NS) & 1, status);
                __syncwarp();
                tc_fence_after();
                ok = __all_sync(0xffffffffu, ok);
                if (mode != RD_MAX) {
                    int mask = 3;
                    if (!ok) l = NAN;                      // a wait has run out: the result says so
                    if (mode == RD_AGAIN) {
                        const uint32_t marks = sh.redo[2 + (num >> 2)] >> (8 * (num & 3) + quad);
                        mask = (marks & 1) | ((marks >> 3) & 2);
                        if (l == 0.f) m = -INFINITY;
                    }
                    attn_finish<OWN>(w, fin ? g : 0, fin ? 1 : 2, mask, tO, fin ? 0u : o_free, trow, m, l, D, pl, out,
                                part_o, mode == RD_FIRST && ok ? sh.redo : nullptr, it - 1);
                }
            }
            w = wn;
        }
        if (!ok && lane == 0) atomicOr(sh.redo, ATTN_EXPIRED);
    }
}

// The items with marked rows once more, each twice.  Not inlined: the first walk's code is as if this were not there.
// After a wait that has run out the marked rows are NaN (and counted: the tile's other splits may be waited for).
template <int KB, bool OWN, bool DEALT>
static __device__ __noinline__ void attn_again(const AttnShared<KB> sh, const CUtensorMap &tmQ, const CUtensorMap &tmK,
                                               const CUtensorMap &tmV, const StepParams *sp, const Dims &D, int layer,
                                               const AttnPlan &pl, int end, bf16 *out, float *part_o, int *status) {
    using A = AttnCfg<KB>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = (warp - A::SM_WARP0) >> 2, quad = warp & 3;
    AttnItem w;
    int num = 0;                                           // items with blocks so far
    for (int item = attn_first<DEALT>(); (item = w.find<DEALT>(item, end, sh.tab, sp, D, pl)) < end; item += attn_step<DEALT>(), ++num) {
        const uint32_t marks = (sh.redo[2 + (num >> 2)] >> (8 * (num & 3))) & 255;
        if (!marks) continue;
        int mode = RD_MAX;
#pragma unroll 1
        for (; mode <= RD_AGAIN && !(sh.redo[0] & ATTN_EXPIRED); ++mode) {
            // (every completion of the last walk has been waited for)
            if (threadIdx.x == 0) sh.inval_bars(), sh.init_bars();
            __syncthreads();
            tc_fence_after();
            attn_items<KB, OWN, DEALT>(sh, tmQ, tmK, tmV, sp, D, layer, pl, w, item, item + 1, mode, num, out, part_o, status, 0);
            tc_fence_before();
            __syncthreads();
        }
        // (the second walk writes its rows in any case)
        if (mode <= RD_AGAIN && warp >= A::SM_WARP0 && g < 2)
            attn_finish<OWN>(w, g, 1, (marks >> quad & 1) | (marks >> quad >> 3 & 2), sh.tmem + A::TM_O + ((uint32_t)(quad * 32) << 16), 0u,
                        quad * 32 + lane, 0.f, NAN, D, pl, out, part_o, nullptr, 0);
    }
}

template <int KB>
__device__ __forceinline__ void attn_set_up(AttnShared<KB> &sh, const CUtensorMap &tmQ, const CUtensorMap &tmK, const CUtensorMap &tmV) {
    using A = AttnCfg<KB>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&tmQ);
        tma_prefetch_desc(&tmK);
        tma_prefetch_desc(&tmV);
        sh.init_bars();
    }
    for (int i = threadIdx.x; i < 2 + ATTN_CTA_ITEMS / 4; i += A::THREADS) sh.redo[i] = 0;
    if (warp == 1) {
        tmem_alloc(smem_u32(sh.tmem_slot()), A::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    sh.tmem = *sh.tmem_slot();
}

template <int KB, bool DEALT>
__global__ void __launch_bounds__(AttnCfg<KB>::THREADS, 1)
k_attn_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
          const __grid_constant__ CUtensorMap tmV, const StepParams *sp, const __grid_constant__ Dims D, int layer,
          const __grid_constant__ AttnPlan pl, bf16 *out, float *part_o, unsigned int *counters, int *status, int test_skip) {
    extern __shared__ uint8_t smem_raw[];
    NFD_TRACE_T0();
    AttnShared<KB> sh(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int first = attn_first<DEALT>(), step = attn_step<DEALT>(), end = DEALT ? attn_dealt_count(blockIdx.x, pl) : pl.n_items;
    // The first item's descriptor: its loads are in flight during the set-up.  (In a pass the descriptor was written by the
    // first kernel, for whose end the kernels between have waited; where its writer is this kernel's predecessor, the launch
    // is in plain stream order.)
    AttnItem w0;
    w0.set<DEALT>(DEALT ? attn_dealt(blockIdx.x, 0, pl) : blockIdx.x, sp, D, pl);
    if (DEALT)
        for (int n = threadIdx.x; n < end; n += AttnCfg<KB>::THREADS) sh.tab[n] = attn_dealt(blockIdx.x, n, pl);

    attn_set_up<KB>(sh, tmQ, tmK, tmV);
    attn_items<KB, false, DEALT>(sh, tmQ, tmK, tmV, sp, D, layer, pl, w0, first, end, RD_FIRST, 0, out, part_o, status, test_skip);
    NFD_TRACE_MARK_T(TRK_OTHER + 16, 128);
    unsigned int *cnt = nullptr, all = 0;
    if (warp == 2 && pl.MAXSPLIT > 1) cnt = attn_counter<DEALT>(first + lane * step, end, sh.tab, sp, D, pl, counters, all);
    tc_fence_before();
    __syncthreads();
    if (sh.redo[0] & ATTN_MARKED) {
        attn_again<KB, false, DEALT>(sh, tmQ, tmK, tmV, sp, D, layer, pl, end, out, part_o, status);
        __syncthreads();                                   // (it writes states too)
    }
    if (pl.MAXSPLIT > 1) {
#pragma unroll 1
        for (int i0 = first; i0 < end; i0 += 32 * step) {
            if (warp == 2) {
                if (i0 != first) cnt = attn_counter<DEALT>(i0 + lane * step, end, sh.tab, sp, D, pl, counters, all);
                const uint32_t last = attn_count(cnt, all);
                if (lane == 0) sh.redo[1] = last;
                sh.redo[2 + lane] = all;                   // (the marks have been seen to)
            }
            __syncthreads();                               // what that warp has acquired is handed to the others
            attn_merge<DEALT>(sh.redo[1], i0, sh.tab, sh.redo + 2, D, pl, out, part_o);
            if (i0 + 32 * step < end) __syncthreads();
        }
    }
    if (warp == 1) tmem_dealloc(sh.tmem, AttnCfg<KB>::TMEM_COLS);
    NFD_TRACE_END(TRK_ATTN);
}

// The caller's pages (nfd_attention_noalloc), for which there is no memory for states: the pieces of a split key range are the
// CTAs of a cluster, an item each.  Each leaves its state in its own shared memory, and after a cluster barrier they merge them
// through distributed shared memory, in split order, each CTA some quarters of the columns.  Without a split k_attn_tc takes the
// call (run as clusters of one here: 4 heads x 32, 8 x 336 queries behind 32 frames 72.6 -> 74.5 us, 16 x 64 200.0 -> 202.5).
// Measured, 16 heads x 64, 336 queries behind 16 frames of 336 (48 query tiles), us with both launches of the call: one CTA to a
// tile 43.1, two 30.8.  (Three would want 48 clusters, and the machine holds 45.)
template <int KB>
__global__ void __launch_bounds__(AttnCfg<KB>::THREADS, 1)
k_attn_own(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
           const __grid_constant__ CUtensorMap tmV, const StepParams *sp, const __grid_constant__ Dims D,
           const __grid_constant__ AttnPlan pl, bf16 *out, int *status, int test_skip) {
    using A = AttnCfg<KB>;
    extern __shared__ uint8_t smem_raw[];
    AttnShared<KB> sh(smem_raw);
    float *state = reinterpret_cast<float *>(sh.base + A::STATE_AT);
    AttnItem w0;
    w0.set<false>(blockIdx.x, sp, D, pl);
    attn_set_up<KB>(sh, tmQ, tmK, tmV);
    const int end = blockIdx.x + 1;
    attn_items<KB, true, false>(sh, tmQ, tmK, tmV, sp, D, 0, pl, w0, blockIdx.x, end, RD_FIRST, 0, out, state, status, test_skip);
    tc_fence_before();
    __syncthreads();
    if (sh.redo[0] & ATTN_MARKED) attn_again<KB, true, false>(sh, tmQ, tmK, tmV, sp, D, 0, pl, end, out, state, status);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncwarp();
    cluster_sync_all();                                    // every state of the cluster is in place
    w0.set<false>(blockIdx.x, sp, D, pl);
    const int cq = warp >> 2, trow = (warp & 3) * 32 + lane;
    // (rows beyond the frame's are left alone: every value that is read has to be used, see below)
    if (w0.nsplit > 1 && w0.split < w0.nsplit && cq % w0.nsplit == w0.split && 16 * cq < D.dh && w0.qt * 128 + trow < D.T) {
        const uint32_t st = smem_u32(state);
        float O[16], lt = 0.f, mx = -INFINITY;
#pragma unroll
        for (int e = 0; e < 16; ++e) O[e] = 0.f;
#pragma unroll 1
        for (int s = 0; s < w0.nsplit; ++s) {
            const float2 ml = ld_cluster_f2(cluster_map(st + attn_ml_at(cq >> 1, trow), s));
            float4 v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = ld_cluster_f4(cluster_map(st + attn_o_at(4 * cq + e, trow), s));
            const float mb = fmaxf(mx, ml.x);
            // (a state with nothing but scores of -inf has m = -inf and counts for nothing)
            const float fo = mx == mb ? 1.0f : ex2_approx(mx - mb), wgt = ml.x == -INFINITY ? 0.f : ex2_approx(ml.x - mb);
            mx = mb, lt = fmaf(ml.y, wgt, __fmul_rn(lt, fo));
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                O[4 * e] = fmaf(v[e].x, wgt, __fmul_rn(O[4 * e], fo));
                O[4 * e + 1] = fmaf(v[e].y, wgt, __fmul_rn(O[4 * e + 1], fo));
                O[4 * e + 2] = fmaf(v[e].z, wgt, __fmul_rn(O[4 * e + 2], fo));
                O[4 * e + 3] = fmaf(v[e].w, wgt, __fmul_rn(O[4 * e + 3], fo));
            }
        }
        attn_write<16>(w0, w0.qt * 128 + trow, 16 * cq, O, lt, D, out);
    }
    __syncwarp();
    // No CTA leaves while a peer may still read its state.  The barrier orders nothing: what a thread has read went into its
    // results, which it has stored.  (With release, which lets reads be that nothing waits for, 0.5 us more.)
    cluster_arrive_relaxed();
    cluster_wait();
    if (warp == 1) tmem_dealloc(sh.tmem, A::TMEM_COLS);
}
