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
//                         sum, bf16 P written back to tensor memory over
//                         the first half of the S columns it came from
//     O += P V            UMMA 128 x 64 x KB, P read from tensor memory, V used
//                         straight from its page (MN-major B operand in shared
//                         memory), accumulated in tensor memory
// The reference maximum m of a row is that of its first block and is raised only when
// a block's sum exceeds 2^16; only then is the row's O accumulator rescaled (in tensor
// memory), so that in the steady state no maximum is taken and O is never read back.  The
// final normalisation by the running sum makes the result independent of that choice.
//
// Warps 0 and 3 = TMA producers (Q and K, V), warp 1 = issuer of the S products,
// warp 2 = issuer of the P V products, warps 4-7 and 8-11 = two softmax groups.  Group g takes
// the key blocks b of an item with b % 2 == g and keeps its own (m, sum, O)
// state, so that one group's waits overlap the other's arithmetic.
// S has three accumulators in tensor memory, the CTA's n-th block using number n % 3
// (and a "P is stored" barrier of its own: a warp of a group may be a whole block ahead of another, so one barrier
// per group would count its second arrival in place of the other's first);
// S(n + 3) is issued once P V(n), which reads P(n) from that accumulator, is
// complete: a group finds its next S ready when it comes back for it.  K blocks go
// through a ring of three stages (free again when S(n) is complete, which the barrier
// of accumulator n % 3 tells), V blocks through a ring of four (free when P V is complete).
//
// What bounds it: the softmax warps.  Their loop alone takes 825 clocks per 128 x 112 block (registers, tensor memory
// and the two arithmetic pipes; no products), the products 490.
// Measured, 16 heads x 64 on one B200 (events around a launch; with one thread issuing loads and one all products, and a
// maximum pass over S): one frame of 336 tokens behind 16: 28.4 -> 25.0 us; four frames: 88.8 -> 74.3; eight frames
// behind 32: 232 -> 188 (650 TFLOP/s).  Pages of 220 tokens ran on the plain kernel, 1342 us a layer; now 21 us.
//
// The grid is persistent: a CTA takes items blockIdx.x, + gridDim.x, ...; producers and
// issuers run ahead into the next item while the groups finish the last one.  At the
// end of an item the two groups' states are folded in shared memory.  A key range
// longer than CH blocks is split over several items; each publishes its
// unnormalised (O, m, l) state in global memory, stored so that a warp writes and reads
// whole lines, and the CTA that finishes last (a counter per query tile) reads the
// others and merges the states in split order.  CH depends only on the configuration, so
// a frame's result does not depend on which other frames share its pass.
#pragma once
#include "nfd_sm100.cuh"

struct AttnPlan {
    int KB = 0;          // keys per block
    int BPF = 0;         // blocks per frame page
    int QT = 0;          // 128-row query tiles per frame
    int CH = 0;          // key blocks per split
    int MAXSPLIT = 0;    // splits of the longest window
    FastDiv split_div, qt_div, h_div, ch_div, bpf_div;      // by MAXSPLIT, QT, heads, CH, BPF
};

// A published state: [16 groups of 4 columns][128 rows] float4, then [128 rows] (m, l).
#define ATTN_STATE_BYTES (128 * 64 * 4 + 128 * 8)

template <int KB> struct AttnCfg {
    static constexpr int NK = 3;                           // K ring stages = S accumulators
    static constexpr int NV = 4;                           // V ring stages
    static constexpr int Q_BYTES = 128 * 128;              // two of them: the next item's Q is loaded ahead
    static constexpr int KV_BYTES = KB * 128;              // one K (or V) block
    static constexpr int PARK_BYTES = 128 * 64 * 4;        // half of each group's O, on its way to the other group
    static constexpr int ML_BYTES = 2 * 128 * 8;           // (m, l) of every softmax thread
    static constexpr int SMEM = 2 * Q_BYTES + (NK + NV) * KV_BYTES + PARK_BYTES + ML_BYTES + 256 + 1024;
    static constexpr int TMEM_COLS = 512;                  // S0 @0, S1 @128, S2 @256, O0 @384, O1 @448
    static constexpr int SM_WARP0 = 4;                     // first softmax warp
    static constexpr int THREADS = 32 * (SM_WARP0 + 8);
    static_assert(KB % 16 == 0 && KB <= 128, "key block");
    static_assert(SMEM <= 232448, "shared memory of a CTA");
};

__host__ __device__ constexpr uint32_t umma_idesc_bf16_bmn(int M, int N) {
    return umma_idesc_bf16(M, N) | (1u << 16);             // B operand MN-major
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 2^y for two values y = S c - m on the FMA pipe: 2^n 2^f with n = round(y), f in [-1/2, 1/2], and 2^f by a
// polynomial of degree 4 fitted for equal relative error (2.7e-6; the result is rounded to bf16, 2e-3, afterwards).
// y is brought into [-125, 127] by the saturation of an FMA that maps this range to [0, 1]: ca = c / 252,
// cb = (125 - m) / 252.
#define EXP2_RANGE 252.0f
#define EXP2_LOW 125.0f
__device__ __forceinline__ float2 exp2_fma2(float s0, float s1, float ca, float cb) {
    const float M = 12582912.0f;                           // 1.5 * 2^23: adding it rounds to an integer
    auto k2 = [](float v) { return make_float2(v, v); };
    float2 z;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(z.x) : "f"(s0), "f"(ca), "f"(cb));
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(z.y) : "f"(s1), "f"(ca), "f"(cb));
    const float2 t = ffma2(z, k2(EXP2_RANGE), k2(M - EXP2_LOW));     // M + n
    const float2 n = fadd2(t, k2(EXP2_LOW - M));                     // n + 125
    const float2 f = ffma2(z, k2(EXP2_RANGE), make_float2(-n.x, -n.y));
    float2 p = ffma2(k2(0.009570100344717503f), f, k2(0.05591785907745361f));
    p = ffma2(p, f, k2(0.240247443318367f));
    p = ffma2(p, f, k2(0.6931217908859253f));
    p = ffma2(p, f, k2(0.9999992847442627f));
    return make_float2(__int_as_float(__float_as_int(p.x) + (__float_as_int(t.x) << 23)),
                       __int_as_float(__float_as_int(p.y) + (__float_as_int(t.y) << 23)));
}
// Maximum over the KB columns of a row of S.  Tensor-memory loads are warp-wide: only ever called by a whole warp.
template <int KB> __device__ __forceinline__ float row_max(uint32_t tS) {
    float m = -INFINITY;
#pragma unroll 1
    for (int cc = 0; cc < KB; cc += 16) {
        uint32_t s[16];
        tmem_ld16(tS + cc, s);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) m = fmaxf(m, __uint_as_float(s[e]));
    }
    return m;
}

__device__ __forceinline__ void named_bar_sync(int id, int n_threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n_threads) : "memory");
}

// One item of the grid.
struct AttnItem {
    int j, h, qt, split;     // frame of the pass, head, query tile, split
    int b0, nb, nsplit;      // key blocks of this split (nb = 0: the frame's window has no such split)
    FrameDesc fr;
    __device__ __forceinline__ void set(int item, const StepParams *sp, const Dims &D, const AttnPlan &pl) {
        const int a = pl.split_div.div(item), b = pl.qt_div.div(a);
        split = item - a * pl.MAXSPLIT, qt = a - b * pl.QT;
        j = pl.h_div.div(b), h = b - j * D.H;
        fr = sp->fr[j];
        const int nbt = (fr.frame - fr.win_first + 1) * pl.BPF;      // key blocks of this frame's window
        nsplit = pl.ch_div.div(nbt + pl.CH - 1);
        b0 = split * pl.CH;
        nb = min(nbt, b0 + pl.CH) - b0;
        if (nb < 0) nb = 0;
    }
};

template <int KB>
__global__ void __launch_bounds__(AttnCfg<KB>::THREADS, 1)
k_attn_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
          const __grid_constant__ CUtensorMap tmV, const StepParams *sp, Dims D, int layer, AttnPlan pl, int n_items,
          bf16 *out, float *part_o, unsigned int *counters, int *status) {
    using A = AttnCfg<KB>;
    extern __shared__ uint8_t smem_raw[];
    NFD_TRACE_T0();
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *sKV = smem + 2 * A::Q_BYTES, *sPark = sKV + (A::NK + A::NV) * A::KV_BYTES;
    uint4 *park = reinterpret_cast<uint4 *>(sPark);                          // [column half][8][128]
    float2 *s_ml = reinterpret_cast<float2 *>(sPark + A::PARK_BYTES);        // [group][128]
    uint64_t *bars = reinterpret_cast<uint64_t *>(sPark + A::PARK_BYTES + A::ML_BYTES);
    // barriers: q_full[2] | q_empty[2] | k_full[NK] | s_full[NK] | v_full[NV] | v_empty[NV] | p_full[NK]
    const uint32_t q_full = smem_u32(bars), q_empty = q_full + 16, k_full = q_empty + 16, s_full = k_full + 8 * A::NK,
                   v_full = s_full + 8 * A::NK, v_empty = v_full + 8 * A::NV, p_full = v_empty + 8 * A::NV;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 4 + 3 * A::NK + 2 * A::NV);
    int *last_flag = reinterpret_cast<int *>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&tmQ);
        tma_prefetch_desc(&tmK);
        tma_prefetch_desc(&tmV);
        for (int s = 0; s < 2; ++s) {
            mbar_init(q_full + 8 * s, 1);
            mbar_init(q_empty + 8 * s, 1);
        }
        for (int s = 0; s < A::NK; ++s) {
            mbar_init(k_full + 8 * s, 1);
            mbar_init(s_full + 8 * s, 1);
            mbar_init(p_full + 8 * s, 4);                  // one arrival per softmax warp of the group
        }
        for (int s = 0; s < A::NV; ++s) {
            mbar_init(v_full + 8 * s, 1);
            mbar_init(v_empty + 8 * s, 1);
        }
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), A::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // Blocks are numbered through the CTA's items (n): ring stages, accumulators and barrier phases follow n.
    if (warp == 0 || warp == 3) {
        // ---------------- TMA producers: Q and K (warp 0), V (warp 3) ----------------
        // The two loops are kept short and free of divisions: as one thread with a division per block they took
        // 900 clocks a load (instruction fetches and the special-function unit are what the softmax warps saturate),
        // and this thread, not the softmax, set the pace of the whole kernel.
        if (elect_one()) {
            const bool is_k = warp == 0;
            const uint32_t sQ = smem_u32(smem), ring = smem_u32(sKV) + (is_k ? 0 : A::NK * A::KV_BYTES);
            const CUtensorMap *tm = is_k ? &tmK : &tmV;
            const uint32_t full = is_k ? k_full : v_full, empty = is_k ? s_full : v_empty;
            const int n_ring = is_k ? A::NK : A::NV;
            bool waited = false, ok = true;
            int it = 0, st = 0, lap = 0;                   // ring stage of the next block, how often the ring was filled
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                AttnItem w;
                w.set(item, sp, D, pl);
                if (w.nb == 0) continue;
                bool have_q = !is_k;
                auto need_pred = [&]() {             // from here on the predecessor's output is needed
                    if (!waited) pdl_wait();
                    waited = true;
                };
                auto load_q = [&]() {
                    have_q = true;
                    need_pred();
                    NFD_TRACE_MARK(TRK_OTHER + 10);
                    const int qs = it & 1;
                    if (it >= 2) ok = mbar_wait(q_empty + 8 * qs, ((it >> 1) - 1) & 1, status);
                    mbar_expect_tx(q_full + 8 * qs, A::Q_BYTES);
                    tma_load_3d(sQ + qs * A::Q_BYTES, &tmQ, q_full + 8 * qs, 0, w.j * D.T + w.qt * 128, w.h);
                };
                if (it > 0 && is_k) load_q();
                const int f = pl.bpf_div.div(w.b0);
                int kb = w.b0 - f * pl.BPF;
                int left = w.fr.first_new - (w.fr.win_first + f);      // frames until the pages that this pass writes
                int slot = w.fr.win_slot + f;
                if (slot >= D.R) slot -= D.R;
                int page = ((w.fr.stream * D.L + layer) * D.R + slot) * D.H + w.h;
                const int wrap = D.R * D.H;
                int to_wrap = D.R - slot;            // frames until the ring of this layer wraps
                for (int b = 0; b < w.nb && ok; ++b) {
                    if (lap > 0 || left <= 0) {
                        // a K stage is freed by an S product, which needs Q
                        if (!have_q) load_q();
                        need_pred();
                        if (lap > 0) ok = ok && mbar_wait(empty + 8 * st, (lap - 1) & 1, status);
                        if (!ok) break;
                    }
                    mbar_expect_tx(full + 8 * st, A::KV_BYTES);
                    tma_load_3d(ring + st * A::KV_BYTES, tm, full + 8 * st, 0, kb * KB, page);
                    if (++st == n_ring) st = 0, ++lap;
                    if (++kb == pl.BPF) {
                        kb = 0, --left, page += D.H;
                        if (--to_wrap == 0) page -= wrap, to_wrap = D.R;
                    }
                }
                if (!have_q && ok) load_q();
                ++it;
            }
        }
    } else if (warp == 1) {
        // ---------------- issuer of S = Q K^T ----------------
        if (elect_one()) {
            pdl_launch();
            constexpr uint32_t idesc_s = umma_idesc_bf16(128, KB);
            const uint32_t sQ = smem_u32(smem), sK = smem_u32(sKV);
            bool ok = true;
            int n = 0, it = 0;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                AttnItem w;
                w.set(item, sp, D, pl);
                if (w.nb == 0) continue;
                const int qs = it & 1;
                const uint64_t qd = umma_desc_k128(sQ + qs * A::Q_BYTES);
                ok = mbar_wait(q_full + 8 * qs, (it >> 1) & 1, status);
                for (int b = 0; b < w.nb && ok; ++b, ++n) {
                    const int st = n % A::NK;
                    // the accumulator is free when P V of the block three back, which reads P from it, is complete
                    if (n >= A::NK) {
                        const int m = n - A::NK;
                        ok = mbar_wait(v_empty + 8 * (m % A::NV), (m / A::NV) & 1, status);
                    }
                    ok = ok && mbar_wait(k_full + 8 * st, (n / A::NK) & 1, status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t kd = umma_desc_k128(sK + st * A::KV_BYTES);
#pragma unroll
                    for (int k4 = 0; k4 < 4; ++k4)
                        umma_bf16_ss(tmem + 128 * st, qd + 2 * k4, kd + 2 * k4, idesc_s, k4 != 0);
                    umma_commit(s_full + 8 * st);    // S(n) is ready; K's stage is free
                }
                umma_commit(q_empty + 8 * qs);
                ++it;
            }
        }
    } else if (warp == 2) {
        // ---------------- issuer of O += P V ----------------
        if (elect_one()) {
            constexpr uint32_t idesc_pv = umma_idesc_bf16_bmn(128, 64);
            const uint32_t sV = smem_u32(sKV) + A::NK * A::KV_BYTES;
            bool ok = true;
            int n = 0;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                AttnItem w;
                w.set(item, sp, D, pl);
                for (int b = 0; b < w.nb && ok; ++b, ++n) {
                    const int g = b & 1, sv = n % A::NV;
                    ok = mbar_wait(v_full + 8 * sv, (n / A::NV) & 1, status) &&
                         mbar_wait(p_full + 8 * (n % A::NK), (n / A::NK) & 1, status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t vd = umma_desc_k128(sV + sv * A::KV_BYTES);
                    const uint32_t tP = tmem + 128 * (n % A::NK);
#pragma unroll
                    for (int i = 0; i < KB / 16; ++i) {
                        // P: 16 keys = 8 columns of packed bf16 pairs; V: MN-major, 16 keys = 2 KiB per step
                        umma_bf16_ts(tmem + 384 + 64 * g, tP + 8 * i, vd + (uint64_t)(i * (2048 >> 4)), idesc_pv,
                                     (uint32_t)((b >> 1) != 0 || i != 0));
                    }
                    umma_commit(v_empty + 8 * sv);   // P V(n) is complete: V's stage and the accumulator are free
                }
            }
        }
    } else {
        // ---------------- softmax: one thread per query row, two groups ----------------
        const int g = (warp - A::SM_WARP0) >> 2;           // group: blocks b with (b & 1) == g
        const int quad = warp & 3;                         // tensor-memory lanes this warp may touch
        const int trow = quad * 32 + lane;
        const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
        const uint32_t tO = tmem + 384 + 64 * g + lane_off;
        const float c = (1.0f / sqrtf((float)D.dh)) * 1.4426950408889634f;   // softmax scale in the log2 domain
        bool ok = true;
        int n0 = 0;
        for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
            AttnItem w;
            w.set(item, sp, D, pl);
            if (w.nb == 0) continue;
            float m_run = -INFINITY, l_run = 0.f;
            int i = 0, kb = w.b0 + g;                      // block of the page, for the mask of its last block
            kb -= pl.bpf_div.div(kb) * pl.BPF;
            for (int b = g; b < w.nb; b += 2, ++i) {
                const int n = n0 + b;
                const uint32_t tS = tmem + 128 * (n % A::NK) + lane_off;
                const int nvalid = D.T - kb * KB;          // keys of this block (>= KB except at the end of a page)
                kb += 2;
                while (kb >= pl.BPF) kb -= pl.BPF;
                // (a warp whose wait has run out goes on without waiting, on whatever the accumulators hold: it has to take
                // part in the barriers below)
                ok = ok && mbar_wait(s_full + 8 * (n % A::NK), (n / A::NK) & 1, status);
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
                if (i == 0) {
                    // the group's first block: the row maximum itself is the reference
                    NFD_TRACE_MARK_T(TRK_OTHER + 11, 128);
                    m_run = row_max<KB>(tS) * c;
                }
                // One pass over S, 16 columns at a time with the next load in flight: p = exp2(S c - m) against the
                // reference maximum as it stands, packed to bf16 pairs in registers.  No maximum is taken: a reference
                // that is too low shows in the sum of the block, and any sum up to 2^16 is as exact as any other in
                // floating point.  Beyond that (after the first block: rare) the reference is raised, O is rescaled and
                // the pass repeated (once: against the block's own maximum no sum exceeds KB); S is intact until P is
                // stored.
                uint32_t pk[KB / 2];
                float ls;
                for (int pass = 0;; ++pass) {
                    const float c252 = c * (1.0f / EXP2_RANGE), b252 = (EXP2_LOW - m_run) * (1.0f / EXP2_RANGE);
                    float2 ls2[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                    uint32_t sa[16], sb[16];
                    tmem_ld16(tS, sa);
#pragma unroll
                    for (int cc = 0; cc < KB; cc += 16) {
                        uint32_t *cur = ((cc >> 4) & 1) ? sb : sa, *nxt = ((cc >> 4) & 1) ? sa : sb;
                        tmem_ld_wait();
                        if (cc + 16 < KB) tmem_ld16(tS + cc + 16, nxt);
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const float s0 = __uint_as_float(cur[2 * u]), s1 = __uint_as_float(cur[2 * u + 1]);
                            float2 p;
                            if (u == 3 || u == 7) {      // a quarter on the FMA pipe
                                p = exp2_fma2(s0, s1, c252, b252);
                            } else {
                                const float2 y = ffma2(make_float2(s0, s1), make_float2(c, c), make_float2(-m_run, -m_run));
                                p = make_float2(ex2_approx(y.x), ex2_approx(y.y));
                            }
                            ls2[u & 3] = fadd2(ls2[u & 3], p);
                            const __nv_bfloat162 hp = __floats2bfloat162_rn(p.x, p.y);
                            pk[(cc >> 1) + u] = *reinterpret_cast<const uint32_t *>(&hp);
                        }
                    }
                    ls = ((ls2[0].x + ls2[0].y) + (ls2[1].x + ls2[1].y)) + ((ls2[2].x + ls2[2].y) + (ls2[3].x + ls2[3].y));
                    const bool raise = ls > 65536.0f;
                    if (pass == 1 || !__any_sync(0xffffffffu, raise)) break;
                    const float m_blk = row_max<KB>(tS) * c;       // by the whole warp, whichever rows need it
                    const float m_new = raise ? fmaxf(m_run, m_blk) : m_run;
                    const float f = ex2_approx(m_run - m_new);     // 1 for rows that keep their reference
                    if (i > 0) {
                        // the previous P V product of this group must be complete before O is touched
                        ok = ok && mbar_wait(v_empty + 8 * ((n - 2) % A::NV), ((n - 2) / A::NV) & 1, status);
                        __syncwarp();
                        tc_fence_after();
#pragma unroll 1
                        for (int cc = 0; cc < 64; cc += 16) {
                            uint32_t r[16];
                            tmem_ld16(tO + cc, r);
                            tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * f);
                            tmem_st16(tO + cc, r);
                        }
                        tmem_st_wait();
                    }
                    l_run *= f;
                    m_run = m_new;
                }
                l_run += ls;
                // P over the first half of the columns it came from
#pragma unroll
                for (int cc = 0; cc < KB / 2; cc += 8) tmem_st8(tS + cc, pk + cc);
                tmem_st_wait();                            // P is in tensor memory
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(p_full + 8 * (n % A::NK));
            }
            NFD_TRACE_MARK_T(TRK_OTHER + 12, 128);
            // ---- this group's O (unnormalised, relative to m_run) and the fold of the two groups: group g finishes
            // columns 32 g .. 32 g + 31 and hands the other half of its accumulator over ----
            uint32_t Ob[32], Og[32];                       // own half, the other group's half
#pragma unroll
            for (int e = 0; e < 32; ++e) Ob[e] = Og[e] = 0u;
            if (i > 0) {                                   // (the same for the whole warp)
                const int bl = n0 + g + 2 * (i - 1);       // this group's last block
                ok = ok && mbar_wait(v_empty + 8 * (bl % A::NV), (bl / A::NV) & 1, status);
                __syncwarp();
                tc_fence_after();
                tmem_ld32(tO + 32 * g, Ob);
                tmem_ld32(tO + 32 * (g ^ 1), Og);
                tmem_ld_wait();
                tc_fence_before();
            }
            named_bar_sync(1, 256);                        // the last item's fold has been read
            s_ml[g * 128 + trow] = make_float2(m_run, l_run);
#pragma unroll
            for (int e = 0; e < 8; ++e)
                park[((g ^ 1) * 8 + e) * 128 + trow] = make_uint4(Og[4 * e], Og[4 * e + 1], Og[4 * e + 2], Og[4 * e + 3]);
            named_bar_sync(1, 256);
            n0 += w.nb;
            // (every rounding of the fold is spelled out: both groups, and whichever CTA merges the splits, have to
            // arrive at the same bits)
            const float2 ml0 = s_ml[trow], ml1 = s_ml[128 + trow];
            const float m_cta = fmaxf(ml0.x, ml1.x);       // (a group without a block has m = -inf, l = 0)
            const float w0 = ex2_approx(ml0.x - m_cta), w1 = ex2_approx(ml1.x - m_cta);
            const float l_cta = fmaf(ml0.y, w0, __fmul_rn(ml1.y, w1));
            const float w_own = g == 0 ? w0 : w1, w_oth = g == 0 ? w1 : w0;
            float O[32];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint4 v = park[(g * 8 + e) * 128 + trow];
                O[4 * e] = fmaf(__uint_as_float(Ob[4 * e]), w_own, __fmul_rn(__uint_as_float(v.x), w_oth));
                O[4 * e + 1] = fmaf(__uint_as_float(Ob[4 * e + 1]), w_own, __fmul_rn(__uint_as_float(v.y), w_oth));
                O[4 * e + 2] = fmaf(__uint_as_float(Ob[4 * e + 2]), w_own, __fmul_rn(__uint_as_float(v.z), w_oth));
                O[4 * e + 3] = fmaf(__uint_as_float(Ob[4 * e + 3]), w_own, __fmul_rn(__uint_as_float(v.w), w_oth));
            }
            NFD_TRACE_MARK_T(TRK_OTHER + 13, 128);
            bool write_out = true;
            float l_tot = l_cta;
            if (w.nsplit > 1) {
                // ---- publish this item's state; the CTA that finishes last merges the splits in split order ----
                const size_t item_q = ((size_t)w.j * D.H + w.h) * pl.QT + w.qt;
                uint8_t *states = reinterpret_cast<uint8_t *>(part_o) + item_q * pl.MAXSPLIT * ATTN_STATE_BYTES;
                {
                    uint8_t *st = states + (size_t)w.split * ATTN_STATE_BYTES;
                    float4 *so = reinterpret_cast<float4 *>(st) + g * 8 * 128 + trow;
#pragma unroll
                    for (int e = 0; e < 8; ++e) so[e * 128] = make_float4(O[4 * e], O[4 * e + 1], O[4 * e + 2], O[4 * e + 3]);
                    if (g == 0) reinterpret_cast<float2 *>(st + 128 * 64 * 4)[trow] = make_float2(m_cta, l_cta);
                }
                named_bar_sync(1, 256);
                if (threadIdx.x == 32 * A::SM_WARP0) {
                    __threadfence();
                    const unsigned int prev = atomicAdd(counters + item_q, 1u);
                    const int last = prev == (unsigned int)(w.nsplit - 1);
                    if (last) counters[item_q] = 0;        // ready for the next launch
                    __threadfence();
                    *last_flag = last;
                }
                NFD_TRACE_MARK_T(TRK_OTHER + 14, 128);
                named_bar_sync(1, 256);
                write_out = *last_flag != 0;
                if (write_out) {
                    // 16 columns at a time (registers); every state's loads of a chunk are in flight together
#pragma unroll
                    for (int hc = 0; hc < 2; ++hc) {
                        float acc[16], l = 0.f, mx = -INFINITY;
#pragma unroll
                        for (int e = 0; e < 16; ++e) acc[e] = 0.f;
                        for (int sidx = 0; sidx < w.nsplit; ++sidx) {
                            float2 ml = make_float2(m_cta, l_cta);
                            float4 v[4];
                            if (sidx == w.split) {
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    v[e] = make_float4(O[16 * hc + 4 * e], O[16 * hc + 4 * e + 1], O[16 * hc + 4 * e + 2], O[16 * hc + 4 * e + 3]);
                            } else {
                                const uint8_t *st = states + (size_t)sidx * ATTN_STATE_BYTES;
                                const float4 *so = reinterpret_cast<const float4 *>(st) + (g * 8 + hc * 4) * 128 + trow;
                                ml = __ldcg(reinterpret_cast<const float2 *>(st + 128 * 64 * 4) + trow);
#pragma unroll
                                for (int e = 0; e < 4; ++e) v[e] = __ldcg(so + e * 128);
                            }
                            const float mb = fmaxf(mx, ml.x);
                            // (a state without any key has m = -inf, l = 0: it must count for nothing)
                            const float fo = mx == mb ? 1.0f : ex2_approx(mx - mb);
                            const float wgt = ml.x == -INFINITY ? 0.f : ex2_approx(ml.x - mb);
                            mx = mb;
                            l = fmaf(ml.y, wgt, __fmul_rn(l, fo));
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                acc[4 * e] = fmaf(v[e].x, wgt, __fmul_rn(acc[4 * e], fo));
                                acc[4 * e + 1] = fmaf(v[e].y, wgt, __fmul_rn(acc[4 * e + 1], fo));
                                acc[4 * e + 2] = fmaf(v[e].z, wgt, __fmul_rn(acc[4 * e + 2], fo));
                                acc[4 * e + 3] = fmaf(v[e].w, wgt, __fmul_rn(acc[4 * e + 3], fo));
                            }
                        }
                        l_tot = l;
#pragma unroll
                        for (int e = 0; e < 16; ++e) O[16 * hc + e] = acc[e];
                    }
                }
            }
            const int row = w.qt * 128 + trow;
            if (write_out && row < D.T && g * 32 < D.dh) {
                const float inv = 1.0f / l_tot;
                bf16 *o = out + (size_t)(w.j * D.T + row) * D.d + w.h * D.dh + g * 32;
#pragma unroll
                for (int e = 0; e < 32; e += 8) {
                    float t[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) t[u] = O[e + u] * inv;
                    *reinterpret_cast<uint4 *>(o + e) = pack_bf16x8(t);
                }
            }
        }
    }
    NFD_TRACE_MARK_T(TRK_OTHER + 16, 128);
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, A::TMEM_COLS);
    NFD_TRACE_END(TRK_ATTN);
}
