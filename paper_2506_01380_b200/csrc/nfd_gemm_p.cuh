// Persistent tensor-core GEMM for passes of several frames, and for one frame's projection into the MLP (bf16 operands, fp32
// accumulation in tensor memory).
//
//   C[M,N] = A[M,K] * Wt[N,K]^T  followed by the row form of a fused epilogue functor.
//
// k_gemm_tc (nfd_gemm_tc.cuh) is built for one frame: one tile per CTA, the K range split over a cluster, and an
// epilogue that starts when the products have ended.  With several row blocks the tiles outnumber the SMs, and there a
// wave of it took 34k clocks per 128 x 256 tile of which the products need 8.4k: start, exit and the epilogue
// through a staging tile (16 items of 250 instructions per thread) are all exposed.  Here
//   - a CTA takes tiles blockIdx.x, + gridDim.x, ...; the producer and the issuer run on into the next tile;
//   - the accumulator has two halves of tensor memory, so that a tile's epilogue runs under the next one's products;
//   - the epilogue has one thread per row, 32 columns at a time straight from tensor memory, and touches global memory
//     through shared memory by TMA only: the residual stream and the rotary table come in, results go out in boxes of
//     32 rows x 32 columns.  (With loads and stores of the threads' own the epilogue was bound by the load-store unit,
//     about two clocks per line and instruction: 3.5k clocks for 16 columns of an output-projection tile, and turning
//     the rows around for whole lines cost 760 instructions per 32 x 32 outputs with GELU; now about 450.);
//   - a warp of its own fetches what depends on the column and the frame only (u, v / bias, gate, scale) into a table in
//     shared memory, a tile ahead.
// The K range is summed in the S segments of the one-frame plan (each in an accumulator of its own, added up in
// segment order in registers), so that a row's bits are those of k_gemm_tc.
//
// Warps 0 and 2 = TMA producers (activations, weights: one thread for both took 369 clocks per 64-element k-block), warp 1
// = tensor-memory allocation and UMMA issue, warp 3 = tables (and L2 prefetch of the next GEMM's weights), warps 4 and up
// = epilogue (two per tensor-memory lane quadrant, three for 96 columns, which share the columns).
#pragma once
#include "nfd_gemm_tc.cuh"

template <int BN, int FORM> struct GemmPCfg {
    static constexpr int A_BYTES = 128 * 128, B_BYTES = BN * 128, ST_BYTES = A_BYTES + B_BYTES;
    // a stage (64 elements of K) comes back about 1200 clocks after it was asked for: the ring holds about what the
    // products use in that time
    static constexpr int STAGES = BN <= 96 ? (FORM == FORM_MLP ? 6 : 5) : (BN <= 128 ? (FORM == FORM_MLP ? 5 : 4) : (BN <= 192 && FORM == FORM_MLP ? 4 : 3));
    static constexpr int RING_BYTES = STAGES * ST_BYTES;
    static constexpr int PARTS = BN == 96 ? 3 : 2;             // epilogue warps per tensor-memory lane quadrant
    static constexpr int EPI_WARP0 = 4, EPI_WARPS = 4 * PARTS;
    static constexpr int HC = BN / PARTS, NG = HC / 32;        // columns and 32-column groups per epilogue warp
    // side operands: the tile's rows of the rotary table (two halves of 32 floats), or of the residual stream
    static constexpr int SIDE_BYTES = FORM == FORM_QKV ? 2 * 128 * 128 : (FORM == FORM_RES ? 128 * BN * 4 : 0);
    static constexpr int NOUT = FORM == FORM_RES ? 1 : 2;      // result boxes of 32 x 32 bf16 per warp
    static constexpr int OUT_BYTES = EPI_WARPS * NOUT * 2048;
    static constexpr int MAX_FR = 3;                           // frames a 128-row tile may span (the caller checks)
    static constexpr int TAB_BYTES = MAX_FR * BN * (FORM == FORM_RES ? 3 : 2) * 4;    // one tile's table; two of them
    static constexpr int SMEM = RING_BYTES + SIDE_BYTES + OUT_BYTES + 2 * TAB_BYTES + EPI_WARPS * 256 /*row statistics*/ +
                                256 /*barriers*/ + 1024 /*align*/;
    static constexpr int TMEM_COLS = BN <= 128 ? 256 : 512;
    static constexpr int ACC_STRIDE = BN <= 128 ? 128 : 256;
    static constexpr int THREADS = 32 * (EPI_WARP0 + EPI_WARPS);
    static_assert(SMEM <= 232448, "shared memory of a CTA");
};

// The k-blocks of a CTA's tiles in order.
template <int BN> struct GemmIter {
    int tiles, n_nt, nkb, S, step;
    int t, seg, kb, kb1, m0, n0;
    __device__ __forceinline__ GemmIter(int M, int N, int K, int S_)
        : n_nt((N + BN - 1) / BN), nkb((K + 63) / 64), S(S_), step(gridDim.x), t(blockIdx.x) {
        tiles = ((M + 127) / 128) * n_nt;
        open();
    }
    __device__ __forceinline__ bool done() const { return t >= tiles; }
    __device__ __forceinline__ void open() {
        const int mt = t / n_nt;
        m0 = mt * 128, n0 = (t - mt * n_nt) * BN, seg = 0;
        open_seg();
    }
    __device__ __forceinline__ void open_seg() { kb = nkb * seg / S, kb1 = nkb * (seg + 1) / S; }
    __device__ __forceinline__ bool last() const { return t + step >= tiles && seg == S - 1 && kb + 1 >= kb1; }
    __device__ __forceinline__ void next() {
        if (++kb < kb1) return;
        if (++seg < S) {
            open_seg();
        } else {
            t += step;
            if (t < tiles) open();
        }
    }
};

// Result and side-operand maps: QKV q, k, v, rotary table; residual z, next operand; MLP hidden activation.
template <int BN, typename Epi, bool SPLIT>
__global__ void __launch_bounds__(GemmPCfg<BN, Epi::kForm>::THREADS, 1)
k_gemm_p(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
         const __grid_constant__ CUtensorMap tm0, const __grid_constant__ CUtensorMap tm1,
         const __grid_constant__ CUtensorMap tm2, const __grid_constant__ CUtensorMap tm3, int M, int N, int K, int S_rt,
         Epi epi, L2Prefetch pf, int T, int *status) {
    constexpr int FORM = Epi::kForm;
    using G = GemmPCfg<BN, FORM>;
    const int S = SPLIT ? S_rt : 1;
    extern __shared__ uint8_t smem_raw[];
    NFD_TRACE_T0();
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *s_side = smem + G::RING_BYTES, *s_out = s_side + G::SIDE_BYTES;
    float *s_tab = reinterpret_cast<float *>(s_out + G::OUT_BYTES);                    // [2][kTab][frame][BN]
    float2 *s_stat = reinterpret_cast<float2 *>(reinterpret_cast<uint8_t *>(s_tab) + 2 * G::TAB_BYTES);   // [warp][32]
    uint64_t *bars = reinterpret_cast<uint64_t *>(reinterpret_cast<uint8_t *>(s_stat) + G::EPI_WARPS * 256);
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * G::STAGES, acc_full = empty0 + 8 * G::STAGES,
                   acc_empty = acc_full + 16, tab_full = acc_empty + 16, tab_empty = tab_full + 16, side_full = tab_empty + 16;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * G::STAGES + 8 + G::EPI_WARPS);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        for (int s = 0; s < G::STAGES; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(acc_full + 8 * s, 1);
            mbar_init(acc_empty + 8 * s, G::EPI_WARPS);
            mbar_init(tab_full + 8 * s, 32);
            mbar_init(tab_empty + 8 * s, G::EPI_WARPS);
        }
        for (int s = 0; s < G::EPI_WARPS; ++s) mbar_init(side_full + 8 * s, 1);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), G::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0 || warp == 2) {
        // ---------------- TMA producers: activations (warp 0), weights (warp 2) ----------------
        if (elect_one()) {
            const bool is_a = warp == 0;
            const uint32_t ring = smem_u32(smem) + (is_a ? 0 : G::A_BYTES);
            const CUtensorMap *tm = is_a ? &tmA : &tmB;
            // test switch (see nfd_sm100.cuh): leave out the last stage, so that the wait for it runs out
            const int skip_last = is_a ? *reinterpret_cast<volatile int *>(status + 2) : 0;
            if (is_a) pdl_wait();                              // weights never depend on the previous kernel
            int s = 0, lap = 0;
            for (GemmIter<BN> i(M, N, K, S); !i.done(); i.next()) {
                if (skip_last && i.last()) break;
                if (lap > 0 && !mbar_wait(empty0 + 8 * s, (lap - 1) & 1, status)) break;
                if (is_a) mbar_expect_tx(full0 + 8 * s, G::ST_BYTES);
                tma_load_2d(ring + s * G::ST_BYTES, tm, full0 + 8 * s, i.kb * 64, is_a ? i.m0 : i.n0);
                if (++s == G::STAGES) s = 0, ++lap;
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            pdl_launch();
            constexpr uint32_t idesc = umma_idesc_bf16(128, BN);
            const uint32_t ring = smem_u32(smem);
            int s = 0, lap = 0, ab = 0;                        // ring stage, laps, accumulators filled
            bool ok = true, first = true;
            for (GemmIter<BN> i(M, N, K, S); !i.done(); i.next()) {
                const uint32_t acc = tmem_base + (ab & 1) * G::ACC_STRIDE;
                if (first && ab >= 2) {
                    ok = mbar_wait(acc_empty + 8 * (ab & 1), ((ab >> 1) - 1) & 1, status);
                    tc_fence_after();
                }
                ok = ok && mbar_wait(full0 + 8 * s, lap & 1, status);
                if (!ok) break;
                tc_fence_after();
                const uint64_t ad = umma_desc_k128(ring + s * G::ST_BYTES), bd = umma_desc_k128(ring + s * G::ST_BYTES + G::A_BYTES);
#pragma unroll
                for (int k4 = 0; k4 < 4; ++k4) umma_bf16_ss(acc, ad + 2 * k4, bd + 2 * k4, idesc, !(first && k4 == 0));
                umma_commit(empty0 + 8 * s);
                if (++s == G::STAGES) s = 0, ++lap;
                first = i.kb + 1 >= i.kb1;                     // the segment ends: its accumulator is complete
                if (first) umma_commit(acc_full + 8 * (ab & 1)), ++ab;
            }
        }
    } else if (warp == 3) {
        // ---------------- tables: (frame, column) values of the CTA's tiles, a tile ahead ----------------
        if (elect_one()) {
            // this CTA's slice of the next GEMM's weights, towards L2 in 8 KiB pieces
            const unsigned long long n_cta = gridDim.x, cta = blockIdx.x;
            const unsigned long long per = ((pf.bytes / n_cta + 15) / 16 + 1) * 16;
            unsigned long long b = cta * per, e = b + per;
            if (e > pf.bytes) e = pf.bytes;
            if (!pf.bytes) b = e = 0;
            for (; b < e; b += 8192) {
                const unsigned long long n = e - b < 8192 ? e - b : 8192;
                bulk_prefetch_l2(reinterpret_cast<const uint8_t *>(pf.ptr) + b, (uint32_t)n);
            }
        }
        __syncwarp();
        const int n_nt = (N + BN - 1) / BN, tiles = ((M + 127) / 128) * n_nt;
        bool ok = true;
        int it = 0;
        pdl_wait();
        for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++it) {
            const int tb = it & 1;
            const int mt = t / n_nt, m0 = mt * 128, n0 = (t - mt * n_nt) * BN;
            const int f0 = m0 / T, m_last = m0 + 127 < M ? m0 + 127 : M - 1;
            const int n_fr = m_last / T - f0 + 1;
            if (it >= 2) ok = mbar_wait(tab_empty + 8 * tb, ((it >> 1) - 1) & 1, status);
            if (!__all_sync(0xffffffffu, ok)) break;
            float *tab = s_tab + (size_t)tb * (G::TAB_BYTES / 4);
            int row[G::MAX_FR];
#pragma unroll
            for (int f = 0; f < G::MAX_FR; ++f) row[f] = epi.cond_row(f < n_fr ? f0 + f : f0);
#pragma unroll
            for (int f = 0; f < G::MAX_FR; ++f) {
                if (f >= n_fr) break;
                float v[BN / 32][Epi::kTab];                   // every load is issued before the first store
#pragma unroll
                for (int c = 0; c < BN / 32; ++c)
                    if (n0 + 32 * c + lane < N) epi.tab(row[f], n0 + 32 * c + lane, v[c]);
#pragma unroll
                for (int c = 0; c < BN / 32; ++c)
#pragma unroll
                    for (int x = 0; x < Epi::kTab; ++x) tab[(x * G::MAX_FR + f) * BN + 32 * c + lane] = v[c][x];
            }
            mbar_arrive(tab_full + 8 * tb);
        }
    } else {
        // ---------------- epilogue: one thread per row ----------------
        const int quad = warp & 3, part = (warp - G::EPI_WARP0) >> 2, ew = warp - G::EPI_WARP0;
        const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
        float2 *stat = s_stat + ew * 32;                       // of this warp's rows
        uint8_t *outb = s_out + ew * G::NOUT * 2048;
        const uint32_t sidebar = side_full + 8 * (FORM == FORM_QKV ? quad : ew);
        const int n_nt = (N + BN - 1) / BN, tiles = ((M + 127) / 128) * n_nt;
        bool ok = true, fold = false;
        if constexpr (Epi::kRowStats) fold = epi.ln.on();
        int ab = 0, it = 0, ob = 0;
        pdl_wait();
        for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++it) {
            const int tb = it & 1;
            const int mt = t / n_nt, m0 = mt * 128, n0 = (t - mt * n_nt) * BN + part * G::HC;
            const int mw = m0 + quad * 32, m = mw + lane;      // the warp's first row, this thread's row
            const int f0 = m0 / T, b1 = (f0 + 1) * T, b2 = b1 + T;     // first rows of the tile's second and third frame
            const bool valid = m < M;
            const int fo = valid ? (m >= b1) + (m >= b2) : 0;  // frame of the row, relative to f0
            const float *tab = s_tab + (size_t)tb * (G::TAB_BYTES / 4) + fo * BN + part * G::HC;
            // side operands of this tile (no copy is begun after a wait has run out)
            if constexpr (FORM == FORM_RES) {
                if (lane == 0 && ok) {
                    bulk_wait_read<0>();                       // the last tile's stores have read the buffers
                    mbar_expect_tx(sidebar, G::NG * 4096);
                    for (int g = 0; g < G::NG; ++g)
                        tma_load_2d(smem_u32(s_side) + (ew * G::NG + g) * 4096, &tm0, sidebar, n0 + 32 * g, mw);
                }
            }
            if constexpr (FORM == FORM_QKV) {
                // the rotary rows of a quadrant are shared by its warps: one loads them when all are done with the last
                if (it > 0) asm volatile("bar.sync %0, %1;" ::"r"(1 + quad), "n"(32 * G::PARTS) : "memory");
                if (part == 0 && lane == 0 && ok) {
                    const int nb = epi.D.dh > 32 ? 2 : 1;
                    mbar_expect_tx(sidebar, nb * 4096);
                    for (int h = 0; h < nb; ++h) tma_load_2d(smem_u32(s_side) + (quad * 2 + h) * 4096, &tm3, sidebar, 32 * h, mw);
                }
            }
            // pages of the tile's frames (QKV)
            int page[3] = {0, 0, 0}, fa = 0;
            bool one_frame = true;
            if constexpr (FORM == FORM_QKV) {
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const FrameDesc &f = epi.sp->fr[f0 + i < M / T ? f0 + i : f0];
                    page[i] = ((f.stream * epi.D.L + epi.layer) * epi.D.R + f.frame % epi.D.R) * epi.D.H;
                }
                fa = (mw >= b1) + (mw >= b2);
                const int ml = mw + 31 < M ? mw + 31 : M - 1;
                one_frame = (ml >= b1) + (ml >= b2) == fa;
            }
            if constexpr (Epi::kRowStats) {
                if (fold) {
                    // (mean, rstd) of the warp's rows from the producer's partial sums, 8 lanes per row; every load is issued
                    // before the first sum, the order of the additions is that of k_gemm_tc
                    const int sub = lane & 7, r0 = mw + (lane >> 3);
                    float2 pv[8][4];
#pragma unroll
                    for (int v = 0; v < 8; ++v)
#pragma unroll
                        for (int u = 0; u < 4; ++u) pv[v][u] = epi.ln.part(r0 + 4 * v < M ? r0 + 4 * v : -1, sub + 8 * u);
#pragma unroll
                    for (int v = 0; v < 8; ++v)
#pragma unroll
                        for (int u = 1; u < 4; ++u) pv[v][0].x += pv[v][u].x, pv[v][0].y += pv[v][u].y;
                    if (epi.ln.npart > 32) {                   // rows wider than 1024
                        for (int i = sub + 32; i < epi.ln.npart; i += 8)
#pragma unroll
                            for (int v = 0; v < 8; ++v) {
                                const float2 q = epi.ln.part(r0 + 4 * v < M ? r0 + 4 * v : -1, i);
                                pv[v][0].x += q.x, pv[v][0].y += q.y;
                            }
                    }
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                        for (int v = 0; v < 8; ++v) {
                            pv[v][0].x += __shfl_xor_sync(0xffffffffu, pv[v][0].x, o);
                            pv[v][0].y += __shfl_xor_sync(0xffffffffu, pv[v][0].y, o);
                        }
                    __syncwarp();
#pragma unroll
                    for (int v = 0; v < 8; ++v)
                        if (sub == v) stat[(lane >> 3) + 4 * v] = epi.ln.finish(pv[v][0].x, pv[v][0].y);
                    __syncwarp();
                }
            }
            float2 ms = make_float2(0.f, 1.f);
            if (fold) ms = stat[lane];
            // (a warp whose wait has run out goes on without waiting and stores nothing more)
            auto wait_acc = [&]() {
                ok = ok && mbar_wait(acc_full + 8 * (ab & 1), (ab >> 1) & 1, status);
                ok = __all_sync(0xffffffffu, ok);
                tc_fence_after();
            };
            auto free_acc = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_empty + 8 * (ab & 1));
                ++ab;
            };
            if constexpr (SPLIT) {
                // the segments' accumulators added up in order; the sum goes back into the last one's place
                uint32_t a[G::HC];
#pragma unroll 1
                for (int sg = 0; sg < S; ++sg) {
                    wait_acc();
                    const uint32_t ta = tmem_base + (ab & 1) * G::ACC_STRIDE + lane_off + part * G::HC;
#pragma unroll
                    for (int c = 0; c < G::HC; c += 16) {
                        uint32_t r[16];
                        tmem_ld16(ta + c, r);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            a[c + e] = sg == 0 ? r[e] : __float_as_uint(__uint_as_float(a[c + e]) + __uint_as_float(r[e]));
                    }
                    if (sg + 1 < S) {
                        free_acc();
                    } else {
#pragma unroll
                        for (int c = 0; c < G::HC; c += 16) tmem_st16(ta + c, a + c);
                        tmem_st_wait();
                    }
                }
            } else {
                wait_acc();
            }
            ok = ok && mbar_wait(tab_full + 8 * tb, (it >> 1) & 1, status);
            if (FORM != FORM_MLP) ok = ok && mbar_wait(sidebar, it & 1, status);
            ok = __all_sync(0xffffffffu, ok);
            const uint32_t ta = tmem_base + (ab & 1) * G::ACC_STRIDE + lane_off + part * G::HC;
#pragma unroll 1
            for (int g = 0; g < G::NG; ++g) {
                const int n = n0 + 32 * g;                     // columns n .. n + 31
                float a[32];
                tmem_ld32(ta + 32 * g, reinterpret_cast<uint32_t *>(a));
                tmem_ld_wait();
                if (g + 1 == G::NG) free_acc();
                if (n >= N || !ok || mw >= M) continue;        // (the same for the whole warp)
                const float4 *t0 = reinterpret_cast<const float4 *>(tab + 32 * g), *t1 = t0 + G::MAX_FR * BN / 4;
                if constexpr (FORM != FORM_RES) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float4 u = t0[i], w = t1[i];
                        a[4 * i] = fmaf(ms.y, fmaf(-ms.x, u.x, a[4 * i]), w.x);
                        a[4 * i + 1] = fmaf(ms.y, fmaf(-ms.x, u.y, a[4 * i + 1]), w.y);
                        a[4 * i + 2] = fmaf(ms.y, fmaf(-ms.x, u.z, a[4 * i + 2]), w.z);
                        a[4 * i + 3] = fmaf(ms.y, fmaf(-ms.x, u.w, a[4 * i + 3]), w.w);
                    }
                }
                // a free result box
                uint8_t *box = outb + ob * 2048;
                if (lane == 0) bulk_wait_read<G::NOUT - 1>();
                __syncwarp();
                // 16-byte word c of this thread's row in a box of 64-byte rows with the 64-byte swizzle
                auto put = [&](int c, const float *v) {
                    *reinterpret_cast<uint4 *>(box + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4)) = pack_bf16x8(v);
                };
                if constexpr (FORM == FORM_MLP) {
                    if (epi.act == 0) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            gelu4(a + 8 * c), gelu4(a + 8 * c + 4);
                            put(c, a + 8 * c);
                        }
                    } else {
                        // 16 results: rows of 32 bytes, 32-byte swizzle
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            *reinterpret_cast<uint4 *>(box + lane * 32 + ((c ^ ((lane >> 2) & 1)) << 4)) =
                                make_uint4(gated4(a + 16 * c), gated4(a + 16 * c + 4), gated4(a + 16 * c + 8), gated4(a + 16 * c + 12));
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&tm0, smem_u32(box), epi.act ? n >> 1 : n, mw);
                        bulk_commit();
                    }
                }
                if constexpr (FORM == FORM_QKV) {
                    const int d = epi.D.d, which = n >= 2 * d ? 2 : (n >= d ? 1 : 0), col = n - which * d;
                    const int lg = 31 - __clz(epi.D.dh), head = col >> lg, e = col & (epi.D.dh - 1);
                    if (which < 2) {
                        const uint8_t *cs = s_side + (quad * 2 + (e >> 5)) * 4096 + lane * 128;
#pragma unroll
                        for (int c = 0; c < 8; ++c) rope4(a + 4 * c, *reinterpret_cast<const float4 *>(cs + ((c ^ (lane & 7)) << 4)));
                    }
                    if (which == 0 || one_frame) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) put(c, a + 8 * c);
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            const int pg = fa == 0 ? page[0] : (fa == 1 ? page[1] : page[2]);
                            // rows beyond the end of the pass, or of the frame's page, fall outside the map
                            if (which == 0) tma_store_3d(&tm0, smem_u32(box), e, mw, head);
                            else tma_store_3d(which == 1 ? &tm1 : &tm2, smem_u32(box), e, mw - (f0 + fa) * T, pg + head);
                            bulk_commit();
                        }
                    } else {
                        // the warp's rows belong to two frames, hence two pages
                        if (valid) {
                            const int pg = fo == 0 ? page[0] : (fo == 1 ? page[1] : page[2]);
                            uint4 *dst = reinterpret_cast<uint4 *>((which == 1 ? epi.kc : epi.vc) +
                                                                   ((size_t)(pg + head) * T + (m - (f0 + fo) * T)) * epi.D.dh + e);
#pragma unroll
                            for (int c = 0; c < 4; ++c) dst[c] = pack_bf16x8(a + 8 * c);
                        }
                        // No box was used and no store is under way from one: the next group takes this one, whose last
                        // store has read it.  (The other one's may not have.)
                        continue;
                    }
                }
                if constexpr (FORM == FORM_RES) {
                    uint8_t *zb = s_side + (ew * G::NG + g) * 4096 + lane * 128;
                    const float4 *t2 = t1 + G::MAX_FR * BN / 4;
                    float2 sum[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        float z[8], o[8];
#pragma unroll
                        for (int x = 0; x < 2; ++x) {
                            float4 *zp = reinterpret_cast<float4 *>(zb + (((2 * c + x) ^ (lane & 7)) << 4));
                            const float4 zo = *zp, b = t0[2 * c + x], gt = t1[2 * c + x], sc = t2[2 * c + x];
                            const float *v = a + 8 * c + 4 * x;
                            float *zn = z + 4 * x;
                            zn[0] = fmaf(gt.x, v[0] + b.x, zo.x), zn[1] = fmaf(gt.y, v[1] + b.y, zo.y);
                            zn[2] = fmaf(gt.z, v[2] + b.z, zo.z), zn[3] = fmaf(gt.w, v[3] + b.w, zo.w);
                            *zp = make_float4(zn[0], zn[1], zn[2], zn[3]);
                            o[4 * x] = zn[0] * sc.x, o[4 * x + 1] = zn[1] * sc.y;
                            o[4 * x + 2] = zn[2] * sc.z, o[4 * x + 3] = zn[3] * sc.w;
                        }
                        const float2 sa = sums4(z), sb = sums4(z + 4);
                        sum[c] = make_float2(sa.x + sb.x, sa.y + sb.y);
                        if (epi.a_out) put(c, o);
                    }
                    if (epi.stats && valid)
                        epi.stats[(size_t)m * (epi.D.d >> 5) + (n >> 5)] = make_float2((sum[0].x + sum[1].x) + (sum[2].x + sum[3].x),
                                                                                      (sum[0].y + sum[1].y) + (sum[2].y + sum[3].y));
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&tm0, smem_u32(s_side) + (ew * G::NG + g) * 4096, n, mw);
                        if (epi.a_out) tma_store_2d(&tm1, smem_u32(box), n, mw);
                        bulk_commit();
                    }
                }
                ob = ob + 1 == G::NOUT ? 0 : ob + 1;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(tab_empty + 8 * tb);
        }
        if (lane == 0) bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, G::TMEM_COLS);
    NFD_TRACE_END(TRK_GEMM + 16 * (int)(K > 2048) + 32 * (int)(N / 1024));
}
