// Tensor-core path of libnfd (bf16 only): tcgen05/TMEM GEMM fed by TMA with the
// fused epilogues of nfd_kernels.cuh, and the dispatch hooks used by
// nfd_api.cu.  fast_gemm / fast_attention return false when they do not handle
// a case; the caller then launches the plain kernels.
#pragma once
#include <atomic>
#include <map>
#include <tuple>
#include <type_traits>
#include <utility>

#include "nfd_sm100.cuh"
#include "nfd_gemm_tc.cuh"
#include "nfd_gemm_p.cuh"
#include "nfd_attn_tc.cuh"

#define NFD_MAX_DEVICES 64       // devices of a process that the allocation-free call knows

typedef CUresult (*PFN_encodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                    const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct FastState {
    bool ready = false;
    PFN_encodeTiled encode = nullptr;
    int *d_status = nullptr;
    int n_sm = 0, dh = 0;
    size_t a_rows = 0;     // rows of every activation buffer (NFD_MAX_PASS_FRAMES * T)
    AttnPlan plan;         // KB == 0: tensor-core attention not available for this shape
    float *part_o = nullptr;           // per-split states of the attention kernel: [query tile][split] x ATTN_STATE_BYTES
    unsigned int *attn_counters = nullptr;   // one per query tile; zero between launches
    size_t cache_pages = 0;            // (stream, layer, ring slot, head) pages of T rows
    std::map<std::tuple<const void *, int, int, int>, CUtensorMap> maps;   // (ptr, rows, cols, box_rows)
};

static PFN_encodeTiled get_encode_fn() {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
        qres != cudaDriverEntryPointSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return (PFN_encodeTiled)fn;
}

static int fast_create(FastState &fs, const Dims &D, bool bf16_mode, cudaStream_t st, int *d_status) {
    (void)st;
    fs.ready = false;
    fs.d_status = d_status;
    fs.a_rows = (size_t)NFD_MAX_PASS_FRAMES * D.T, fs.dh = D.dh;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&fs.n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return NFD_E_CUDA;
    }
    if (!bf16_mode) return NFD_OK;
    fs.encode = get_encode_fn();
    if (!fs.encode) {
        // no silent change of path: without tensor maps a bf16 context would run the plain validation kernels
        fprintf(stderr, "libnfd: the driver does not provide cuTensorMapEncodeTiled; a bf16 context needs it\n");
        return NFD_E_CUDA;
    }
    fs.ready = true;
    // attention plan: any number of tokens per frame, head dimension 64 or 32
    AttnPlan pl;
    fs.cache_pages = (size_t)D.n_streams * D.L * D.R * D.H;
    if ((D.dh == 64 || D.dh == 32) && fs.cache_pages < 0x7fffffffull) {
        attn_blocks(pl, D.T);
        attn_split_plan(pl, D.H * pl.QT, D.n_streams, (D.W + 1) * pl.BPF, fs.n_sm);
        if (attn_divisors(pl, NFD_MAX_PASS_FRAMES, D.W, fs.n_sm)) {
            if (pl.SP > 0 && pl.MAXSPLIT > 1) {
                // (the largest pass of this context: per stream a speculation and the deferred frames of the last one)
                const int nf_max = D.n_streams * (D.R - D.W);
                const size_t tiles = (size_t)(nf_max < NFD_MAX_PASS_FRAMES ? nf_max : NFD_MAX_PASS_FRAMES) * pl.SP;
                if (cudaMalloc((void **)&fs.part_o, tiles * pl.MAXSPLIT * (size_t)ATTN_STATE_BYTES) != cudaSuccess ||
                    cudaMalloc((void **)&fs.attn_counters, tiles * sizeof(unsigned int)) != cudaSuccess ||
                    cudaMemset(fs.attn_counters, 0, tiles * sizeof(unsigned int)) != cudaSuccess) {
                    cudaGetLastError();
                    return NFD_E_NOMEM;
                }
            }
            fs.plan = pl;
        }
    }
    return NFD_OK;
}

static void fast_destroy(FastState &fs) {
    fs.maps.clear();
    if (fs.part_o) cudaFree(fs.part_o);
    if (fs.attn_counters) cudaFree(fs.attn_counters);
    fs.part_o = nullptr, fs.attn_counters = nullptr;
    fs.ready = false;
}

// 2D bf16 tensor map [rows][cols], box = 64 columns (128 bytes) x box_rows, 128-byte swizzle.
static const CUtensorMap *get_map_2d(FastState &fs, const void *ptr, int rows, int cols, int box_rows) {
    auto key = std::make_tuple(ptr, rows, cols, box_rows);
    auto it = fs.maps.find(key);
    if (it != fs.maps.end()) return &it->second;
    CUtensorMap m;
    cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t gstr[1] = {(cuuint64_t)cols * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fs.encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), gdim, gstr, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        fprintf(stderr, "libnfd: cuTensorMapEncodeTiled failed (%d) for [%d x %d] box %d\n", (int)r, rows, cols,
                box_rows);
        return nullptr;
    }
    return &fs.maps.emplace(key, m).first->second;
}

// 3D bf16 tensor map [pages][rows][cols] for the attention operands: box = 1 page x box_rows x 64 columns, 128-byte
// swizzle.  Rows beyond a page's end and, for head dimension 32, columns beyond the row's end read as zero.
static bool encode_map_3d(PFN_encodeTiled encode, CUtensorMap *m, const void *ptr, size_t pages, int rows, int cols,
                          int box_rows) {
    cuuint64_t gdim[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)pages};
    cuuint64_t gstr[2] = {(cuuint64_t)cols * 2, (cuuint64_t)cols * 2 * rows};
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), gdim, gstr, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        fprintf(stderr, "libnfd: cuTensorMapEncodeTiled failed (%d) for [%zu x %d x %d] box %d\n", (int)r, pages, rows,
                cols, box_rows);
    return r == CUDA_SUCCESS;
}

// ---------------------------------------------------------------------------
// Kernel launch, with programmatic stream serialisation where `early` is set (the kernel may start while its
// predecessor runs) and with an optional cluster along x.  Works the same under stream capture.
// ---------------------------------------------------------------------------
template <typename... KArgs, typename... Args>
static cudaError_t launch_kernel(bool early, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 int cluster_x, Args &&...args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid, cfg.blockDim = block, cfg.dynamicSmemBytes = smem, cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int na = 0;
    if (early) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    if (cluster_x > 1) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = (unsigned)cluster_x, attr[na].val.clusterDim.y = 1, attr[na].val.clusterDim.z = 1;
        ++na;
    }
    cfg.attrs = attr, cfg.numAttrs = (unsigned)na;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              int cluster_x, Args &&...args) {
    return launch_kernel(true, kern, grid, block, smem, st, cluster_x, std::forward<Args>(args)...);
}

// More than 48 KB of shared memory for a kernel, on the current device.  Asked for before every launch: the limit belongs to
// a device, and a process may have contexts on several.
template <typename... KArgs> static bool allow_smem(void (*kern)(KArgs...), int bytes) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}

// ---------------------------------------------------------------------------
// Tile width BN and cluster split S of a GEMM [M x N x K].
// ---------------------------------------------------------------------------
struct GemmPlan {
    int BN, S;
    bool p;        // k_gemm_p instead of k_gemm_tc
};

// Tile width of k_gemm_p for a GEMM [M x N x K] with a K split of S, or 0 where k_gemm_tc is the better one.  The line
// lies where the row blocks times 128-wide column tiles fill the machine; measured on a 148-SM B200, k_gemm_tc -> k_gemm_p
// in us with launch, for the projections into QKV and the MLP (K 768 to 1536): 72 tiles 12.9 -> 14.4, 96 tiles 14.9 ->
// 14.8, 108 tiles 14.7 -> 13.0, 129 tiles 16.5 -> 14.6, 192 tiles 20.6 -> 16.9, 264 tiles 24 -> 19, 672 tiles 52 -> 32.
// For those onto the residual stream, out of attention / out of the MLP, k_gemm_tc -> k_gemm_p 96 wide, 128 wide (the rule
// below takes the former or the latter), frames of 336 rows: hidden 1024, MLP 4096: 48 tiles of 128 columns 13.6 / 18.8 ->
// 14.7 / 23.1, 14.8 / 26.9; 64 tiles 14.5 / 20.8 -> 14.7 / 23.2, 15.1 / 27.0; 88 tiles 15.8 / 34.1 -> 14.7 / 23.6, 15.2 /
// 27.5; 112 tiles 18.8 / 34.3 -> 17.1 / 33.9, 15.5 / 27.7; 168 tiles 29.5 / 48.4 -> 20.1 / 37.4, 20.9 / 40.0.  Hidden 1536,
// MLP 4096: 72 tiles 17.0 / 21.6 -> 16.9 / 23.9, 18.8 / 28.0; 96 tiles 20.6 / 34.1 -> 18.7 / 24.3, 19.9 / 28.1.  Hidden 768,
// MLP 2048: 66 tiles 13.2 / 15.9 -> 12.7 / 16.7, 14.4 / 18.0; 84 tiles 14.7 / 17.8 -> 13.3 / 16.7, 14.4 / 18.5; 114 tiles
// 16.8 / 20.0 -> 15.5 / 22.5, 14.7 / 18.8.
static int gemm_p_width(int n_sm, int form, int T, int dh, int M, int N, int K, int S) {
    // a 128-row tile must not span more frames than the kernel keeps tables for; rotary rows of 64 floats at most
    if (form == FORM_NONE || 127 / T + 2 > GemmPCfg<128, FORM_MLP>::MAX_FR || (form == FORM_QKV && dh > 64)) return 0;
    const int mt = (M + 127) / 128, t128 = mt * ((N + 127) / 128);
    if (form == FORM_RES) {
        if (t128 < (88 * n_sm) / 148) return 0;
        // 96 columns unless they need a wave more.  128 -> 96 wide, us with launch, K = 4096: 88 -> 121 tiles 27.5 -> 23.6,
        // 152 -> 209 38.5 -> 36.2, 168 -> 231 40.0 -> 37.4 (K = 1024: 20.9 -> 20.1); a wave more: 112 -> 154 27.7 -> 33.9,
        // 252 -> 336 48.6 -> 54.8
        const int t96 = mt * ((N + 95) / 96);
        return (t96 + n_sm - 1) / n_sm <= (t128 + n_sm - 1) / n_sm ? 96 : 128;
    }
    // Into the MLP, where k_gemm_tc would take 96 columns in one wave (its epilogue, GELU or gate behind a staging tile, is the
    // longer half of it): from 100 CTAs on k_gemm_p in the same tiles.  One frame, us: 310M class (129 tiles) 5350 -> 5332,
    // hidden 768 with a gated MLP (129) 2315 -> 2297; 86 tiles (220 tokens) 4203 -> 4211, 12 tiles (64 tokens) 299 -> 307.
    const int t96 = mt * ((N + 95) / 96);
    if (form == FORM_MLP && S == 1 && t96 <= n_sm && t96 >= (100 * n_sm) / 148 && mt * ((N + 63) / 64) > n_sm) return 96;
    if (t128 < (100 * n_sm) / 148) return 0;
    if (S > 1) return 128;
    // microseconds: a base and a wave, fitted to K = 768, 1024 and 1536 (within 2 us up to ten waves)
    const float nkb = (float)((K + 63) / 64);
    const int bns[3] = {128, 192, 256};
    const float base[3] = {10.3f, 10.9f, 12.2f};
    const float wave[3] = {nkb * 0.231f > 4.2f ? nkb * 0.231f : 4.2f, nkb * 0.25f + 1.4f, nkb * 0.4f};
    int best = 128;
    float t_best = 1e30f;
    for (int i = 0; i < 3; ++i) {
        const int tiles = mt * ((N + bns[i] - 1) / bns[i]);
        const float t = base[i] + wave[i] * (float)((tiles + n_sm - 1) / n_sm);
        if (t < t_best) t_best = t, best = bns[i];
    }
    return best;
}
// CTAs of k_gemm_tc that can be resident at once: one per SM, less what clusters cannot use (a cluster lives inside one
// GPC; on a 148-SM B200 cudaOccupancyMaxActiveClusters gives 148 CTAs for clusters of 1 and 2, 132 for clusters of 4; the
// formula goes through this one measured point, so that plans, and with them the bits, follow from sizes alone).
static int gemm_slots(int n_sm, int S) { return S >= 4 ? (n_sm / 4 - 4) * 4 : n_sm; }
// The narrowest tile whose CTAs fit the machine at once, 0 if none does.
static int gemm_tc_width(int n_sm, int M, int N, int S) {
    const int bns[4] = {32, 64, 96, 128};
    for (int bn : bns) {
        if (bn > 32 && bn > N) break;
        if ((long long)((M + 127) / 128) * ((N + bn - 1) / bn) * S <= gemm_slots(n_sm, S)) return bn;
    }
    return 0;
}
// K split and tile width of a GEMM [M x N x K].  The split is chosen for a one-frame pass (T rows) and kept for every M:
// the order in which the K range is summed, and with it every bit of the result, must not depend on how many frames share
// a pass.  The rules go by sizes alone, so that every process sums alike.  Measured on one B200 (us with launch), one
// frame of 336 rows unless stated:
//   split: K = 4096 onto 1024 columns: 1, 2, 4 -> 17.7, 15.6, 16.9 (two frames 20.5, 18.8, 23.5; 96 rows 17.0, 14.5,
//     12.8); K = 2736: 15.9, 14.8, 15.6; K = 2048 onto 768: 12.8, 12.5, 14.3; K = 1024: 11.1, 12.8, 14.2.  Hence none
//     below 40 blocks of 64; two CTAs to a tile above, four where there is a single row block.
//   width: the narrowest that needs one wave (the CTAs that a wider tile saves stay idle, and its epilogue is longer):
//     K = 1024 onto 1024 columns 32, 64, 96 wide 11.1, 12.8, 14.8; onto 3072 columns 64, 96, 128 wide 12.7, 14.8, 15.5;
//     two frames, K = 4096 in two, 96, 128 wide (64 needs two waves) 18.8, 20.3, 25.1.
static GemmPlan plan_gemm(const FastState &fs, int M, int N, int K, int form) {
    const int T = (int)(fs.a_rows / NFD_MAX_PASS_FRAMES), nkb = (K + 63) / 64;
    int S = nkb < 40 ? 1 : (T > 128 ? 2 : 4);
    while (S > 1 && !gemm_tc_width(fs.n_sm, T, N, S)) S /= 2;
    if (const int bn = gemm_p_width(fs.n_sm, form, T, fs.dh, M, N, K, S)) return {bn, S, true};
    const int bn = gemm_tc_width(fs.n_sm, M, N, S);
    return {bn ? bn : (N >= 128 ? 128 : 32), S, false};
}

template <int BN, typename Epi, int SC>
static bool launch_gemm_tc_sc(FastState &fs, cudaStream_t st, const bf16 *A, const bf16 *Wt, int M, int N, int K, int S,
                              Epi epi, L2Prefetch pf) {
    using G = GemmCfg<BN>;
    auto kern = k_gemm_tc<BN, Epi, SC>;
    if (!allow_smem(kern, G::SMEM)) return false;
    const CUtensorMap *ma = get_map_2d(fs, A, (int)fs.a_rows, K, 128);
    const CUtensorMap *mb = get_map_2d(fs, Wt, N, K, BN);
    if (!ma || !mb) return false;
    dim3 grid(((N + BN - 1) / BN) * S, (M + 127) / 128);
    // Always early: in a pass the kernels before the first projection release their dependents after their own wait, so that
    // the descriptor and the modulation cache, which this one reads before its wait, are complete.
    cudaError_t e = launch_pdl(kern, grid, dim3(G::THREADS), (size_t)G::SMEM, st, S, *ma, *mb, M, N, K, S, epi, pf,
                               fs.d_status);
    if (e != cudaSuccess) {
        fprintf(stderr, "libnfd: tensor-core GEMM launch failed (BN %d, S %d): %s\n", BN, S, cudaGetErrorString(e));
        cudaGetLastError();
        return false;
    }
    return true;
}

// the unsplit case has a kernel of its own (see k_gemm_tc)
template <int BN, typename Epi>
static bool launch_gemm_tc(FastState &fs, cudaStream_t st, const bf16 *A, const bf16 *Wt, int M, int N, int K, int S,
                           Epi epi, L2Prefetch pf) {
    if (S == 1) return launch_gemm_tc_sc<BN, Epi, 1>(fs, st, A, Wt, M, N, K, S, epi, pf);
    return launch_gemm_tc_sc<BN, Epi, 0>(fs, st, A, Wt, M, N, K, S, epi, pf);
}

// Tensor map [pages][rows][cols] (pages = 0: two dimensions) with boxes of 32 rows x box_cols, for the results and side
// operands of k_gemm_p; the swizzle spans the box's row.
static bool encode_map_box(const FastState &fs, CUtensorMap *m, const void *ptr, bool f32, size_t pages, int rows, int cols,
                           int box_cols) {
    const int es = f32 ? 4 : 2;
    cuuint64_t gdim[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)pages};
    cuuint64_t gstr[2] = {(cuuint64_t)cols * es, (cuuint64_t)cols * es * rows};
    cuuint32_t box[3] = {(cuuint32_t)box_cols, 32, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    const int bytes = box_cols * es;
    CUresult r = fs.encode(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, pages ? 3 : 2,
                           const_cast<void *>(ptr), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B),
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) fprintf(stderr, "libnfd: cuTensorMapEncodeTiled failed (%d) for a box of 32 x %d\n", (int)r, box_cols);
    return r == CUDA_SUCCESS;
}
static bool epi_maps(const FastState &fs, const EpiQKV<bf16> &e, int M, int, CUtensorMap *m) {
    return encode_map_box(fs, m, e.q, false, e.D.H, M, e.D.dh, 32) &&
           encode_map_box(fs, m + 1, e.kc, false, fs.cache_pages, e.D.T, e.D.dh, 32) &&
           encode_map_box(fs, m + 2, e.vc, false, fs.cache_pages, e.D.T, e.D.dh, 32) &&
           encode_map_box(fs, m + 3, e.rope_cs, true, 0, M, e.D.dh, 32);
}
static bool epi_maps(const FastState &fs, const EpiGateRes<bf16> &e, int M, int, CUtensorMap *m) {
    return encode_map_box(fs, m, e.z, true, 0, M, e.D.d, 32) && (!e.a_out || encode_map_box(fs, m + 1, e.a_out, false, 0, M, e.D.d, 32));
}
static bool epi_maps(const FastState &fs, const EpiGelu<bf16> &e, int M, int N, CUtensorMap *m) {
    return encode_map_box(fs, m, e.out, false, 0, M, e.act ? N / 2 : N, e.act ? 16 : 32);
}

template <int BN, typename Epi, bool SPLIT>
static bool launch_gemm_p(FastState &fs, cudaStream_t st, const bf16 *A, const bf16 *Wt, int M, int N, int K, int S,
                          Epi epi, L2Prefetch pf) {
    using G = GemmPCfg<BN, Epi::kForm>;
    auto kern = k_gemm_p<BN, Epi, SPLIT>;
    if (!allow_smem(kern, G::SMEM)) return false;
    const CUtensorMap *ma = get_map_2d(fs, A, (int)fs.a_rows, K, 128);
    const CUtensorMap *mb = get_map_2d(fs, Wt, N, K, BN);
    CUtensorMap me[4];
    memset(me, 0, sizeof(me));
    if (!ma || !mb || !epi_maps(fs, epi, M, N, me)) return false;
    const int tiles = ((M + 127) / 128) * ((N + BN - 1) / BN);
    cudaError_t e = launch_pdl(kern, dim3(tiles < fs.n_sm ? tiles : fs.n_sm), dim3(G::THREADS), (size_t)G::SMEM, st, 1, *ma,
                               *mb, me[0], me[1], me[2], me[3], M, N, K, S, epi, pf, (int)(fs.a_rows / NFD_MAX_PASS_FRAMES),
                               fs.d_status);
    if (e != cudaSuccess) {
        fprintf(stderr, "libnfd: persistent GEMM launch failed (BN %d, S %d): %s\n", BN, S, cudaGetErrorString(e));
        cudaGetLastError();
        return false;
    }
    return true;
}
template <typename Epi>
static bool launch_gemm_p_any(FastState &fs, cudaStream_t st, const bf16 *A, const bf16 *Wt, int M, int N, int K, int BN,
                              int S, Epi epi, L2Prefetch pf) {
    if constexpr (Epi::kForm == FORM_RES) {
        if (BN == 96) return S > 1 ? launch_gemm_p<96, Epi, true>(fs, st, A, Wt, M, N, K, S, epi, pf)
                                   : launch_gemm_p<96, Epi, false>(fs, st, A, Wt, M, N, K, S, epi, pf);
    }
    if (S > 1) return launch_gemm_p<128, Epi, true>(fs, st, A, Wt, M, N, K, S, epi, pf);
    if constexpr (Epi::kForm == FORM_MLP) {
        if (BN == 96) return launch_gemm_p<96, Epi, false>(fs, st, A, Wt, M, N, K, S, epi, pf);
    }
    if constexpr (Epi::kForm != FORM_RES) {
        if (BN == 256) return launch_gemm_p<256, Epi, false>(fs, st, A, Wt, M, N, K, S, epi, pf);
        if (BN == 192) return launch_gemm_p<192, Epi, false>(fs, st, A, Wt, M, N, K, S, epi, pf);
    }
    return launch_gemm_p<128, Epi, false>(fs, st, A, Wt, M, N, K, S, epi, pf);
}

template <typename TS, typename Epi>
static bool fast_gemm(bool enabled, FastState &fs, cudaStream_t st, const TS *A, const TS *Wt, int M, int N, int K,
                      Epi epi, L2Prefetch pf) {
    if constexpr (!std::is_same<TS, bf16>::value) {
        return false;
    } else {
        if (!enabled || !fs.ready) return false;
        if (K % 8 || K < 64 || N < 32 || (N & 7)) return false;
        if (((uintptr_t)A & 15) || ((uintptr_t)Wt & 15)) return false;
        const GemmPlan pl = plan_gemm(fs, M, N, K, Epi::kForm);
        if constexpr (Epi::kForm != FORM_NONE) {
            if (pl.p) return launch_gemm_p_any<Epi>(fs, st, A, Wt, M, N, K, pl.BN, pl.S, epi, pf);
        }
        switch (pl.BN) {
            case 128: return launch_gemm_tc<128, Epi>(fs, st, A, Wt, M, N, K, pl.S, epi, pf);
            case 96: return launch_gemm_tc<96, Epi>(fs, st, A, Wt, M, N, K, pl.S, epi, pf);
            case 64: return launch_gemm_tc<64, Epi>(fs, st, A, Wt, M, N, K, pl.S, epi, pf);
            default: return launch_gemm_tc<32, Epi>(fs, st, A, Wt, M, N, K, pl.S, epi, pf);
        }
    }
}

template <int KB, bool DEALT>
static int launch_attn_tc(bool early, int test_skip, PFN_encodeTiled encode, int n_sm, cudaStream_t st, const StepParams *sp, const Dims &D, int nf,
                          int layer, const AttnPlan &pl, size_t pages, const bf16 *q, const bf16 *kc, const bf16 *vc,
                          bf16 *out, float *part_o, unsigned int *counters, int *status) {
    using A = AttnCfg<KB>;
    auto kern = k_attn_tc<KB, DEALT>;
    constexpr int smem = DEALT ? A::DEALT_SMEM : A::SMEM;
    if (!allow_smem(kern, smem)) return 0;
    CUtensorMap mq, mk, mv;
    if (!encode_map_3d(encode, &mq, q, D.H, nf * D.T, D.dh, 128) || !encode_map_3d(encode, &mk, kc, pages, D.T, D.dh, KB) ||
        !encode_map_3d(encode, &mv, vc, pages, D.T, D.dh, KB))
        return 0;
    cudaError_t e = launch_kernel(early, kern, dim3(pl.grid), dim3(A::THREADS), (size_t)smem, st, 1, mq, mk, mv, sp, D, layer, pl, out, part_o, counters, status, test_skip);
    if (e != cudaSuccess) {
        fprintf(stderr, "libnfd: tensor-core attention launch failed: %s\n", cudaGetErrorString(e));
        cudaGetLastError();
        return 0;
    }
    return 1;
}

// Clusters of k CTAs of k_attn_own that device `dev`, the current one, holds at once (0: it runs none).  Asked for once.
template <int KB> static int attn_own_clusters(int dev, int k) {
    static std::atomic<int> known[NFD_MAX_DEVICES][9];                     // and one
    int n = known[dev][k].load(std::memory_order_relaxed);
    if (n) return n - 1;
    using A = AttnCfg<KB>;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(k), cfg.blockDim = dim3(A::THREADS), cfg.dynamicSmemBytes = A::OWN_SMEM;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)k, attr.val.clusterDim.y = 1, attr.val.clusterDim.z = 1;
    cfg.attrs = &attr, cfg.numAttrs = 1;
    if (!allow_smem(k_attn_own<KB>, A::OWN_SMEM) || cudaOccupancyMaxActiveClusters(&n, k_attn_own<KB>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    known[dev][k].store(n + 1, std::memory_order_relaxed);
    return n;
}
// Test switches of the allocation-free call: K does not come, the launch of clusters is refused.
enum { NFD_TEST_SKIP = 1, NFD_TEST_REFUSE = 2 };
// Split key ranges of the caller's pages: see k_attn_own.
template <int KB>
static bool launch_attn_own(int test, PFN_encodeTiled encode, cudaStream_t st, const StepParams *sp, int nf, const Dims &D, AttnPlan pl,
                            size_t pages, const bf16 *q, const bf16 *kc, const bf16 *vc, bf16 *out, int *status) {
    using A = AttnCfg<KB>;
    auto kern = k_attn_own<KB>;
    constexpr int smem = A::OWN_SMEM;
    if (!allow_smem(kern, smem)) return false;
    CUtensorMap mq, mk, mv;
    if (!encode_map_3d(encode, &mq, q, D.H, nf * D.T, D.dh, 128) || !encode_map_3d(encode, &mk, kc, pages, D.T, D.dh, KB) ||
        !encode_map_3d(encode, &mv, vc, pages, D.T, D.dh, KB))
        return false;
    attn_deal(pl, nf, 0x7fffffff);                         // an item to a CTA
    // (test switch: a cluster size that the runtime refuses)
    const cudaError_t e = launch_kernel(false, kern, dim3(pl.grid), dim3(A::THREADS), (size_t)smem, st,
                                        test & NFD_TEST_REFUSE ? 64 : pl.MAXSPLIT, mq, mk, mv, sp, D, pl, out, status, test & NFD_TEST_SKIP);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess;
}

// Attention of a pass by plan `pl` over `pages` (stream, layer, ring slot, head) pages of K and V.  `early`: the kernel may
// start before its predecessor ends.  It reads the pass descriptor, and pages that the pass does not write, without waiting
// for the predecessor: that must not be the kernel that writes them.  `test_skip`: the test switch of nfd_sm100.cuh.
static int launch_attn_plan(bool early, int test_skip, PFN_encodeTiled encode, int n_sm, cudaStream_t st, const StepParams *sp, const Dims &D, int nf,
                            int layer, AttnPlan pl, size_t pages, const bf16 *q, const bf16 *kc, const bf16 *vc,
                            bf16 *out, float *part_o, unsigned int *counters, int *status) {
    attn_deal(pl, nf, n_sm);
    auto go = [&](auto kb, auto dealt) {
        return launch_attn_tc<decltype(kb)::value, decltype(dealt)::value>(early, test_skip, encode, n_sm, st, sp, D, nf, layer, pl, pages, q, kc,
                                                                           vc, out, part_o, counters, status);
    };
    auto width = [&](auto dealt) {
        switch (pl.KB) {
            case 128: return go(std::integral_constant<int, 128>(), dealt);
            case 112: return go(std::integral_constant<int, 112>(), dealt);
            case 96: return go(std::integral_constant<int, 96>(), dealt);
            default: return go(std::integral_constant<int, 64>(), dealt);
        }
    };
    return pl.dealt() ? width(std::true_type()) : width(std::false_type());
}

// Returns the number of kernels launched (0: not handled, use the plain kernel).
template <typename TS>
static int fast_attention(bool enabled, bool early, int test_skip, FastState &fs, cudaStream_t st, const StepParams *sp, const Dims &D, int nf,
                          int layer, const TS *q, const TS *kc, const TS *vc, TS *out) {
    if constexpr (!std::is_same<TS, bf16>::value) {
        return 0;
    } else {
        if (!enabled || !fs.ready || fs.plan.KB == 0) return 0;
        return launch_attn_plan(early, test_skip, fs.encode, fs.n_sm, st, sp, D, nf, layer, fs.plan, fs.cache_pages, q, kc, vc, out, fs.part_o,
                                fs.attn_counters, fs.d_status);
    }
}
