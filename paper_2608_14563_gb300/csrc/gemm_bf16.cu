// gemm_bf16.cu -- host launchers of the four tcgen05 GEMMs of the FPO step.
//
//   logits pass      z = yhat W_U^T      M=T  N=V    K=d   A K-major, B K-major
//   recompute pass   same GEMM, epilogue writes E = s (softmax - onehot)
//   direct logits    same GEMM, epilogue writes P = exp(z - c) (target zero)
//   projection       g = E W_U           M=T  N=d    K=V   A K-major, B MN-major
//                    (or g = alpha P W_U + beta W_U[y] in the direct algorithm, whose
//                    epilogue applies the final-norm VJP and writes g~)
//   update           G = g~^T A_l        M=d  N=d_ff K=T   A MN-major, B MN-major
//
// Tensor maps are encoded per call (a few microseconds of host work) through
// the driver entry point of cuTensorMapEncodeTiled, so the library does not
// link libcuda directly.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <mutex>

#include <atomic>

#include "epilogues.cuh"
#include "internal.h"
#include "slot_sum.cuh"
#include "tc_gemm.cuh"
#include "tc_gemm_pair.cuh"

namespace fpo {
namespace {

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// 2-D tensor [outer, inner] of bf16 (esz 2) or fp32 (esz 4) with row stride
// `ld` elements, box {box_inner, box_outer}, 128-byte swizzle, zero fill
// outside the tensor on loads (and clipping on stores).  L2 promotion of 128 bytes:
// one box row; 256-byte promotion fetched 15-55% more from DRAM in the step's GEMMs
// for the same time.
bool make_map(CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer, uint64_t ld,
              uint32_t box_inner, uint32_t box_outer, int esz = 2) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {ld * static_cast<uint64_t>(esz)};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t es[2] = {1, 1};
    const CUtensorMapDataType dt =
        esz == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    return fn(m, dt, 2, const_cast<void*>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Output maps of the epilogues: 32 rows x 128 bytes per store.
bool map_out_f32(CUtensorMap* m, void* base, int rows, int cols) {
    return make_map(m, base, cols, rows, cols, 32, 32, 4);
}
bool map_out_bf16(CUtensorMap* m, void* base, int rows, int cols) {
    return make_map(m, base, cols, rows, cols, 64, 32, 2);
}

// K-major operand [rows, K]: box {64 (K), rows_per_tile}
bool map_kmajor(CUtensorMap* m, const void* base, int rows, int K, int box_rows) {
    return make_map(m, base, K, rows, K, kBK, box_rows);
}
// MN-major operand [K, mn]: box {64 (MN), 64 (K)}
bool map_mnmajor(CUtensorMap* m, const void* base, int K, int mn) {
    return make_map(m, base, mn, K, mn, 64, kBK);
}

GemmShape make_shape(int M, int N, int K, int BN, int groups, int band, int BM = kBM) {
    GemmShape sh;
    sh.M = M;
    sh.N = N;
    sh.K = K;
    sh.m_blocks = (M + BM - 1) / BM;
    sh.n_blocks = (N + BN - 1) / BN;
    sh.k_blocks = (K + kBK - 1) / kBK;
    sh.groups = groups;
    sh.band = band;
    sh.tiles = static_cast<long long>(groups) * sh.m_blocks * sh.n_blocks;
    sh.tail_tiles = 0;
    sh.tail_split = 0;
    sh.sk_scratch = nullptr;
    sh.m_dev = nullptr;
    return sh;
}

template <int BN, bool A_MN, bool B_MN, int STAGES, int MAXG, class Epi>
cudaError_t run_gemm(const GemmMaps<MAXG>& maps, const typename Epi::Params& ep,
                     const GemmShape& sh, unsigned* status, cudaStream_t st) {
    if (sh.tiles <= 0 || sh.k_blocks <= 0) return cudaSuccess;
    using L = GemmSmem<BN, STAGES>;
    constexpr auto kern = tc_gemm_kernel<BN, A_MN, B_MN, STAGES, MAXG, Epi>;
    const cudaError_t attr_err = set_smem_limit<kern>(L::kBytes);
    if (attr_err != cudaSuccess) return attr_err;
    DevInfo di;
    if (!current_device_info(&di)) return cudaErrorUnknown;
    const long long grid = sh.tiles < di.sm_count ? sh.tiles : di.sm_count;
    return launch_chained(kern, dim3(static_cast<unsigned>(grid)), gemm_threads<Epi>(), L::kBytes, st,
                          maps, ep, sh, status, wait_limit_ns());
}

// Clusters (of `cta` CTAs, the kernel's cluster size) that can be resident at once for a
// pair-kernel instantiation.
template <class Kern>
int pair_clusters(Kern kern, int threads, int smem_bytes, int sm_count, int cta) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(sm_count / cta * cta), 1, 1);
    cfg.blockDim = dim3(static_cast<unsigned>(threads), 1, 1);
    cfg.dynamicSmemBytes = static_cast<size_t>(smem_bytes);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = sm_count / cta;
    }
    return n;
}

// pair_clusters for the current device, computed once per device (after the kernel's
// shared-memory limit is raised there).
template <auto Kern>
int resident_clusters(int threads, int smem_bytes, int sm_count, int cta) {
    static std::atomic<int> cache[kMaxDevices];
    const int dev = current_device();
    if (dev < 0) return sm_count / cta;
    int n = cache[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
    n = pair_clusters(Kern, threads, smem_bytes, sm_count, cta);
    cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

// Split-K tail of one launch: tail_tiles tiles, each in tail_split k ranges (0: whole).
struct SkPlan {
    long long tail_tiles = 0;
    int tail_split = 0;
};

// Units of split tail tiles a scratch area must hold: up to three waves of pair clusters.
constexpr int kTailWaves = 3;

// The split of the last partial wave of `tiles` tiles over `clusters` clusters: R tail
// tiles in S k ranges, S chosen so that the R S units fill whole waves as nearly as
// possible (at most kTailWaves waves, at least 8 k-blocks per range); none if no split
// beats the plain partial wave.
SkPlan tail_plan(long long tiles, long long clusters, int k_blocks) {
    SkPlan p;
    const long long R = tiles % clusters;
    if (tiles < clusters || R == 0) return p;
    double best = static_cast<double>(R) / clusters;  // busy fraction of the plain last wave
    for (int S = 2; S <= 64; ++S) {
        if (R * S > kTailWaves * clusters || k_blocks / S < 8) break;
        const long long waves = (R * S + clusters - 1) / clusters;
        const double eff = static_cast<double>(R * S) / (waves * clusters);
        if (eff > best + 1e-9) {
            best = eff;
            p.tail_tiles = R;
            p.tail_split = S;
        }
    }
    return p;
}

// With sk_scratch non-null, the tiles are split by `split` k ranges each when that is above
// 1, else those of the last partial wave by tail_plan (SegCursor); the caller then runs
// sk_fixup over them (plan->tail_tiles > 0).  sk_scratch holds 256 x BN fp32 per unit.
template <int BN, bool A_MN, bool B_MN, int STAGES, int MAXG, class Epi>
cudaError_t run_gemm_pair(const GemmMaps<MAXG>& maps, const typename Epi::Params& ep,
                          const GemmShape& sh_in, unsigned* status, cudaStream_t st,
                          float* sk_scratch = nullptr, SkPlan* plan = nullptr, int split = 0) {
    if (plan) *plan = SkPlan{};
    if (sh_in.tiles <= 0 || sh_in.k_blocks <= 0) return cudaSuccess;
    using L = GemmPairSmem<BN, STAGES, pair_ksub<BN, A_MN, B_MN>()>;
    static_assert(L::kBytes + 2 * kSmemReserve <= kSmemPerSm,
                  "the stages leave the shared memory that a block of the host-input copy takes");
    constexpr auto kern = tc_gemm_pair_kernel<BN, A_MN, B_MN, STAGES, MAXG, Epi>;
    const cudaError_t attr_err = set_smem_limit<kern>(L::kBytes);
    if (attr_err != cudaSuccess) return attr_err;
    DevInfo di;
    if (!current_device_info(&di)) return cudaErrorUnknown;
    const int max_clusters = resident_clusters<kern>(gemm_threads<Epi>(), L::kBytes, di.sm_count, 2);
    const long long units = split > 1 ? sh_in.tiles * split : sh_in.tiles;
    const long long clusters = units < max_clusters ? units : max_clusters;
    GemmShape sh = sh_in;
    if (sk_scratch) {
        SkPlan p;
        if (split > 1) {
            p.tail_tiles = sh.tiles;
            p.tail_split = split;
        } else {
            p = tail_plan(sh.tiles, clusters, sh.k_blocks);
        }
        if (p.tail_tiles > 0) {
            sh.tail_tiles = p.tail_tiles;
            sh.tail_split = p.tail_split;
            sh.sk_scratch = sk_scratch;
            if (plan) *plan = p;
        }
    }
    return launch_chained(kern, dim3(static_cast<unsigned>(2 * clusters)), gemm_threads<Epi>(),
                          L::kBytes, st, maps, ep, sh, status, wait_limit_ns());
}

// Fixups of the split-K tail: sum the tail_split k-range partials of every split tail
// tile in range order, then apply the epilogue the whole tiles got.
// Grid (tail tiles, 256 rows / rows per block): one thread per 4 columns of a row.
constexpr int kFixupThreads = 256;

// The summed partials of this thread's 4 columns; false outside the matrix.
template <int BN>
__device__ __forceinline__ bool sk_tail_sum(const GemmShape& sh, const float* scratch,
                                            int& row, int& n, float (&s4)[4]) {
    constexpr int kThreadsPerRow = BN / 4;
    constexpr int kRowsPerBlock = kFixupThreads / kThreadsPerRow;
    const long long R = sh.tail_tiles;
    const long long r_tile = blockIdx.x;
    const int r = blockIdx.y * kRowsPerBlock + threadIdx.x / kThreadsPerRow;
    const int col = (threadIdx.x % kThreadsPerRow) * 4;
    int g, mp, nb;
    tile_coords(sh.tiles - R + r_tile, sh, g, mp, nb);
    row = mp * kPairBM + r;
    n = nb * BN + col;
    if (row >= sh.M || n >= sh.N) return false;  // N % 8 == 0: whole groups of 4
    s4[0] = s4[1] = s4[2] = s4[3] = 0.f;
    const float* p = scratch + (static_cast<size_t>(r_tile) * kPairBM + r) * BN + col;
    const size_t step = static_cast<size_t>(R) * kPairBM * BN;  // one range to the next
#pragma unroll 4
    for (int q = 0; q < sh.tail_split; ++q) {
        const float4 u = *reinterpret_cast<const float4*>(p + q * step);
        s4[0] += u.x;
        s4[1] += u.y;
        s4[2] += u.z;
        s4[3] += u.w;
    }
    return true;
}

// Plain fp32 sums, as EpiStoreF32 writes whole tiles (the projection g = E W_U).
template <int BN>
__global__ void __launch_bounds__(kFixupThreads)
    sk_fixup_kernel(const GemmShape sh, const float* scratch, float* __restrict__ C) {
    grid_dependency_trigger();
    grid_dependency_wait();
    int row, n;
    float s4[4];
    if (!sk_tail_sum<BN>(sh, scratch, row, n, s4)) return;
    *reinterpret_cast<float4*>(C + static_cast<size_t>(row) * sh.N + n) =
        make_float4(s4[0], s4[1], s4[2], s4[3]);
}

// The direct algorithm's projection with the final-norm VJP fused in, as EpiProjVjp
// writes whole tiles: g = alpha sum + beta W_U[y], out = bf16 of
// (w g - (h / rho) cv / d) / max(rho, min_rms).
struct VjpArgs {
    const float* alpha;
    const float* beta;
    const float* cv;
    const float* rho;
    const int* y;
    const __nv_bfloat16* W_U;
    const __nv_bfloat16* h;
    const __nv_bfloat16* w;
    float min_rms, inv_d;
};

// N summed columns from n of a row of P W_U to those of g~.
template <int N>
__device__ __forceinline__ void vjp_row(const VjpArgs& va, int row, int n, int d,
                                        const float (&acc)[N], float (&o)[N]) {
    const float a = va.alpha[row], bb = va.beta[row];
    const float rr = va.rho[row];
    const float kd = va.cv[row] * va.inv_d;
    const float pref = 1.0f / fmaxf(rr, va.min_rms);
    // the same association as EpiProjVjp: w (a pref sum + b pref W_U[y]) - h (kd pref / rho)
    const float ap = a * pref, bp = bb * pref, nk = -(kd * (1.0f / rr)) * pref;
    const __nv_bfloat16* wy =
        (a != 0.f && bb != 0.f) ? va.W_U + static_cast<long long>(va.y[row]) * d : nullptr;
    const __nv_bfloat16* hr = va.h + static_cast<long long>(row) * d;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const float yv = wy ? __bfloat162float(wy[n + j]) : 0.f;
        const float t = fmaf(bp, yv, ap * acc[j]);
        o[j] = a == 0.f ? 0.f
                        : fmaf(__bfloat162float(va.w[n + j]), t,
                               nk * __bfloat162float(hr[n + j]));
    }
}

template <int BN>
__global__ void __launch_bounds__(kFixupThreads)
    sk_fixup_vjp_kernel(const GemmShape sh, const float* scratch,
                        __nv_bfloat16* __restrict__ out, const VjpArgs va) {
    grid_dependency_trigger();
    grid_dependency_wait();
    int row, n;
    float s4[4];
    if (!sk_tail_sum<BN>(sh, scratch, row, n, s4)) return;
    float o[4];
    vjp_row<4>(va, row, n, sh.N, s4, o);
    *reinterpret_cast<uint2*>(out + static_cast<size_t>(row) * sh.N + n) =
        make_uint2(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]));
}

template <int BN>
dim3 sk_fixup_grid(const SkPlan& plan) {
    constexpr int kRowsPerBlock = kFixupThreads / (BN / 4);
    return dim3(static_cast<unsigned>(plan.tail_tiles), kPairBM / kRowsPerBlock);
}

GemmShape sk_fixup_shape(const SkPlan& plan, const GemmShape& sh_in) {
    GemmShape sh = sh_in;
    sh.tail_tiles = plan.tail_tiles;
    sh.tail_split = plan.tail_split;
    return sh;
}

template <int BN>
cudaError_t launch_sk_fixup(const SkPlan& plan, const GemmShape& sh, const float* scratch,
                            float* C, cudaStream_t st) {
    if (plan.tail_tiles <= 0) return cudaSuccess;
    return launch_chained(sk_fixup_kernel<BN>, sk_fixup_grid<BN>(plan), kFixupThreads, 0, st,
                          sk_fixup_shape(plan, sh), scratch, C);
}

template <int BN>
cudaError_t launch_sk_fixup_vjp(const SkPlan& plan, const GemmShape& sh, const float* scratch,
                                void* out, const VjpArgs& va, cudaStream_t st) {
    if (plan.tail_tiles <= 0) return cudaSuccess;
    return launch_chained(sk_fixup_vjp_kernel<BN>, sk_fixup_grid<BN>(plan), kFixupThreads, 0, st,
                          sk_fixup_shape(plan, sh), scratch, static_cast<__nv_bfloat16*>(out), va);
}

// Fixup of the projection computed with its tokens along N (run_proj_tokens_n): the parts are
// [d, tokens] tiles of 256 x BN.  A block sums 64 d x 32 tokens in range order, turns them
// around in shared memory and writes 8 columns of a token per thread.  kVjp: out is bf16
// g~ as above; else fp32 g.
constexpr int kTurnD = 64, kTurnT = 32;

template <int BN, bool kVjp>
__global__ void __launch_bounds__(kFixupThreads)
    sk_fixup_turn_kernel(const GemmShape sh, const float* scratch,
                         void* __restrict__ out, const VjpArgs va) {
    static_assert(kTurnD * kTurnT == 8 * kFixupThreads && BN % kTurnT == 0, "8 elements per thread");
    __shared__ float tile[kTurnT][kTurnD + 1];
    grid_dependency_trigger();
    grid_dependency_wait();
    const long long R = sh.tail_tiles;
    int g, mb, nb;
    tile_coords(blockIdx.x, sh, g, mb, nb);
    const int d0 = blockIdx.y * kTurnD, t0 = blockIdx.z * kTurnT;  // in the tile
    if (mb * kPairBM + d0 >= sh.M || nb * BN + t0 >= sh.N) return;
    const int r = threadIdx.x / 8, c = threadIdx.x % 8;
    float4 s[2] = {};
    const float* p = scratch + (static_cast<size_t>(blockIdx.x) * kPairBM + d0 + r) * BN + t0 + 4 * c;
    const size_t step = static_cast<size_t>(R) * kPairBM * BN;  // one range to the next
#pragma unroll 4
    for (int q = 0; q < sh.tail_split; ++q) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float4 u = *reinterpret_cast<const float4*>(p + q * step + 32 * i * BN);
            s[i].x += u.x;
            s[i].y += u.y;
            s[i].z += u.z;
            s[i].w += u.w;
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        tile[4 * c][r + 32 * i] = s[i].x;
        tile[4 * c + 1][r + 32 * i] = s[i].y;
        tile[4 * c + 2][r + 32 * i] = s[i].z;
        tile[4 * c + 3][r + 32 * i] = s[i].w;
    }
    __syncthreads();
    const int row = nb * BN + t0 + r;           // token
    const int n = mb * kPairBM + d0 + 8 * c;    // column of g; d is a multiple of 8
    if (row >= sh.N || n >= sh.M) return;
    float acc[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = tile[r][8 * c + j];
    if constexpr (!kVjp) {
        float4* o = reinterpret_cast<float4*>(static_cast<float*>(out) +
                                              static_cast<size_t>(row) * sh.M + n);
        o[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        o[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    } else {
        float o[8];
        vjp_row<8>(va, row, n, sh.M, acc, o);
        *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(out) +
                                  static_cast<size_t>(row) * sh.M + n) =
            make_uint4(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]), pack_bf16x2(o[4], o[5]),
                       pack_bf16x2(o[6], o[7]));
    }
}

constexpr int kProjBN = 256;     // projection tiles where 512 columns are too wide
constexpr int kProjStages = 4;   // (single-CTA kernel)
constexpr int kPairStages = 3;   // 256 x 256 pair tiles: 64 KB stages of two k-blocks
constexpr int kWideBN = 512;     // pair tiles 256 x 512: 48 KB stages
constexpr int kWideStages = 4;

// 0 = single-CTA tiles, 1 = CTA-pair tiles, 2 = CTA-pair tiles with 256 x 512 tiles for
// the projection (default: its K loop runs over the whole vocabulary, so the epilogue
// that the single accumulator cannot overlap costs ~1%, while a quarter less operand
// traffic per FLOP made the projection 6-7% faster)
std::atomic<int> g_gemm_variant{2};
std::atomic<int> g_band_override{0};  // > 0: rasterisation band height (tests / tuning)

bool use_pair() { return g_gemm_variant.load(std::memory_order_relaxed) >= 1; }

// Whether the GEMMs over the vocabulary of a chunk of T tokens run on CTA pairs: not, by
// default, when an odd number of 128-row blocks, at most 5, leaves half of a pair's 256 rows
// empty.  The single-CTA kernel is up to 20% slower per row but wastes at most 127 of them.
// Logits pass in us, on pairs and on single CTAs, at T 128, 333, 600 and 1100 (9 blocks):
//   d 2048, V  50304    52  49    75  64    95  96   145 154
//   d 2048, V 100352    91  80   132 118   181 175   283 301
//   d 4096, V  50304    89  87   137 118   177 181   270 292
//   d 4096, V 100352   163 142   245 223   342 334   544 602
// (V 8192: within 5 us up to 5 blocks.  d 512: single CTAs are faster at every T up to 2048,
// 96 against 108 us there with V 50304.)  Same sums either way.
bool use_pair_rows(int T) {
    const int blocks = (T + kBM - 1) / kBM;
    return use_pair() &&
           !(g_gemm_variant.load(std::memory_order_relaxed) == 2 && blocks % 2 == 1 && blocks <= 5);
}
bool wide_proj() { return g_gemm_variant.load(std::memory_order_relaxed) >= 2; }

// Rasterisation band in tile rows, unless overridden: 16 tile rows, i.e. 2048
// output rows of single-CTA tiles and 4096 of pair tiles.  With pair tiles the
// 4096-row band gave the lowest DRAM traffic of the three GEMMs of the OLMo-2-7B
// shape (band heights 2 to 32 measured).
constexpr int kBandTiles = 16;
int band_for(bool) {
    const int o = g_band_override.load(std::memory_order_relaxed);
    return o > 0 ? o : kBandTiles;
}

// Whether a GEMM of `tiles` 256 x 256 pair tiles runs on tiles of 128 columns instead: when
// twice as many tiles still have a cluster each.  What bounds so small a GEMM is the
// epilogue's traffic through one SM (32 bytes a clock to L2), which twice as many SMs share.
// T 200, d 256, d_ff 384, V 1024, 2 layers: update 13.1 -> 9.5 us, projection 15.1 -> 12.1.
bool half_tiles(long long tiles) {
    DevInfo di;
    return current_device_info(&di) && 2 * tiles <= di.sm_count / 2;
}

constexpr int kHalfBN = 128;     // 48 KB stages of two k-blocks
constexpr int kHalfStages = 4;

// A GEMM with an 8-warp epilogue (MN-major B) on the kernel and tiles its size calls for.
template <bool A_MN, int MAXG, template <int> class Epi>
cudaError_t run_quad(const GemmMaps<MAXG>& maps, const typename Epi<2>::Params& ep, int M, int N,
                     int K, int groups, unsigned* status, cudaStream_t st) {
    constexpr int kBN = 256, kStages = 4;
    if (!use_pair())
        return run_gemm<kBN, A_MN, true, kStages, MAXG, Epi<2>>(
            maps, ep, make_shape(M, N, K, kBN, groups, band_for(false)), status, st);
    const GemmShape sh = make_shape(M, N, K, kBN, groups, band_for(true), kPairBM);
    if (!half_tiles(sh.tiles))
        return run_gemm_pair<kBN, A_MN, true, kPairStages, MAXG, Epi<2>>(maps, ep, sh, status, st);
    GemmShape hs = sh;
    hs.n_blocks = 2 * sh.n_blocks;  // also a last half outside the matrix: its slots are written
    hs.tiles = 2 * sh.tiles;
    return run_gemm_pair<kHalfBN, A_MN, true, kHalfStages, MAXG, Epi<1>>(maps, ep, hs, status, st);
}

}  // namespace

void set_band_override(int b) { g_band_override.store(b > 0 ? b : 0, std::memory_order_relaxed); }

void set_gemm_variant(int v) {
    g_gemm_variant.store(v >= 0 && v <= 2 ? v : 0, std::memory_order_relaxed);
}
int gemm_variant() { return g_gemm_variant.load(std::memory_order_relaxed); }

namespace {

// Pair clusters of the 256 x 512 projection kernel resident at once on the current device
// (an upper bound of 128 without one).
int proj_clusters() {
    using L = GemmPairSmem<kWideBN, kWideStages, pair_ksub<kWideBN, false, true>()>;
    constexpr auto kern = tc_gemm_pair_kernel<kWideBN, false, true, kWideStages, 1, EpiProjVjp>;
    DevInfo di;
    int c = 128;
    if (current_device_info(&di) && set_smem_limit<kern>(L::kBytes) == cudaSuccess)
        c = resident_clusters<kern>(gemm_threads<EpiProjVjp>(), L::kBytes, di.sm_count, 2);
    cudaGetLastError();
    return c;
}

// K ranges per tile of the projection of a batch of T tokens, or 0: batches with at least
// one 256 x 512 tile per pair cluster take those tiles whole, with the split tail of the
// last wave.  Below that the clusters without a tile would idle through a K loop over the
// whole vocabulary, so such a batch runs on 256 x 256 tiles, each in the number of ranges
// that costs least.  Measured, in ns: a 64-deep k-block 344 (at the clock the tensor cores
// hold under load), with a split 2500 per wave of units for the epilogue that stores their
// fp32 parts, the fixup's launch 4000 and its read of the parts 4.3 bytes a ns.  Ranges
// have at least 32 k-blocks, and the units fit the scratch.  T is the whole batch, so that
// its sums do not depend on the chunking.  Projection with its fixup, T x d x V:
// 333 x 4096 x 100352 (16 tiles of 512 columns on 76 clusters) 887 us whole, 246 us in 7
// ranges; 2048 x 2048 x 50304 (32 such tiles) 434 us, 276 in 7 ranges of 256 columns and
// about the same in whole 256-column tiles, which draw less power (step 818 and 777 us).
//
// The split projection can also run the other way around, g^T = W_U^T P^T with the tokens
// along N, in 256 x 384 tiles: a 64-deep k-block takes 560 ns, but 40 KB of operands per SM
// serve up to 384 tokens where two 256 x 256 tiles take 64 KB.  The costs choose it where
// about a third of the other form's rows would be empty.  Error signal, T x d x V: 333 x
// 4096 x 100352 497 -> 464 us, 333 x 2048 x 50304 182 -> 172, 1100 x 4096 x 100352 1234 ->
// 1120; 512 x 4096 x 100352 would take 629 instead of 535, 768 x 4096 x 100352 the same.
//
// Ranges of 256 x 512 tiles (670 ns a k-block, and 5000 for the store, which the next unit
// of their single accumulator waits for) leave half as many parts to add: 200 x 4096 x
// 100352 350 -> 338 us, 200 x 5120 x 152064 600 -> 570, 600 x 4096 x 100352 715 -> 695.
//
// The constants are of one state of the clock; what the choice needs is their ratios.  Over d
// 512, 2048, 4096 x V 8192, 50304, 100352 x 13 T from 64 to 2048, the projection with its
// fixup took 0.09 to 1.02 of its time in whole 256-column tiles.
struct ProjPlan {
    int split = 0;        // K ranges per tile; 0: whole 512-column tiles
    int width = kWideBN;  // columns of a tile: of g, or kTurnBN tokens
};

constexpr int kTurnBN = 384;     // tokens of a tile with the tokens along N
constexpr int kTurnStages = 4;   // 40 KB stages

ProjPlan proj_plan(int T, int d, int V) {
    const long long clusters = proj_clusters();
    const long long m_blocks = (T + kPairBM - 1) / kPairBM;
    ProjPlan best;
    if (m_blocks * ((d + kWideBN - 1) / kWideBN) >= clusters) return best;
    const int kb = (V + kBK - 1) / kBK;
    double best_cost = 0.0;
    auto consider = [&](int width, long long tiles, double k_block_ns, double store_ns) {
        const long long cap = kTailWaves * clusters * kWideBN / width;  // units of scratch
        for (int S = width == kProjBN ? 1 : 2; S <= 64; ++S) {
            if (S > 1 && (kb / S < 32 || tiles * S > cap)) break;
            const double waves = static_cast<double>((tiles * S + clusters - 1) / clusters);
            double cost = waves * ((kb + S - 1) / S) * k_block_ns;
            if (S > 1) cost += waves * store_ns + 4000.0 + tiles * S * (width * 1024.0) / 4300.0;
            if (best.split == 0 || cost < best_cost) {
                best_cost = cost;
                best.split = S;
                best.width = width;
            }
        }
    };
    consider(kProjBN, m_blocks * ((d + kProjBN - 1) / kProjBN), 344.0, 2500.0);
    consider(kWideBN, m_blocks * ((d + kWideBN - 1) / kWideBN), 670.0, 5000.0);
    consider(kTurnBN, ((d + kPairBM - 1) / kPairBM) * static_cast<long long>((T + kTurnBN - 1) / kTurnBN),
             560.0, 2500.0);
    return best;
}

// A chunk of Tc of the batch's T_all tokens.  A large batch's sums run over the whole of K in
// every chunk of less than a wave (the last one of T 9000 has 808 tokens), whichever the
// chunking; its tiles are 256 columns wide where all of them then have a cluster at once
// (344 against 670 ns a k-block, the same sums).  Error signal, T x d x V, in
// 512-column tiles and so: 9000 x 4096 x 50304 4490 and 4328 us, 9000 x 2048 x 100352 4840 and
// 4560, 9984 x 1024 x 8192 in chunks of 1024 1425 and 710.  (K ranges chosen from the chunk
// are 0.1-1.9% faster still, 14% in the last, but make the sums depend on the chunking.)
ProjPlan proj_plan(int T_all, int Tc, int d, int V) {
    ProjPlan p = proj_plan(T_all, d, V);
    const long long narrow = static_cast<long long>((Tc + kPairBM - 1) / kPairBM) *
                             ((d + kProjBN - 1) / kProjBN);
    if (p.split == 0 && narrow <= proj_clusters()) {
        p.split = 1;
        p.width = kProjBN;
    }
    return p;
}

// The split projection with the tokens along N, and its fixup.
template <bool kVjp>
cudaError_t run_proj_tokens_n(const void* E, const void* W_U, int Tc, int d, int V, int split,
                              float* sk_scratch, void* out, const VjpArgs& va, unsigned* status,
                              cudaStream_t st) {
    GemmMaps<1> maps;
    if (!map_mnmajor(&maps.a[0], W_U, V, d) || !map_kmajor(&maps.b[0], E, Tc, V, kTurnBN / 4))
        return cudaErrorInvalidValue;
    const GemmShape sh = make_shape(d, Tc, V, kTurnBN, 1, band_for(true), kPairBM);
    SkPlan plan;
    const cudaError_t e = run_gemm_pair<kTurnBN, true, false, kTurnStages, 1, EpiParts>(
        maps, EpiParts::Params{}, sh, status, st, sk_scratch, &plan, split);
    if (e != cudaSuccess || plan.tail_tiles <= 0) return e;
    const dim3 grid(static_cast<unsigned>(plan.tail_tiles), kPairBM / kTurnD, kTurnBN / kTurnT);
    return launch_chained(sk_fixup_turn_kernel<kTurnBN, kVjp>, grid, kFixupThreads, 0, st,
                          sk_fixup_shape(plan, sh), static_cast<const float*>(sk_scratch), out, va);
}

}  // namespace

size_t proj_sk_scratch_bytes() {
    // kTailWaves x clusters units of 256 x 512 fp32 (twice as many of 256 x 256)
    return static_cast<size_t>(kTailWaves) * proj_clusters() * kPairBM * kWideBN * sizeof(float);
}

constexpr int kLseBN = 256;
constexpr int kLseStages = 4;
int lse_tile_n_bf16() { return kLseBN; }

cudaError_t launch_lse_partial_bf16(const void* yhat, const void* W_U, const int32_t* y, int T,
                                    int d, int V, float2* part, int part_ld, float* zy, float* z,
                                    unsigned* status, cudaStream_t st) {
    const bool pair = use_pair_rows(T);
    GemmMaps<1> maps;
    if (!map_kmajor(&maps.a[0], yhat, T, d, kBM) ||
        !map_kmajor(&maps.b[0], W_U, V, d, pair ? kLseBN / 2 : kLseBN))
        return cudaErrorInvalidValue;
    const GemmShape sh = make_shape(T, V, d, kLseBN, 1, band_for(pair), pair ? kPairBM : kBM);
    if (z) {
        EpiLseStoreZ::Params ep;
        if (!map_out_f32(&ep.zmap, z, T, V)) return cudaErrorInvalidValue;
        ep.part = part;
        ep.part_ld = part_ld;
        ep.zy = zy;
        ep.y = y;
        ep.M = T;
        ep.N = V;
        if (pair)
            return run_gemm_pair<kLseBN, false, false, kPairStages, 1, EpiLseStoreZ>(maps, ep, sh,
                                                                                     status, st);
        return run_gemm<kLseBN, false, false, kLseStages, 1, EpiLseStoreZ>(maps, ep, sh, status, st);
    }
    EpiLsePartial::Params ep;
    ep.zmap = maps.a[0];  // unused
    ep.part = part;
    ep.part_ld = part_ld;
    ep.zy = zy;
    ep.y = y;
    ep.M = T;
    ep.N = V;
    if (pair)
        return run_gemm_pair<kLseBN, false, false, kPairStages, 1, EpiLsePartial>(maps, ep, sh,
                                                                                  status, st);
    return run_gemm<kLseBN, false, false, kLseStages, 1, EpiLsePartial>(maps, ep, sh, status, st);
}

cudaError_t launch_error_bf16(const void* yhat, const void* W_U, const int32_t* y, const float* lse,
                              int Tc, int d, int V, float s, void* E, unsigned* status,
                              cudaStream_t st) {
    const bool pair = use_pair_rows(Tc);
    GemmMaps<1> maps;
    if (!map_kmajor(&maps.a[0], yhat, Tc, d, kBM) ||
        !map_kmajor(&maps.b[0], W_U, V, d, pair ? kLseBN / 2 : kLseBN))
        return cudaErrorInvalidValue;
    EpiError::Params ep;
    if (!map_out_bf16(&ep.Emap, E, Tc, V)) return cudaErrorInvalidValue;
    ep.lse = lse;
    ep.y = y;
    ep.M = Tc;
    ep.N = V;
    ep.s = s;
    const GemmShape sh = make_shape(Tc, V, d, kLseBN, 1, band_for(pair), pair ? kPairBM : kBM);
    if (pair)
        return run_gemm_pair<kLseBN, false, false, kPairStages, 1, EpiError>(maps, ep, sh, status,
                                                                             st);
    return run_gemm<kLseBN, false, false, kLseStages, 1, EpiError>(maps, ep, sh, status, st);
}

cudaError_t launch_anchor_prob_bf16(const void* yhat, const void* W_U, const int32_t* y,
                                    const float* anchor, int T, int d, int V, float* su, float* sx,
                                    float* qz, int part_ld, void* P, unsigned* status,
                                    cudaStream_t st) {
    const bool pair = use_pair_rows(T);
    GemmMaps<1> maps;
    if (!map_kmajor(&maps.a[0], yhat, T, d, kBM) ||
        !map_kmajor(&maps.b[0], W_U, V, d, pair ? kLseBN / 2 : kLseBN))
        return cudaErrorInvalidValue;
    EpiAnchorProb::Params ep;
    if (!map_out_bf16(&ep.pmap, P, T, V)) return cudaErrorInvalidValue;
    ep.su = su;
    ep.sx = sx;
    ep.qz = qz;
    ep.part_ld = part_ld;
    ep.y = y;
    ep.anchor = anchor;
    ep.M = T;
    ep.N = V;
    const GemmShape sh = make_shape(T, V, d, kLseBN, 1, band_for(pair), pair ? kPairBM : kBM);
    if (pair)
        return run_gemm_pair<kLseBN, false, false, kPairStages, 1, EpiAnchorProb>(maps, ep, sh,
                                                                                  status, st);
    return run_gemm<kLseBN, false, false, kLseStages, 1, EpiAnchorProb>(maps, ep, sh, status, st);
}

// The fixup passes: the same GEMM as the logits pass on the gathered rows outside the
// anchor window.  Always the pair kernel (the only one that reads its row count on the
// device): the recomputed rows are identical whichever kernel variant the other GEMMs use.
cudaError_t launch_fixup_lse_bf16(const void* yfix, const void* W_U, const int* fix,
                                  const int* fix_count, int Tc, int d, int V, float2* part,
                                  int part_ld, unsigned* status, cudaStream_t st) {
    GemmMaps<1> maps;
    if (!map_kmajor(&maps.a[0], yfix, Tc, d, kBM) || !map_kmajor(&maps.b[0], W_U, V, d, kLseBN / 2))
        return cudaErrorInvalidValue;
    EpiFixLse::Params ep;
    ep.part = part;
    ep.part_ld = part_ld;
    ep.fix = fix;
    ep.count = fix_count;
    ep.N = V;
    GemmShape sh = make_shape(Tc, V, d, kLseBN, 1, band_for(true), kPairBM);
    sh.m_dev = fix_count;
    return run_gemm_pair<kLseBN, false, false, kPairStages, 1, EpiFixLse>(maps, ep, sh, status, st);
}

cudaError_t launch_fixup_logits_bf16(const void* yfix, const void* W_U, const int* fix,
                                     const int* fix_count, const int32_t* y, const float* lse,
                                     int Tc, int d, int V, void* P, float* sx, float* qz,
                                     int n_tiles, unsigned* status, cudaStream_t st) {
    GemmMaps<1> maps;
    if (!map_kmajor(&maps.a[0], yfix, Tc, d, kBM) || !map_kmajor(&maps.b[0], W_U, V, d, kLseBN / 2))
        return cudaErrorInvalidValue;
    EpiFixProb::Params ep;
    ep.P = static_cast<__nv_bfloat16*>(P);
    ep.sx = sx;
    ep.qz = qz;
    ep.fix = fix;
    ep.count = fix_count;
    ep.y = y;
    ep.lse = lse;
    ep.n_tiles = n_tiles;
    ep.N = V;
    GemmShape sh = make_shape(Tc, V, d, kLseBN, 1, band_for(true), kPairBM);
    sh.m_dev = fix_count;
    return run_gemm_pair<kLseBN, false, false, kPairStages, 1, EpiFixProb>(maps, ep, sh, status, st);
}

cudaError_t launch_proj_vjp_bf16(const void* P, const void* W_U, const int32_t* y,
                                 const float* alpha, const float* beta, const float* cv,
                                 const float* rho, const void* h, const void* w, float min_rms,
                                 int Tc, int T_all, int d, int V, void* g_tilde,
                                 float* sk_scratch, unsigned* status, cudaStream_t st) {
    GemmMaps<1> maps;
    if (!map_kmajor(&maps.a[0], P, Tc, V, kBM) || !map_mnmajor(&maps.b[0], W_U, V, d))
        return cudaErrorInvalidValue;
    EpiProjVjp::Params ep;
    if (!map_out_bf16(&ep.omap, g_tilde, Tc, d)) return cudaErrorInvalidValue;
    VjpArgs va;
    va.alpha = ep.alpha = alpha;
    va.beta = ep.beta = beta;
    va.cv = ep.cv = cv;
    va.rho = ep.rho = rho;
    va.y = ep.y = y;
    va.W_U = ep.W_U = static_cast<const __nv_bfloat16*>(W_U);
    va.h = ep.h = static_cast<const __nv_bfloat16*>(h);
    va.w = ep.w = static_cast<const __nv_bfloat16*>(w);
    va.min_rms = ep.min_rms = min_rms;
    va.inv_d = ep.inv_d = 1.0f / static_cast<float>(d);
    ep.M = Tc;
    ep.N = d;
    if (wide_proj()) {
        SkPlan plan;
        const ProjPlan pp = proj_plan(T_all, Tc, d, V);
        if (pp.width == kTurnBN)
            return run_proj_tokens_n<true>(P, W_U, Tc, d, V, pp.split, sk_scratch, g_tilde, va,
                                           status, st);
        if (pp.width == kWideBN) {
            ep.tile_n = kWideBN;
            const GemmShape sh = make_shape(Tc, d, V, kWideBN, 1, band_for(true), kPairBM);
            const cudaError_t e = run_gemm_pair<kWideBN, false, true, kWideStages, 1, EpiProjVjp>(
                maps, ep, sh, status, st, sk_scratch, &plan, pp.split);
            if (e != cudaSuccess) return e;
            return launch_sk_fixup_vjp<kWideBN>(plan, sh, sk_scratch, g_tilde, va, st);
        }
        const GemmShape sh = make_shape(Tc, d, V, kProjBN, 1, band_for(true), kPairBM);
        if (pp.split == 1 && half_tiles(sh.tiles)) {
            ep.tile_n = kHalfBN;
            return run_gemm_pair<kHalfBN, false, true, kHalfStages, 1, EpiProjVjp>(
                maps, ep, make_shape(Tc, d, V, kHalfBN, 1, band_for(true), kPairBM), status, st);
        }
        ep.tile_n = kProjBN;
        const cudaError_t e = run_gemm_pair<kProjBN, false, true, kPairStages, 1, EpiProjVjp>(
            maps, ep, sh, status, st, pp.split > 1 ? sk_scratch : nullptr, &plan, pp.split);
        if (e != cudaSuccess) return e;
        return launch_sk_fixup_vjp<kProjBN>(plan, sh, sk_scratch, g_tilde, va, st);
    }
    ep.tile_n = kProjBN;
    if (use_pair())
        return run_gemm_pair<kProjBN, false, true, kPairStages, 1, EpiProjVjp>(
            maps, ep, make_shape(Tc, d, V, kProjBN, 1, band_for(true), kPairBM), status, st);
    return run_gemm<kProjBN, false, true, kProjStages, 1, EpiProjVjp>(
        maps, ep, make_shape(Tc, d, V, kProjBN, 1, band_for(false)), status, st);
}

cudaError_t launch_proj_bf16(const void* E, const void* W_U, int Tc, int T_all, int d, int V,
                             float* g, float* sk_scratch, unsigned* status, cudaStream_t st) {
    GemmMaps<1> maps;
    if (!map_kmajor(&maps.a[0], E, Tc, V, kBM) || !map_mnmajor(&maps.b[0], W_U, V, d))
        return cudaErrorInvalidValue;
    EpiStoreF32::Params ep;
    if (!map_out_f32(&ep.Cmap, g, Tc, d)) return cudaErrorInvalidValue;
    ep.M = Tc;
    ep.N = d;
    if (wide_proj()) {
        SkPlan plan;
        const ProjPlan pp = proj_plan(T_all, Tc, d, V);
        if (pp.width == kTurnBN)
            return run_proj_tokens_n<false>(E, W_U, Tc, d, V, pp.split, sk_scratch, g, VjpArgs{},
                                            status, st);
        if (pp.width == kWideBN) {
            const GemmShape sh = make_shape(Tc, d, V, kWideBN, 1, band_for(true), kPairBM);
            const cudaError_t e = run_gemm_pair<kWideBN, false, true, kWideStages, 1, EpiStoreF32>(
                maps, ep, sh, status, st, sk_scratch, &plan, pp.split);
            if (e != cudaSuccess) return e;
            return launch_sk_fixup<kWideBN>(plan, sh, sk_scratch, g, st);
        }
        // (no tiles of 128 columns as in the direct algorithm: bf16 runs here only when the
        // stored-logits or recompute algorithm is asked for)
        const GemmShape sh = make_shape(Tc, d, V, kProjBN, 1, band_for(true), kPairBM);
        const cudaError_t e = run_gemm_pair<kProjBN, false, true, kPairStages, 1, EpiStoreF32>(
            maps, ep, sh, status, st, pp.split > 1 ? sk_scratch : nullptr, &plan, pp.split);
        if (e != cudaSuccess) return e;
        return launch_sk_fixup<kProjBN>(plan, sh, sk_scratch, g, st);
    }
    if (use_pair())
        return run_gemm_pair<kProjBN, false, true, kPairStages, 1, EpiStoreF32>(
            maps, ep, make_shape(Tc, d, V, kProjBN, 1, band_for(true), kPairBM), status, st);
    return run_gemm<kProjBN, false, true, kProjStages, 1, EpiStoreF32>(
        maps, ep, make_shape(Tc, d, V, kProjBN, 1, band_for(false)), status, st);
}

constexpr int kUpdBN = 256;  // columns of a group of partial-sum slots

cudaError_t launch_update_bf16(int n, int T, int d, int d_ff, const void* const* g,
                               const void* const* A, float lr, float* const* W_master,
                               void* const* W_out, void* const* G_out, unsigned* status,
                               cudaStream_t st) {
    if (n < 1 || n > kMaxGroups) return cudaErrorInvalidValue;
    static GemmMaps<kMaxGroups> maps;  // host staging; copied into the launch parameters
    static EpiUpdateBase::Params ep;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    for (int l = 0; l < n; ++l) {
        if (l > 0 && g[l] == g[0])
            maps.a[l] = maps.a[0];
        else if (!map_mnmajor(&maps.a[l], g[l], T, d))
            return cudaErrorInvalidValue;
        if (!map_mnmajor(&maps.b[l], A[l], T, d_ff)) return cudaErrorInvalidValue;
        ep.W_master[l] = W_master ? W_master[l] : nullptr;
        ep.W_out[l] = W_out ? static_cast<__nv_bfloat16*>(W_out[l]) : nullptr;
        ep.G_out[l] = G_out ? static_cast<__nv_bfloat16*>(G_out[l]) : nullptr;
    }
    for (int l = n; l < kMaxGroups; ++l) {
        maps.a[l] = maps.a[0];
        maps.b[l] = maps.b[0];
        ep.W_master[l] = nullptr;
        ep.W_out[l] = nullptr;
        ep.G_out[l] = nullptr;
    }
    ep.ld = d_ff;
    ep.M = d;
    ep.N = d_ff;
    ep.neg_lr = -lr;
    return run_quad<true, kMaxGroups, EpiUpdate>(maps, ep, d, d_ff, T, n, status, st);
}

cudaError_t launch_grad_bf16(int n, int T, int d, int d_ff, const void* const* g,
                             const void* const* A, float* const* G_out,
                             float* const* W_master, float* part, unsigned* status,
                             cudaStream_t st) {
    if (n < 1 || n > kMaxGroups) return cudaErrorInvalidValue;
    static GemmMaps<kMaxGroups> maps;
    static EpiStoreGroupF32Base::Params ep;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    for (int l = 0; l < n; ++l) {
        if (l > 0 && g[l] == g[0])
            maps.a[l] = maps.a[0];
        else if (!map_mnmajor(&maps.a[l], g[l], T, d))
            return cudaErrorInvalidValue;
        if (!map_mnmajor(&maps.b[l], A[l], T, d_ff)) return cudaErrorInvalidValue;
        ep.G[l] = G_out[l];
        ep.W_master[l] = W_master ? W_master[l] : nullptr;
    }
    for (int l = n; l < kMaxGroups; ++l) {
        maps.a[l] = maps.a[0];
        maps.b[l] = maps.b[0];
        ep.G[l] = G_out[0];
        ep.W_master[l] = ep.W_master[0];
    }
    ep.part = part;
    ep.ld = d_ff;
    ep.M = d;
    ep.N = d_ff;
    ep.m256 = (d + 255) / 256;
    ep.n_blocks = (d_ff + kUpdBN - 1) / kUpdBN;
    if (W_master && !use_pair()) {  // as in launch_opt_step_bf16
        const cudaError_t e = cudaMemsetAsync(part, 0, n * opt_step_partial_bytes(1, d, d_ff), st);
        if (e != cudaSuccess) return e;
    }
    return run_quad<true, kMaxGroups, EpiStoreGroupF32>(maps, ep, d, d_ff, T, n, status, st);
}

cudaError_t launch_opt_step_bf16(int n, int T, int d, int d_ff, const void* const* g,
                                 const void* const* A, const OptimParams& op,
                                 float* const* W_master, float* const* s1, float* const* s2,
                                 float* const* D, float* part, unsigned* status, cudaStream_t st) {
    if (n < 1 || n > kMaxGroups) return cudaErrorInvalidValue;
    static GemmMaps<kMaxGroups> maps;
    static EpiOptStepBase::Params ep;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    for (int l = 0; l < kMaxGroups; ++l) {
        const int k = l < n ? l : 0;
        if (l < n) {
            if (l > 0 && g[l] == g[0])
                maps.a[l] = maps.a[0];
            else if (!map_mnmajor(&maps.a[l], g[l], T, d))
                return cudaErrorInvalidValue;
            if (!map_mnmajor(&maps.b[l], A[l], T, d_ff)) return cudaErrorInvalidValue;
        } else {
            maps.a[l] = maps.a[0];
            maps.b[l] = maps.b[0];
        }
        ep.W_master[l] = W_master[k];
        ep.s1[l] = s1 ? s1[k] : nullptr;
        ep.s2[l] = s2 ? s2[k] : nullptr;
        ep.D[l] = D ? D[k] : nullptr;
    }
    ep.part = part;
    ep.op = op;
    ep.ld = d_ff;
    ep.M = d;
    ep.N = d_ff;
    ep.m256 = (d + 255) / 256;
    ep.n_blocks = (d_ff + kUpdBN - 1) / kUpdBN;
    // single-CTA 128-row tiles leave the upper half of a last, short 256-row block of slots
    // unwritten: start from zeros
    if (!use_pair()) {
        const cudaError_t e = cudaMemsetAsync(part, 0, n * opt_step_partial_bytes(1, d, d_ff), st);
        if (e != cudaSuccess) return e;
    }
    return run_quad<true, kMaxGroups, EpiOptStep>(maps, ep, d, d_ff, T, n, status, st);
}

size_t opt_step_partial_bytes(int n_layers, int d, int d_ff) {
    return static_cast<size_t>(n_layers) * ((d + 255) / 256) * ((d_ff + kUpdBN - 1) / kUpdBN) *
           kColSlots * 2 * sizeof(float);
}

// Second pass of the fused cosine: a cluster per layer adds the layer's slot triples in a
// fixed order and writes <G, Y>, ||G||^2, ||Y||^2 and the cosine.
__global__ void __cluster_dims__(kSlotBlocks, 1, 1) __launch_bounds__(kSlotThreads)
    grad_cosine_final_kernel(const float* part, int slots, double* __restrict__ out) {
    grid_dependency_trigger();
    grid_dependency_wait();
    const int layer = blockIdx.x / kSlotBlocks;
    double t[3];
    if (!slot_sum<3>(part + static_cast<size_t>(layer) * slots * 3, slots, t)) return;
    double* o = out + 4 * layer;
    o[0] = t[0];
    o[1] = t[1];
    o[2] = t[2];
    o[3] = (t[1] > 0.0 && t[2] > 0.0) ? t[0] / (sqrt(t[1]) * sqrt(t[2])) : 0.0;
}

size_t grad_cosine_partial_bytes(int n, int d, int d_ff) {
    const size_t m256 = (static_cast<size_t>(d) + 255) / 256;
    const size_t nb = (static_cast<size_t>(d_ff) + kUpdBN - 1) / kUpdBN;
    return static_cast<size_t>(n) * m256 * nb * kColSlots * 3 * sizeof(float);
}

cudaError_t launch_grad_cosine_bf16(int n, int T, int d, int d_ff, const void* const* g,
                                    const void* const* A, const void* const* Y,
                                    void* const* G_out, float* part, double* out,
                                    unsigned* status, cudaStream_t st) {
    if (n < 1 || n > kMaxGroups) return cudaErrorInvalidValue;
    static GemmMaps<kMaxGroups> maps;
    static EpiGradCosBase::Params ep;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    for (int l = 0; l < n; ++l) {
        if (l > 0 && g[l] == g[0])
            maps.a[l] = maps.a[0];
        else if (!map_mnmajor(&maps.a[l], g[l], T, d))
            return cudaErrorInvalidValue;
        if (!map_mnmajor(&maps.b[l], A[l], T, d_ff)) return cudaErrorInvalidValue;
        ep.G_out[l] = static_cast<__nv_bfloat16*>(G_out[l]);
        ep.Y[l] = static_cast<const __nv_bfloat16*>(Y[l]);
    }
    for (int l = n; l < kMaxGroups; ++l) {
        maps.a[l] = maps.a[0];
        maps.b[l] = maps.b[0];
        ep.G_out[l] = ep.G_out[0];
        ep.Y[l] = ep.Y[0];
    }
    ep.part = part;
    ep.ld = d_ff;
    ep.M = d;
    ep.N = d_ff;
    ep.m256 = (d + 255) / 256;
    ep.n_blocks = (d_ff + kUpdBN - 1) / kUpdBN;
    // every slot is written by a tile (pair kernel), but single-CTA 128-row tiles leave
    // the upper half of a last, short 256-row block unwritten: start from zeros
    cudaError_t e = cudaSuccess;
    if (!use_pair()) e = cudaMemsetAsync(part, 0, grad_cosine_partial_bytes(n, d, d_ff), st);
    if (e != cudaSuccess) return e;
    e = run_quad<true, kMaxGroups, EpiGradCos>(maps, ep, d, d_ff, T, n, status, st);
    if (e != cudaSuccess) return e;
    return launch_chained(grad_cosine_final_kernel, dim3(kSlotBlocks * n), kSlotThreads, 0, st, part,
                          ep.m256 * ep.n_blocks * kColSlots, out);
}

cudaError_t launch_swiglu_bf16(int T, int d, int d_ff, const void* g, const void* W3,
                               const void* a, const void* b, void* dA, void* dB, unsigned* status,
                               cudaStream_t st) {
    GemmMaps<1> maps;
    if (!map_kmajor(&maps.a[0], g, T, d, kBM) || !map_mnmajor(&maps.b[0], W3, d, d_ff))
        return cudaErrorInvalidValue;
    EpiSwigluBase::Params ep;
    ep.dA = static_cast<__nv_bfloat16*>(dA);
    ep.dB = static_cast<__nv_bfloat16*>(dB);
    ep.a = static_cast<const __nv_bfloat16*>(a);
    ep.b = static_cast<const __nv_bfloat16*>(b);
    ep.ld = d_ff;
    ep.M = T;
    ep.N = d_ff;
    return run_quad<false, 1, EpiSwiglu>(maps, ep, T, d_ff, d, 1, status, st);
}

cudaError_t launch_test_gemm_bf16(int M, int N, int K, bool a_mn, bool b_mn, const void* A,
                                  const void* B, float* C, unsigned* status, cudaStream_t st) {
    const bool pair = use_pair();
    GemmMaps<1> maps;
    bool ok = a_mn ? map_mnmajor(&maps.a[0], A, K, M) : map_kmajor(&maps.a[0], A, M, K, kBM);
    ok = ok && (b_mn ? map_mnmajor(&maps.b[0], B, K, N)
                     : map_kmajor(&maps.b[0], B, N, K, pair ? 128 : 256));
    if (!ok) return cudaErrorInvalidValue;
    EpiStoreF32::Params ep;
    if (!map_out_f32(&ep.Cmap, C, M, N)) return cudaErrorInvalidValue;
    ep.M = M;
    ep.N = N;
    if (wide_proj()) {  // every layout on 256 x 512 pair tiles
        const GemmShape sh = make_shape(M, N, K, kWideBN, 1, band_for(true), kPairBM);
        if (!a_mn && !b_mn)
            return run_gemm_pair<kWideBN, false, false, kWideStages, 1, EpiStoreF32>(maps, ep, sh,
                                                                                    status, st);
        if (!a_mn && b_mn)
            return run_gemm_pair<kWideBN, false, true, kWideStages, 1, EpiStoreF32>(maps, ep, sh,
                                                                                   status, st);
        if (a_mn && b_mn)
            return run_gemm_pair<kWideBN, true, true, kWideStages, 1, EpiStoreF32>(maps, ep, sh,
                                                                                  status, st);
        return cudaErrorInvalidValue;
    }
    if (pair) {
        const GemmShape sh = make_shape(M, N, K, 256, 1, band_for(true), kPairBM);
        if (!a_mn && !b_mn)
            return run_gemm_pair<256, false, false, kPairStages, 1, EpiStoreF32>(maps, ep, sh, status, st);
        if (!a_mn && b_mn)
            return run_gemm_pair<256, false, true, kPairStages, 1, EpiStoreF32>(maps, ep, sh, status, st);
        if (a_mn && b_mn)
            return run_gemm_pair<256, true, true, kPairStages, 1, EpiStoreF32>(maps, ep, sh, status, st);
        return cudaErrorInvalidValue;
    }
    const GemmShape sh = make_shape(M, N, K, 256, 1, band_for(false));
    if (!a_mn && !b_mn) return run_gemm<256, false, false, 4, 1, EpiStoreF32>(maps, ep, sh, status, st);
    if (!a_mn && b_mn) return run_gemm<256, false, true, 4, 1, EpiStoreF32>(maps, ep, sh, status, st);
    if (a_mn && b_mn) return run_gemm<256, true, true, 4, 1, EpiStoreF32>(maps, ep, sh, status, st);
    return cudaErrorInvalidValue;
}

}  // namespace fpo
