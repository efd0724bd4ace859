// tc_gemm.cuh -- persistent tcgen05 GEMM core with pluggable epilogues.
//
//   C[g][m, n] = sum_k A(m, k) * B[g](n, k)      (bf16 inputs, fp32 accumulate)
//
// One CTA per SM (persistent over output tiles), 192 or 320 threads:
//   warp 0      TMA producer: streams A/B k-blocks into a STAGES-deep ring of
//               128-byte-swizzled shared-memory buffers (mbarrier full/empty).
//   warp 1      allocates TMEM; lane 0 issues tcgen05.mma (128 x BN x 16) and
//               commits stage releases / accumulator-ready signals.
//   warps 2..   epilogue (Epi::kWarps of them, 4 or 8): tcgen05.ld of the fp32
//               accumulator (one row per thread), hand the values to the
//               Epilogue functor.
// The accumulator is double-buffered in TMEM (2 x BN columns) so the epilogue
// of tile i overlaps the mainloop of tile i+1.
//
// Operands may be K-major (K contiguous) or MN-major (M/N contiguous); both
// are loaded by the TMA engine with the 128-byte swizzle and described to the
// tensor core by the matching shared-memory descriptor.  Every wait is bounded
// (WaitGuard); on a timeout all roles stop issuing, in-flight copies and MMAs
// are drained with a second wait of a fixed, generous limit (kDrainLimitNs), TMEM
// is freed and the kernel returns with the timeout bit set in the status word.
#pragma once

#include "ptx.cuh"

namespace fpo {

constexpr int kBM = 128;       // UMMA M (one TMEM lane per output row)
constexpr int kBK = 64;        // k-block: 64 bf16 = one 128-byte swizzle row
constexpr int kUmmaK = 16;     // K of one tcgen05.mma.kind::f16
// Threads of a GEMM kernel: the producer and MMA warps, then the epilogue's.
template <class Epi>
constexpr int gemm_threads() {
    return 64 + 32 * Epi::kWarps;
}
constexpr int kMaxGroups = 64;
// Limit of the teardown waits for copies and MMAs already issued (they complete in
// microseconds); fixed, so that a short wait limit cannot cut them off.
constexpr uint64_t kDrainLimitNs = 1000000000ull;

struct GemmShape {
    int M, N, K;
    int m_blocks, n_blocks, k_blocks;
    int groups;        // independent problems with equal shapes (target layers)
    int band;          // rasterisation band height in m-blocks (L2 reuse)
    long long tiles;   // groups * m_blocks * n_blocks
    // Split-K tail (pair kernel only): the last tail_tiles tiles (less than one wave)
    // are each split into tail_split equal k-block ranges, and every range leaves its
    // fp32 sums in sk_scratch ([unit][256][BN]) for a fixup kernel.  0 = whole tiles.
    long long tail_tiles;
    int tail_split;
    float* sk_scratch;
    // Pair kernel only: when set, the number of rows of A is read here on the device at
    // kernel start (at most M; the tensor maps cover M rows) and the tiles beyond it are
    // dropped; with no rows the kernel returns before it sets anything up.
    const int* m_dev;
};

template <int MAXG>
struct GemmMaps {
    CUtensorMap a[MAXG];    // one per group (copies of one map when the groups share A)
    CUtensorMap b[MAXG];    // one per group
};

// Output staging for TMA stores: per epilogue warp two 4 KB buffers, each a
// 32-row x 128-byte tile in the 128-byte-swizzled layout (1024-byte aligned).
constexpr int kOutBufBytes = 4096;
constexpr int kOutBytesPerWarp = 2 * kOutBufBytes;

template <int BN, int STAGES>
struct GemmSmem {
    static constexpr int kABytes = kBM * kBK * 2;
    static constexpr int kBBytes = BN * kBK * 2;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kOutOffset = STAGES * kStageBytes;
    static constexpr int kBarOffset = kOutOffset + 4 * kOutBytesPerWarp;
    // full[S], empty[S], tmem_full[2], tmem_empty[2], drain[1]
    static constexpr int kNumBars = 2 * STAGES + 5;
    static constexpr int kMiscOffset = kBarOffset + kNumBars * 8;
    static constexpr int kBytes = kMiscOffset + 16 + 1024;  // + alignment slack
};

__device__ __forceinline__ void tile_coords(long long t, const GemmShape& sh, int& g, int& mb,
                                            int& nb) {
    const long long per = static_cast<long long>(sh.m_blocks) * sh.n_blocks;
    g = static_cast<int>(t / per);
    const int local = static_cast<int>(t - static_cast<long long>(g) * per);
    const int per_band = sh.band * sh.n_blocks;
    const int band = local / per_band;
    const int first_m = band * sh.band;
    const int h = min(sh.m_blocks - first_m, sh.band);
    const int r = local - band * per_band;
    mb = first_m + r % h;
    nb = r / h;
}

// Load one operand k-block.  K-major: a single box {64 (K), ROWS}.  MN-major:
// ROWS/64 boxes {64 (M or N), 64 (K)}, each 8 KB, stacked along M/N.
template <bool MN, int ROWS>
__device__ __forceinline__ void load_operand(const CUtensorMap* map, uint32_t dst, uint32_t bar,
                                             int row0, int k0) {
    if constexpr (!MN) {
        tma_load_2d(map, dst, bar, k0, row0);
    } else {
#pragma unroll
        for (int i = 0; i < ROWS / 64; ++i) tma_load_2d(map, dst + i * (64 * kBK * 2), bar, row0 + 64 * i, k0);
    }
}

// Descriptor of the kk-th K=16 slice of an operand k-block.
//  K-major SW128: rows of 128 B (64 K-elements), 8-row groups 1024 B apart
//                 (SBO); the K slice starts 32 B further along the row.
//  MN-major SW128: 64-element MN chunks of 64 K-rows (8 KB, LBO apart), 8-row
//                 K groups 1024 B apart (SBO); the K slice starts 16 rows
//                 (2048 B) further down.
template <bool MN>
__device__ __forceinline__ uint64_t operand_desc(uint32_t base, int kk) {
    if constexpr (!MN)
        return smem_desc_sw128(base + kk * (kUmmaK * 2), 16, 1024);
    else
        return smem_desc_sw128(base + kk * (kUmmaK * 128), 64 * kBK * 2, 1024);
}

// Per-warp output context of the epilogue: the warp's staging buffers and the
// count of TMA stores it issued (which buffer is next).  All decisions that
// touch it are warp-uniform.
struct EpiIO {
    uint32_t out;     // shared address of this warp's two staging buffers
    int lane;
    int row0;         // absolute output row of lane 0 of this warp
    uint32_t count;   // stores issued so far
};

// Next staging buffer, once the store that last used it has read it.
__device__ __forceinline__ uint32_t out_acquire(const EpiIO& io) {
    if (io.lane == 0) bulk_wait_group_read<1>();
    __syncwarp();
    return io.out + (io.count & 1u) * kOutBufBytes;
}

// Each thread writes its 128-byte row r (32 words) of a staging buffer: 16-byte
// piece c goes to position c ^ (r mod 8), the 128-byte swizzle the TMA store
// undoes; 8 consecutive rows hit 8 different bank groups.
__device__ __forceinline__ void out_stage_row(uint32_t buf, int r, const uint32_t (&w)[32]) {
    const uint32_t row = buf + static_cast<uint32_t>(r) * 128u;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        st_shared_v4(row + ((static_cast<uint32_t>(c) ^ (static_cast<uint32_t>(r) & 7u)) << 4),
                     w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
}

// Chunks of the 8-warp epilogues: kRows of the warp's 32 rows x kCols of its fp32 columns
// (half of the tile's: 128 or 64), staged in the warp's 4 KB of output staging by the lanes
// that hold the rows and read back with kLanes lanes to a row, 4 columns each, so that every
// global access of a warp covers kCols consecutive columns of kAccRows rows.  16-byte pieces
// are swizzled by row, so neither side has bank conflicts.
struct RowChunk {
    static constexpr int kRows = 16;
    static constexpr int kCols = 1024 / kRows;
    static constexpr int kLanes = kCols / 4;
    static constexpr int kAccRows = 32 / kLanes;           // rows of one access
    static constexpr int kAcc = kRows / kAccRows;          // accesses per chunk (8)
    static __device__ __forceinline__ uint32_t piece(uint32_t buf, uint32_t r, uint32_t c) {
        return buf + r * (kCols * 4u) + ((c ^ (r & 7u)) << 4);
    }
    // Columns [32 h, 32 h + 32) of the chunk's, one row per lane; the rows of row group rg
    // go to the staging buffer.
    static __device__ __forceinline__ void stage(uint32_t buf, int lane, int rg, int h,
                                                 const float (&v)[32]) {
        if (lane / kRows != rg) return;
        const uint32_t r = static_cast<uint32_t>(lane % kRows);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            st_shared_v4(piece(buf, r, static_cast<uint32_t>(8 * h + k)),
                         __float_as_uint(v[4 * k]), __float_as_uint(v[4 * k + 1]),
                         __float_as_uint(v[4 * k + 2]), __float_as_uint(v[4 * k + 3]));
    }
    // Access i of the staged chunk: row kAccRows i + lane / kLanes, columns
    // 4 (lane mod kLanes) .. of it.
    static __device__ __forceinline__ float4 read(uint32_t buf, int lane, int i) {
        return ld_shared_f4(piece(buf, static_cast<uint32_t>(kAccRows * i + lane / kLanes),
                                  static_cast<uint32_t>(lane % kLanes)));
    }
};

// The epilogue's warps.  With Epi::kWarps = 4 each warp owns 32 rows of the CTA's 128 and
// walks all BN columns, one row per thread (Epi(params, group, row, n0); chunk(params,
// v[32], column, offset in the tile, io); finish(params, n_block)).  With 8, two warps
// share the rows and take half of the columns each, and every chunk goes through the warp's
// staging buffer (RowChunk; Epi(params, group, first row, first column, lane);
// chunk(params, staged chunk, lane, chunk index); finish(params, lane)).  The functor
// is made before the accumulator is awaited, so that what its constructor loads arrives
// during the mainloop.  `ready` waits for the accumulator (false: give up), `release`
// gives it back once its last columns are in registers.
template <int BN, class Epi, class Ready, class Release>
__device__ __forceinline__ bool epilogue_tile(const typename Epi::Params& ep, int g, int row0,
                                              int nb, int warp_half, uint32_t t_row, EpiIO& io,
                                              Ready ready, Release release) {
    if constexpr (Epi::kWarps == 4) {
        const int n0 = nb * BN;
        io.row0 = row0;
        Epi epi(ep, g, row0 + io.lane, n0);
        if (!ready()) return false;
#pragma unroll 1
        for (int c = 0; c < BN / 32; ++c) {
            float v[32];
            tmem_ld_32x32b_x32(t_row + c * 32, v);
            if (c == BN / 32 - 1) release();
            epi.chunk(ep, v, n0 + c * 32, c * 32, io);
        }
        epi.finish(ep, nb);
    } else {
        using R = RowChunk;
        constexpr int kWarpCols = BN / 2, kColGroups = Epi::kColGroups;
        static_assert(kWarpCols == kColGroups * R::kCols, "the epilogue's share of the columns");
        constexpr int kChunks = 32 / R::kRows * kColGroups;
        const int c0 = warp_half * kWarpCols;
        Epi epi(ep, g, row0, nb * BN + c0, io.lane);
        if (!ready()) return false;
#pragma unroll 1
        for (int c = 0; c < kChunks; ++c) {
            // every lane reads its row's columns again for each row group
#pragma unroll 1
            for (int h = 0; h < R::kCols / 32; ++h) {
                float v[32];
                tmem_ld_32x32b_x32(t_row + c0 + (c % kColGroups) * R::kCols + 32 * h, v);
                if (c == kChunks - 1 && h == R::kCols / 32 - 1) release();
                R::stage(io.out, io.lane, c / kColGroups, h, v);
                __syncwarp();
            }
            epi.chunk(ep, io.out, io.lane, c);
            __syncwarp();
        }
        epi.finish(ep, io.lane);
    }
    return true;
}

// Store a filled staging buffer to (x, y) of `map` (rows/columns outside the
// tensor are clipped by the TMA engine).
__device__ __forceinline__ void out_commit(EpiIO& io, const CUtensorMap* map, uint32_t buf, int x,
                                           int y) {
    fence_proxy_async_smem();
    __syncwarp();
    if (io.lane == 0) {
        tma_store_2d(map, buf, x, y);
        bulk_commit_group();
    }
    ++io.count;
}

template <int BN, bool A_MN, bool B_MN, int STAGES, int MAXG, class Epi>
__global__ void __launch_bounds__(gemm_threads<Epi>(), 1)
    tc_gemm_kernel(const __grid_constant__ GemmMaps<MAXG> maps,
                   const __grid_constant__ typename Epi::Params ep, const GemmShape sh,
                   unsigned int* status, unsigned long long wait_limit_ns) {
    using L = GemmSmem<BN, STAGES>;
    constexpr uint32_t kIdesc = idesc_bf16_f32(kBM, BN, A_MN, B_MN);
    constexpr int kTmemCols = 2 * BN;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
    uint8_t* smem = smem_raw + pad;
    const uint32_t sbase = raw + pad;

    const uint32_t bar0 = sbase + L::kBarOffset;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
    auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * STAGES + a); };
    auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * STAGES + 2 + a); };
    const uint32_t drain_bar = bar0 + 8u * (2 * STAGES + 4);
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + L::kMiscOffset);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kMiscOffset + 4);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(tfull_bar(a), 1);
            mbar_init(tempty_bar(a), Epi::kWarps);
        }
        mbar_init(drain_bar, 1);
        *abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&maps.a[0]);
    }
    if (warp == 1) {
        tmem_alloc<kTmemCols>(smem_u32(tmem_holder));
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    grid_dependency_wait();

    const WaitGuard guard{abort_flag, status, wait_limit_ns};

    if (warp == 0) {
        // ------------------------------------------------------- TMA producer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t issued_mask = 0;       // stages with a copy issued
            uint32_t issued_parity = 0;     // parity of that copy's phase
            bool ok = true;
            for (long long t = blockIdx.x; t < sh.tiles && ok; t += gridDim.x) {
                int g, mb, nb;
                tile_coords(t, sh, g, mb, nb);
                const CUtensorMap* amap = &maps.a[MAXG == 1 ? 0 : g];
                const CUtensorMap* bmap = &maps.b[MAXG == 1 ? 0 : g];
                for (int kb = 0; kb < sh.k_blocks; ++kb) {
                    if (!mbar_wait(empty_bar(stage), phase ^ 1u, guard)) { ok = false; break; }
                    const uint32_t sa = sbase + stage * L::kStageBytes;
                    const uint32_t sb = sa + L::kABytes;
                    mbar_arrive_expect_tx(full_bar(stage), L::kStageBytes);
                    load_operand<A_MN, kBM>(amap, sa, full_bar(stage), mb * kBM, kb * kBK);
                    load_operand<B_MN, BN>(bmap, sb, full_bar(stage), nb * BN, kb * kBK);
                    issued_mask |= 1u << stage;
                    issued_parity = (issued_parity & ~(1u << stage)) | (phase << stage);
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
            }
            grid_dependency_trigger();  // only the last tiles' MMAs and epilogues are left
            // Do not leave copies landing in shared memory after exit: the last copy of
            // every stage is awaited (at once when it was consumed), also when another
            // role gave up first.
            for (int s = 0; s < STAGES; ++s)
                if (issued_mask & (1u << s))
                    mbar_wait_drain(full_bar(s), (issued_parity >> s) & 1u, kDrainLimitNs);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------- MMA issuer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            int acc = 0;
            uint32_t acc_phase = 0;
            bool ok = true, issued_any = false;
            for (long long t = blockIdx.x; t < sh.tiles && ok; t += gridDim.x) {
                if (!mbar_wait(tempty_bar(acc), acc_phase ^ 1u, guard)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * BN);
                for (int kb = 0; kb < sh.k_blocks; ++kb) {
                    if (!mbar_wait(full_bar(stage), phase, guard)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sa = sbase + stage * L::kStageBytes;
                    const uint32_t sb = sa + L::kABytes;
#pragma unroll
                    for (int kk = 0; kk < kBK / kUmmaK; ++kk) {
                        tc_mma_bf16(d_tmem, operand_desc<A_MN>(sa, kk), operand_desc<B_MN>(sb, kk),
                                    kIdesc, (kb | kk) != 0 ? 1u : 0u);
                    }
                    issued_any = true;
                    tc_commit(empty_bar(stage));
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                tc_commit(tfull_bar(acc));
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
            if (issued_any) {
                // Wait for the MMAs already issued before TMEM and smem go away (also
                // when only the epilogue gave up).
                tc_commit(drain_bar);
                mbar_wait_drain(drain_bar, 0, kDrainLimitNs);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------- epilogue
        const int q = warp & 3;  // TMEM lane quarter this warp may access
        constexpr int kOutPerWarp = 4 * kOutBytesPerWarp / Epi::kWarps;
        EpiIO io{sbase + L::kOutOffset + static_cast<uint32_t>((warp - 2) * kOutPerWarp), lane, 0,
                 0u};
        int acc = 0;
        uint32_t acc_phase = 0;
        for (long long t = blockIdx.x; t < sh.tiles; t += gridDim.x) {
            int g, mb, nb;
            tile_coords(t, sh, g, mb, nb);
            const uint32_t t_row = tmem_base + (static_cast<uint32_t>(q * 32) << 16) +
                                   static_cast<uint32_t>(acc * BN);
            const bool ok = epilogue_tile<BN, Epi>(
                ep, g, mb * kBM + q * 32, nb, (warp - 2) / 4, t_row, io,
                [&] {
                    if (!mbar_wait(tfull_bar(acc), acc_phase, guard)) return false;
                    tc_fence_after();
                    return true;
                },
                [&] {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty_bar(acc));
                });
            if (!ok) break;
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (lane == 0) bulk_wait_group_all();  // stores done before shared memory goes away
        __syncwarp();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc<kTmemCols>(tmem_base);
    }
}

}  // namespace fpo
