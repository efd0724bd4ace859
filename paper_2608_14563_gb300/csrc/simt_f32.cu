// simt_f32.cu -- true-fp32 (FFMA, no TF32) GEMMs of the FPO step for dtype
// FPO_F32, with the same four epilogues as the tensor-core path:
//
//   C[m, n] = sum_k A(m, k) B(n, k),  A(m,k) = A[m*sam + k*sak], B(n,k) = B[n*sbn + k*sbk]
//
// 256 threads per block and square output tiles of 128 (8 x 8 outputs per thread) or 64
// (4 x 4), 16-deep k slices double-buffered in shared memory (the next slice is loaded
// into registers while the current one is multiplied), packed f32x2 FMAs.  A block
// cluster of up to 8 blocks can share one tile: each block sums its own range of the k
// slices, the partial sums meet through distributed shared memory in rank order, and each
// block applies the epilogue to its share of the rows.  Any shape is accepted; operands
// and outputs whose rows are 16-byte aligned take 16-byte accesses.
//
// Bound: the FMA pipe.  128-tiles keep it 69% busy over a long launch (logits pass of
// T 777, d 768, V 32001: 1510 us with 64 x 64 tiles and one slice in flight, 850 us now);
// 8 x 16 outputs per thread, scalar FMAs or 32-deep slices were slower (930, 877 and 991
// us).  The split along K is for outputs too small to fill the SMs: the projection of those
// sizes 3154 -> 980 us, at T 128, d 64, V 512 27 -> 10 us.
#include <cuda_runtime.h>
#include <math.h>

#include <atomic>
#include <type_traits>

#include "error_math.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace fpo {
namespace {

constexpr int kKs = 16;         // depth of a k slice
constexpr int kThreads = 256;
constexpr int kMaxG = 64;
constexpr int kMaxSplit = 8;    // portable cluster size

struct SimtOps {
    const float* A[kMaxG];
    const float* B[kMaxG];
    long long lda, ldb;         // stride of the non-contiguous index
    int M, N, K;
    int m_tiles, splits;
    bool vec_a, vec_b;          // 16-byte loads (lda / ldb a multiple of 4)
};

// ------------------------------------------------------------------ epilogues
struct SEpiLse {  // per (row, 64-column tile): (max, sum exp(z - max)) and z_{t,y_t}
    float2* part;
    int part_ld;
    float* zy;
    const int32_t* y;
    float* z;       // [M, ldz] logits for the stored-logits algorithm, or null
    long long ldz;  // a multiple of 4
};
struct SEpiError {  // E = s (exp(z - lse) - [col == y])
    float* E;
    long long ldE;  // a multiple of 4
    const float* lse;
    const int32_t* y;
    float s;
};
struct SEpiStore {
    float* C;
    long long ld;
};
struct SEpiSwiglu {  // dA = e b silu'(a), dB = e silu(a) from e = g W3 and cached a, b
    float* dA;
    float* dB;
    const float* a;
    const float* b;
    long long ld;
};
struct SEpiUpdate {
    float* W_master[kMaxG];
    float* W_out[kMaxG];
    float* G_out[kMaxG];
    long long ld;
    float neg_lr;
};

// Butterflies over the 16 lanes that share a row.
__device__ __forceinline__ float hmax16(float x) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}
__device__ __forceinline__ float hsum16(float x) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Up to 4 consecutive floats of a row, n of them inside it; vec: p is 16-byte aligned.
__device__ __forceinline__ float4 ld4(const float* p, int n, bool vec) {
    if (n >= 4 && vec) return *reinterpret_cast<const float4*>(p);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n > 0) v.x = p[0];
    if (n > 1) v.y = p[1];
    if (n > 2) v.z = p[2];
    if (n > 3) v.w = p[3];
    return v;
}
__device__ __forceinline__ void st4(float* p, const float (&v)[4], int n, bool vec) {
    if (n >= 4 && vec) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
        return;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (j < n) p[j] = v[j];
}

// One operand's k slice: BT rows (M or N) x 16 k, kV vectors of 4 per thread.
// kKC: k is contiguous in memory (a vector runs along k and is scattered to four rows of
// the transposed shared tile); otherwise the row index is contiguous.
template <int BT, bool kKC>
struct SliceLoader {
    static constexpr int kV = BT * kKs / 4 / kThreads;
    static constexpr int kLd = BT + 4;
    float4 r[kV];

    __device__ __forceinline__ void load(const float* p, long long ld, int row0,
                                         int rows, int k0, int K, bool vec) {
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            const int idx = threadIdx.x + kThreads * q;
            if constexpr (kKC) {
                const int row = row0 + (idx >> 2), k = k0 + 4 * (idx & 3);
                r[q] = row < rows ? ld4(p + row * ld + k, K - k, vec)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
                constexpr int kPerK = BT / 4;
                const int k = k0 + idx / kPerK, row = row0 + 4 * (idx % kPerK);
                r[q] = k < K ? ld4(p + k * ld + row, rows - row, vec)
                             : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    }

    __device__ __forceinline__ void store(float* s) const {
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            const int idx = threadIdx.x + kThreads * q;
            if constexpr (kKC) {
                float* d = s + 4 * (idx & 3) * kLd + (idx >> 2);
                d[0] = r[q].x;
                d[kLd] = r[q].y;
                d[2 * kLd] = r[q].z;
                d[3 * kLd] = r[q].w;
            } else {
                constexpr int kPerK = BT / 4;
                *reinterpret_cast<float4*>(s + (idx / kPerK) * kLd + 4 * (idx % kPerK)) = r[q];
            }
        }
    }
};

// Thread (tx, ty) of 16 x 16 owns rows 64 i + 4 ty + 0..3 and columns 64 h + 4 tx + 0..3 of
// the tile for i, h < BT / 64.
template <int BT, bool kAKC, bool kBKC, class Epi>
__global__ void __launch_bounds__(kThreads, 2)
    simt_gemm_kernel(const __grid_constant__ SimtOps ops, const __grid_constant__ Epi ep) {
    constexpr int kH = BT / 64;          // 64-wide halves of the tile
    constexpr int kLd = BT + 4;
    constexpr int kBuf = 2 * kKs * kLd;  // floats of one stage: A slice, then B slice
    constexpr int kR = 4 * kH;           // rows (and columns) per thread
    extern __shared__ __align__(16) float sm[];
    const int S = ops.splits;
    const int g = blockIdx.y / S, rank = blockIdx.y % S;  // cluster rank = blockIdx.y % S
    const int m0 = (blockIdx.x % ops.m_tiles) * BT, n0 = (blockIdx.x / ops.m_tiles) * BT;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const float* A = ops.A[g];
    const float* B = ops.B[g];
    const int slices = (ops.K + kKs - 1) / kKs;
    const int s0 = static_cast<int>(static_cast<long long>(rank) * slices / S);
    const int s1 = static_cast<int>(static_cast<long long>(rank + 1) * slices / S);

    float2 acc[kR][2 * kH];
#pragma unroll
    for (int i = 0; i < kR; ++i)
#pragma unroll
        for (int j = 0; j < 2 * kH; ++j) acc[i][j] = make_float2(0.f, 0.f);

    grid_dependency_wait();
    SliceLoader<BT, kAKC> la;
    SliceLoader<BT, kBKC> lb;
    if (s0 < s1) {
        la.load(A, ops.lda, m0, ops.M, s0 * kKs, ops.K, ops.vec_a);
        lb.load(B, ops.ldb, n0, ops.N, s0 * kKs, ops.K, ops.vec_b);
        la.store(sm);
        lb.store(sm + kKs * kLd);
    }
    __syncthreads();
    for (int s = s0; s < s1; ++s) {
        const float* as = sm + ((s - s0) & 1) * kBuf;
        const float* bs = as + kKs * kLd;
        if (s + 1 < s1) {
            la.load(A, ops.lda, m0, ops.M, (s + 1) * kKs, ops.K, ops.vec_a);
            lb.load(B, ops.ldb, n0, ops.N, (s + 1) * kKs, ops.K, ops.vec_b);
        }
        // (128-tiles unrolled by 2: the logits pass 905 us instead of 852; 4 and 16 slower)
        constexpr int kUnroll = BT == 128 ? 1 : 2;
#pragma unroll kUnroll
        for (int kk = 0; kk < kKs; ++kk) {
            float a[kR];
            float2 b[2 * kH];
#pragma unroll
            for (int h = 0; h < kH; ++h) {
                const float4 v =
                    *reinterpret_cast<const float4*>(as + kk * kLd + 64 * h + 4 * ty);
                a[4 * h] = v.x;
                a[4 * h + 1] = v.y;
                a[4 * h + 2] = v.z;
                a[4 * h + 3] = v.w;
            }
#pragma unroll
            for (int h = 0; h < kH; ++h) {
                const float4 v =
                    *reinterpret_cast<const float4*>(bs + kk * kLd + 64 * h + 4 * tx);
                b[2 * h] = make_float2(v.x, v.y);
                b[2 * h + 1] = make_float2(v.z, v.w);
            }
#pragma unroll
            for (int i = 0; i < kR; ++i)
#pragma unroll
                for (int j = 0; j < 2 * kH; ++j)
                    acc[i][j] = __ffma2_rn(make_float2(a[i], a[i]), b[j], acc[i][j]);
        }
        if (s + 1 < s1) {
            float* nx = sm + ((s + 1 - s0) & 1) * kBuf;
            la.store(nx);
            lb.store(nx + kKs * kLd);
            __syncthreads();
        }
    }

    grid_dependency_trigger();
    // k ranges of the cluster: every block leaves its sums in shared memory, thread by
    // thread, and block `rank` adds the rows i with i mod S = rank in rank order
    if (S > 1) {
        __syncthreads();  // the stages are free
        float4* x = reinterpret_cast<float4*>(sm);
#pragma unroll
        for (int i = 0; i < kR; ++i)
#pragma unroll
            for (int h = 0; h < kH; ++h)
                x[(i * kH + h) * kThreads + threadIdx.x] =
                    make_float4(acc[i][2 * h].x, acc[i][2 * h].y, acc[i][2 * h + 1].x,
                                acc[i][2 * h + 1].y);
        cluster_sync();
        const uint32_t own = smem_u32(sm) + threadIdx.x * 16u;
#pragma unroll
        for (int i = 0; i < kR; ++i) {
            if (i % S != rank) continue;
#pragma unroll
            for (int h = 0; h < kH; ++h) {
                float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int q = 0; q < S; ++q) {
                    const float4 u = ld_shared_cluster_f4(mapa_shared(
                        own + static_cast<uint32_t>((i * kH + h) * kThreads * 16), q));
                    t.x += u.x;
                    t.y += u.y;
                    t.z += u.z;
                    t.w += u.w;
                }
                acc[i][2 * h] = make_float2(t.x, t.y);
                acc[i][2 * h + 1] = make_float2(t.z, t.w);
            }
        }
        cluster_sync();  // no block leaves while another reads its shared memory
    }

#pragma unroll
    for (int i = 0; i < kR; ++i) {
        if (S > 1 && i % S != rank) continue;
        const int row = m0 + 64 * (i / 4) + 4 * ty + i % 4;
        const bool rv = row < ops.M;
        if constexpr (std::is_same_v<Epi, SEpiLse>) {
            // all 16 threads sharing this row take part in the reductions
            const int yt = rv ? ep.y[row] : -1;
#pragma unroll
            for (int h = 0; h < kH; ++h) {
                const int col = n0 + 64 * h + 4 * tx;
                const int nv = ops.N - col;  // columns inside the matrix (4 or more: all)
                const float v[4] = {acc[i][2 * h].x, acc[i][2 * h].y, acc[i][2 * h + 1].x,
                                    acc[i][2 * h + 1].y};
                float mx = -INFINITY;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j < nv) mx = fmaxf(mx, v[j]);
                mx = hmax16(mx);
                float s = 0.f;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j < nv) {
                        s += expf(v[j] - mx);
                        if (rv && col + j == yt && ep.zy) ep.zy[row] = v[j];
                    }
                }
                s = hsum16(s);
                if (rv && ep.z && nv > 0) st4(ep.z + row * ep.ldz + col, v, nv, true);
                if (rv && tx == 0 && n0 + 64 * h < ops.N)
                    ep.part[static_cast<long long>(row) * ep.part_ld + n0 / 64 + h] =
                        make_float2(mx, s);
            }
        } else {
            if (!rv) continue;
#pragma unroll
            for (int h = 0; h < kH; ++h) {
                const int col = n0 + 64 * h + 4 * tx;
                const int nv = ops.N - col;  // columns inside the matrix (4 or more: all)
                if (nv <= 0) continue;
                const float v[4] = {acc[i][2 * h].x, acc[i][2 * h].y, acc[i][2 * h + 1].x,
                                    acc[i][2 * h + 1].y};
                if constexpr (std::is_same_v<Epi, SEpiError>) {
                    const float l = ep.lse[row];
                    const int yt = ep.y[row];
                    float e[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) e[j] = error_value_f32(v[j], l, col + j == yt, ep.s);
                    st4(ep.E + row * ep.ldE + col, e, nv, true);
                } else if constexpr (std::is_same_v<Epi, SEpiStore>) {
                    st4(ep.C + row * ep.ld + col, v, nv, (ep.ld & 3) == 0);
                } else if constexpr (std::is_same_v<Epi, SEpiSwiglu>) {
                    const long long off = row * ep.ld + col;
                    const bool vec = (ep.ld & 3) == 0;
                    const float4 a4 = ld4(ep.a + off, nv, vec), b4 = ld4(ep.b + off, nv, vec);
                    const float xa[4] = {a4.x, a4.y, a4.z, a4.w}, xb[4] = {b4.x, b4.y, b4.z, b4.w};
                    float da[4], db[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float sg = 1.f / (1.f + expf(-xa[j]));
                        da[j] = v[j] * xb[j] * sg * fmaf(xa[j], 1.f - sg, 1.f);
                        db[j] = v[j] * xa[j] * sg;
                    }
                    st4(ep.dA + off, da, nv, vec);
                    st4(ep.dB + off, db, nv, vec);
                } else {
                    const long long off = row * ep.ld + col;
                    const bool vec = (ep.ld & 3) == 0;
                    if (float* wm = ep.W_master[g]) {
                        const float4 w4 = ld4(wm + off, nv, vec);
                        const float nw[4] = {fmaf(ep.neg_lr, v[0], w4.x), fmaf(ep.neg_lr, v[1], w4.y),
                                             fmaf(ep.neg_lr, v[2], w4.z), fmaf(ep.neg_lr, v[3], w4.w)};
                        st4(wm + off, nw, nv, vec);
                        if (ep.W_out[g]) st4(ep.W_out[g] + off, nw, nv, vec);
                    }
                    if (ep.G_out[g]) st4(ep.G_out[g] + off, v, nv, vec);
                }
            }
        }
    }
}

std::atomic<int> g_simt_tile{0};  // > 0: tile width (tests)

int sm_count() {
    DevInfo di;
    return current_device_info(&di) ? di.sm_count : 148;
}

// Estimated cycles of one launch on tiles of BT.  A 16-deep slice measured 3350 (BT 128) or
// 1350 (BT 64) cycles of a block alone on its SM and 2900 or 1080 per block when two share
// it.  Clusters of more than 4 blocks do not pack the GPCs' SMs tightly: about a tenth of
// the slots stay empty, and a launch beyond them takes a second wave (the fp32 projection
// of 42 tiles, K = 32001: 981 us in clusters of 6, 1229 of 7, 1090 of 8).
double simt_cost(int BT, long long tiles, int slices, int S, int sms) {
    const double alone = BT == 128 ? 3350.0 : 1350.0, shared = BT == 128 ? 2900.0 : 1080.0;
    const long long cap = S > 4 ? (2LL * sms / S) * 9 / 10 : 2LL * sms / S;  // clusters at once
    const long long full = tiles / cap, rem = tiles % cap;
    const double last = rem == 0 ? 0.0 : rem * S <= sms ? alone : 2 * shared;
    return ((slices + S - 1) / S) * (full * 2 * shared + last) + (S > 1 ? 3000.0 : 0.0);
}

long long simt_tiles(int M, int N, int BT) {
    return static_cast<long long>((M + BT - 1) / BT) * ((N + BT - 1) / BT);
}

// Blocks per cluster along K: from the problem's own size only (M_ref: the rows of the
// whole batch, not of a token chunk; one layer of a group), so that every chunking and
// grouping sums each output in the same order.  At least 4 slices per block.
int simt_split(int M_ref, int N, int K) {
    const int sms = sm_count(), slices = (K + kKs - 1) / kKs;
    int best_s = 1;
    double best = 0.0;
    for (int S = 1; S <= kMaxSplit && (S == 1 || slices / S >= 4); ++S) {
        const double c = fmin(simt_cost(128, simt_tiles(M_ref, N, 128), slices, S, sms),
                              simt_cost(64, simt_tiles(M_ref, N, 64), slices, S, sms));
        if (S == 1 || c < 0.97 * best) {
            best = c;
            best_s = S;
        }
    }
    return best_s;
}

template <int BT, bool kAKC, bool kBKC, class Epi>
cudaError_t run_tile(SimtOps ops, const Epi& ep, int groups, cudaStream_t st) {
    constexpr auto kern = simt_gemm_kernel<BT, kAKC, kBKC, Epi>;
    constexpr int kStage = 2 * 2 * kKs * (BT + 4) * 4;  // two stages of both slices
    constexpr int kExchange = BT * BT * 4;              // one tile of sums
    const int smem = ops.splits > 1 && kExchange > kStage ? kExchange : kStage;
    const cudaError_t attr = set_smem_limit<kern>(kExchange > kStage ? kExchange : kStage);
    if (attr != cudaSuccess) return attr;
    ops.m_tiles = (ops.M + BT - 1) / BT;
    const long long tiles = simt_tiles(ops.M, ops.N, BT);
    if (tiles > 0x7fffffffll) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(tiles), static_cast<unsigned>(groups * ops.splits), 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = static_cast<size_t>(smem);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_chained
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 1;
    at[1].val.clusterDim.y = static_cast<unsigned>(ops.splits);
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = ops.splits > 1 ? 2 : 1;
    note_launch();
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, ops, ep);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}


// Tiles of 128 or 64, whichever simt_cost estimates faster (the same sums either way).
template <bool kAKC, bool kBKC, class Epi>
cudaError_t run(const SimtOps& ops, const Epi& ep, int groups, cudaStream_t st) {
    if (ops.M <= 0 || ops.N <= 0) return cudaSuccess;
    const int sms = sm_count(), slices = (ops.K + kKs - 1) / kKs;
    const double c128 = simt_cost(128, groups * simt_tiles(ops.M, ops.N, 128), slices, ops.splits, sms);
    const double c64 = simt_cost(64, groups * simt_tiles(ops.M, ops.N, 64), slices, ops.splits, sms);
    const int tile = g_simt_tile.load(std::memory_order_relaxed);
    if (tile ? tile == 128 : c128 <= c64) return run_tile<128, kAKC, kBKC>(ops, ep, groups, st);
    return run_tile<64, kAKC, kBKC>(ops, ep, groups, st);
}

// A single problem: lda / ldb are the strides of the non-contiguous index.
SimtOps ops_of(const float* A, long long lda, const float* B, long long ldb, int M, int N, int K,
               int M_ref) {
    SimtOps o = {};
    o.A[0] = A;
    o.B[0] = B;
    o.lda = lda;
    o.ldb = ldb;
    o.M = M;
    o.N = N;
    o.K = K;
    o.splits = simt_split(M_ref, N, K);
    o.vec_a = lda % 4 == 0;  // the bases are 16-byte aligned
    o.vec_b = ldb % 4 == 0;
    return o;
}

}  // namespace

int simt_tile() { return g_simt_tile.load(std::memory_order_relaxed); }
void set_simt_tile(int tile) {
    g_simt_tile.store(tile == 64 || tile == 128 ? tile : 0, std::memory_order_relaxed);
}

cudaError_t launch_lse_partial_f32(const float* yhat, const float* W_U, const int32_t* y, int T,
                                   int T_all, int d, int V, float2* part, int part_ld, float* zy,
                                   float* z, long long ldz, cudaStream_t st) {
    SEpiLse ep{part, part_ld, zy, y, z, ldz};
    return run<true, true>(ops_of(yhat, d, W_U, d, T, V, d, T_all), ep, 1, st);
}

cudaError_t launch_error_f32(const float* yhat, const float* W_U, const int32_t* y,
                             const float* lse, int Tc, int T_all, int d, int V, float s, float* E,
                             long long ldE, cudaStream_t st) {
    SEpiError ep{E, ldE, lse, y, s};
    return run<true, true>(ops_of(yhat, d, W_U, d, Tc, V, d, T_all), ep, 1, st);
}

cudaError_t launch_proj_f32(const float* E, long long ldE, const float* W_U, int Tc, int T_all,
                            int d, int V, float* g, cudaStream_t st) {
    // g[t, j] = sum_v E[t, v] W_U[v, j]: B(n=j, k=v) = W_U[v*d + j]
    SEpiStore ep{g, d};
    return run<true, false>(ops_of(E, ldE, W_U, d, Tc, d, V, T_all), ep, 1, st);
}

cudaError_t launch_swiglu_f32(int T, int d, int d_ff, const float* g, const float* W3,
                              const float* a, const float* b, float* dA, float* dB,
                              cudaStream_t st) {
    // e[t, f] = sum_j g[t, j] W3[j, f]: A(m=t, k=j) = g[t*d + j], B(n=f, k=j) = W3[j*d_ff + f]
    SEpiSwiglu ep{dA, dB, a, b, d_ff};
    return run<true, false>(ops_of(g, d, W3, d_ff, T, d_ff, d, T), ep, 1, st);
}

cudaError_t launch_update_f32(int n, int T, int d, int d_ff, const float* const* g,
                              const float* const* A, float lr, float* const* W_master,
                              float* const* W_out, float* const* G_out, cudaStream_t st) {
    if (n < 1 || n > kMaxG) return cudaErrorInvalidValue;
    // G[i, j] = sum_t g[t, i] A[t, j]: A-operand(m=i, k=t) = g[t*d + i], B(n=j, k=t) = A[t*d_ff + j]
    SimtOps ops = ops_of(g[0], d, A[0], d_ff, d, d_ff, T, d);
    SEpiUpdate ep = {};
    for (int l = 0; l < n; ++l) {
        ops.A[l] = g[l];
        ops.B[l] = A[l];
        ep.W_master[l] = W_master ? W_master[l] : nullptr;
        ep.W_out[l] = W_out ? W_out[l] : nullptr;
        ep.G_out[l] = G_out ? G_out[l] : nullptr;
    }
    ep.ld = d_ff;
    ep.neg_lr = -lr;
    return run<false, false>(ops, ep, n, st);
}

}  // namespace fpo
