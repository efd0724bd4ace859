// optimizer.cu -- the optimizer step of the target layers on their fp32 master
// copies (Sec. 3.1: AdamW with weight decay, SGD with momentum; App. A: fp32
// masters cast to the working dtype, and each step's relative clip to
// clip_frac * ||W||_F, on the step itself or on the gradient).
//
// bf16 with the step clip: the GEMM's epilogue (EpiOptStep) advances the state and leaves
// the unclipped steps and their norm partials to opt_scale + opt_step_apply below.
// Otherwise, from the pseudogradients G_l (fp32, written by the grouped GEMM):
//   pass 1  optim_norms    per layer, partial sums of ||W||^2, ||G||^2 and
//                          ||step||^2 (step = the unclipped optimizer step)
//   pass 2  optim_scale    per layer, the clip factor from those sums
//   pass 3  optim_apply    W <- W + s * step(c * G), optimizer state, W_out
// Passes 1-2 are skipped without a clip; with bf16 and the clip on the gradient the GEMM's
// epilogue has summed the norms and opt_scale forms the factors.  HBM-bound: 16-byte
// accesses where n is a multiple of 4 (else 4-byte ones), grid of blocks x layers, fp32 per
// thread, fp64 per block, fixed-order reductions.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "internal.h"
#include "optim_math.cuh"
#include "slot_sum.cuh"

namespace fpo {
namespace {

constexpr int kOptThreads = 256;
constexpr int kOptBlocksPerLayerMax = 512;
constexpr int kMaxLayers = 64;

struct LayerPtrs {
    float* G[kMaxLayers];
    float* W[kMaxLayers];
    void* Wo[kMaxLayers];
    float* s1[kMaxLayers];
    float* s2[kMaxLayers];
};

__device__ __forceinline__ double warp_sum_d(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Element i (kV = 1) or elements 4 i .. 4 i + 3 (kV = 4) of an array; zeros for null.
template <int kV>
struct Vec {
    float v[kV];
    __device__ __forceinline__ void load(const float* p, size_t i) {
        if (!p) {
#pragma unroll
            for (int k = 0; k < kV; ++k) v[k] = 0.f;
        } else if constexpr (kV == 4) {
            const float4 x = reinterpret_cast<const float4*>(p)[i];
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        } else {
            v[0] = p[i];
        }
    }
    __device__ __forceinline__ void store(float* p, size_t i) const {
        if constexpr (kV == 4)
            reinterpret_cast<float4*>(p)[i] = make_float4(v[0], v[1], v[2], v[3]);
        else
            p[i] = v[0];
    }
    __device__ __forceinline__ void store(__nv_bfloat16* p, size_t i) const {
        if constexpr (kV == 4) {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(v[0], v[1]);
            const __nv_bfloat162 hi = __floats2bfloat162_rn(v[2], v[3]);
            reinterpret_cast<uint2*>(p)[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&lo),
                                                        *reinterpret_cast<const uint32_t*>(&hi));
        } else {
            p[i] = __float2bfloat16_rn(v[0]);
        }
    }
};

template <int kV>
__global__ void __launch_bounds__(kOptThreads)
    optim_norms_kernel(const __grid_constant__ LayerPtrs lp, size_t n, const OptimParams op,
                       double* __restrict__ partials) {
    const int layer = blockIdx.y;
    const float* G = lp.G[layer];
    const float* W = lp.W[layer];
    // the state is needed for the step's norm only
    const float* S1 = op.clip == 1 ? lp.s1[layer] : nullptr;
    const float* S2 = op.clip == 1 ? lp.s2[layer] : nullptr;
    float ww = 0.f, gg = 0.f, dd = 0.f;
    const size_t stride = static_cast<size_t>(gridDim.x) * kOptThreads;
    for (size_t i = blockIdx.x * static_cast<size_t>(kOptThreads) + threadIdx.x; i < n / kV;
         i += stride) {
        Vec<kV> g, w, s1, s2;
        g.load(G, i);
        w.load(W, i);
        s1.load(S1, i);
        s2.load(S2, i);
#pragma unroll
        for (int k = 0; k < kV; ++k) {
            ww = fmaf(w.v[k], w.v[k], ww);
            gg = fmaf(g.v[k], g.v[k], gg);
            if (op.clip == 1) {
                const float st = opt_step(op, g.v[k], w.v[k], s1.v[k], s2.v[k]);
                dd = fmaf(st, st, dd);
            }
        }
    }
    __shared__ double sh[3][kOptThreads / 32];
    double a = warp_sum_d(ww), b = warp_sum_d(gg), c = warp_sum_d(dd);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        sh[0][wid] = a;
        sh[1][wid] = b;
        sh[2][wid] = c;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double x = 0, y = 0, z = 0;
        for (int k = 0; k < kOptThreads / 32; ++k) {
            x += sh[0][k];
            y += sh[1][k];
            z += sh[2][k];
        }
        double* p = partials + (static_cast<size_t>(layer) * gridDim.x + blockIdx.x) * 3;
        p[0] = x;
        p[1] = y;
        p[2] = z;
    }
}

// One block per layer: thread-strided fp64 sums of the blocks' triples, a fixed butterfly
// per warp, then the warps' sums in warp order (64 us when one thread added them all).
constexpr int kScaleThreads = 256;

__global__ void __launch_bounds__(kScaleThreads)
    optim_scale_kernel(const double* __restrict__ partials, int blocks, const OptimParams op,
                       float* __restrict__ scales) {
    const int layer = blockIdx.x;
    double ww = 0, xx = 0;  // ||W||^2 and the clipped quantity's
    const double* p = partials + static_cast<size_t>(layer) * blocks * 3;
    for (int b = threadIdx.x; b < blocks; b += kScaleThreads) {
        ww += p[3 * b];
        xx += p[3 * b + (op.clip == 1 ? 2 : 1)];
    }
    ww = warp_sum_d(ww);
    xx = warp_sum_d(xx);
    __shared__ double sh[2][kScaleThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        sh[0][wid] = ww;
        sh[1][wid] = xx;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    ww = xx = 0.0;
    for (int k = 0; k < kScaleThreads / 32; ++k) {
        ww += sh[0][k];
        xx += sh[1][k];
    }
    const double lim = static_cast<double>(op.clip_frac) * sqrt(ww);
    scales[layer] = static_cast<float>(sqrt(xx) > lim ? lim / sqrt(xx) : 1.0);
}

template <bool kBf16Out, int kV>
__global__ void __launch_bounds__(kOptThreads)
    optim_apply_kernel(const __grid_constant__ LayerPtrs lp, size_t n, const OptimParams op,
                       const float* __restrict__ scales) {
    using Out = std::conditional_t<kBf16Out, __nv_bfloat16, float>;
    const int layer = blockIdx.y;
    const float* G = lp.G[layer];
    float* W = lp.W[layer];
    float* S1 = lp.s1[layer];
    float* S2 = lp.s2[layer];
    Out* Wo = static_cast<Out*>(lp.Wo[layer]);
    const float sc = scales ? scales[layer] : 1.f;
    const float gscale = op.clip == 2 ? sc : 1.f;
    const float sscale = op.clip == 1 ? sc : 1.f;
    const size_t stride = static_cast<size_t>(gridDim.x) * kOptThreads;
    for (size_t i = blockIdx.x * static_cast<size_t>(kOptThreads) + threadIdx.x; i < n / kV;
         i += stride) {
        Vec<kV> g, w, s1, s2;
        g.load(G, i);
        w.load(W, i);
        s1.load(S1, i);
        s2.load(S2, i);
#pragma unroll
        for (int k = 0; k < kV; ++k) {
            const float st = opt_step(op, gscale * g.v[k], w.v[k], s1.v[k], s2.v[k]);
            w.v[k] = fmaf(sscale, st, w.v[k]);
        }
        w.store(W, i);
        if (S1) s1.store(S1, i);
        if (S2) s2.store(S2, i);
        if (Wo) w.store(Wo, i);
    }
}

// Clip after an epilogue that summed the norms (EpiOptStep: d the unclipped step,
// EpiStoreGroupF32: d the gradient): a cluster per layer adds the layer's
// (||W||^2, ||d||^2) slot pairs in a fixed order and writes the layer's scale
// min(1, clip_frac ||W|| / ||d||).
__global__ void __cluster_dims__(kSlotBlocks, 1, 1) __launch_bounds__(kSlotThreads)
    opt_scale_kernel(const float* part, int slots, const OptimParams op,
                     float* __restrict__ scales) {
    grid_dependency_wait();
    const int layer = blockIdx.x / kSlotBlocks;
    double t[2];
    if (!slot_sum<2>(part + static_cast<size_t>(layer) * slots * 2, slots, t)) return;
    const double lim = static_cast<double>(op.clip_frac) * sqrt(t[0]);
    scales[layer] = static_cast<float>(sqrt(t[1]) > lim ? lim / sqrt(t[1]) : 1.0);
}

// W <- W + s d with the layer's scale, and W_out = bf16(W) (16-byte vectors); d = D, or
// -lr s1 with the momentum just updated (the step opt_step took).
__global__ void __launch_bounds__(kOptThreads)
    opt_step_apply_kernel(const __grid_constant__ LayerPtrs lp, size_t n, const OptimParams op,
                          const float* __restrict__ scales) {
    const int layer = blockIdx.y;
    const float* S1 = lp.s1[layer];
    const float* D = S1 ? S1 : lp.G[layer];
    const float f = S1 ? -op.lr : 1.f;
    float* W = lp.W[layer];
    __nv_bfloat16* Wo = static_cast<__nv_bfloat16*>(lp.Wo[layer]);
    const float s = scales[layer];
    const size_t stride = static_cast<size_t>(gridDim.x) * kOptThreads;
    for (size_t i = blockIdx.x * static_cast<size_t>(kOptThreads) + threadIdx.x; i < n / 4;
         i += stride) {  // n = d d_ff, a multiple of 8
        Vec<4> d, w;
        d.load(D, i);
        w.load(W, i);
#pragma unroll
        for (int k = 0; k < 4; ++k) w.v[k] = fmaf(s, f * d.v[k], w.v[k]);
        w.store(W, i);
        if (Wo) w.store(Wo, i);
    }
}

// Blocks per layer of the element-wise passes: all of them resident at once, which a launch
// beside the end of a GEMM (launch_chained) would spoil: their blocks then crowd the SMs
// that are free first (apply pass 790 -> 1040 us).
int blocks_per_layer(int n_layers) {
    DevInfo di;
    const int sms = current_device_info(&di) ? di.sm_count : 148;
    int b = (sms * 8) / (n_layers > 0 ? n_layers : 1);
    if (b < 1) b = 1;
    return b < kOptBlocksPerLayerMax ? b : kOptBlocksPerLayerMax;
}

}  // namespace

size_t optim_partials_bytes(int n_layers) {
    return static_cast<size_t>(n_layers) * kOptBlocksPerLayerMax * 3 * sizeof(double);
}

namespace {

LayerPtrs layer_ptrs(int n_layers, float* const* G, float* const* W_master, void* const* W_out,
                     float* const* s1, float* const* s2) {
    LayerPtrs lp = {};
    for (int l = 0; l < n_layers; ++l) {
        lp.G[l] = G[l];
        lp.W[l] = W_master[l];
        lp.Wo[l] = W_out ? W_out[l] : nullptr;
        lp.s1[l] = s1 ? s1[l] : nullptr;
        lp.s2[l] = s2 ? s2[l] : nullptr;
    }
    return lp;
}

template <int kV>
cudaError_t run_optimizer(int dtype, int n_layers, size_t n, const OptimParams& op,
                          const LayerPtrs& lp, double* partials, float* scales, bool norms_done,
                          cudaStream_t st) {
    const int bpl = blocks_per_layer(n_layers);
    const dim3 grid(bpl, n_layers);
    if (op.clip != 0 && !norms_done) {
        optim_norms_kernel<kV><<<grid, kOptThreads, 0, st>>>(lp, n, op, partials),
            ::fpo::note_launch();
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        optim_scale_kernel<<<n_layers, kScaleThreads, 0, st>>>(partials, bpl, op, scales),
            ::fpo::note_launch();
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const float* sc = op.clip != 0 ? scales : nullptr;
    if (dtype == 1)
        optim_apply_kernel<true, kV><<<grid, kOptThreads, 0, st>>>(lp, n, op, sc),
            ::fpo::note_launch();
    else
        optim_apply_kernel<false, kV><<<grid, kOptThreads, 0, st>>>(lp, n, op, sc),
            ::fpo::note_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_optimizer(int dtype, int n_layers, size_t n_elem, const OptimParams& op,
                             float* const* G, float* const* W_master, void* const* W_out,
                             float* const* s1, float* const* s2, double* partials, float* scales,
                             bool norms_done, cudaStream_t st) {
    if (n_layers < 1 || n_layers > kMaxLayers) return cudaErrorInvalidValue;
    if (n_elem == 0) return cudaSuccess;
    const LayerPtrs lp = layer_ptrs(n_layers, G, W_master, W_out, s1, s2);
    // the layers' G follow each other in the workspace: aligned like the rest only then
    if (n_elem % 4 == 0)
        return run_optimizer<4>(dtype, n_layers, n_elem, op, lp, partials, scales, norms_done, st);
    return run_optimizer<1>(dtype, n_layers, n_elem, op, lp, partials, scales, norms_done, st);
}

cudaError_t launch_opt_scale(int n_layers, const OptimParams& op, const float* part, int slots,
                             float* scales, cudaStream_t st) {
    if (n_layers < 1 || n_layers > kMaxLayers) return cudaErrorInvalidValue;
    return launch_chained(opt_scale_kernel, dim3(kSlotBlocks * n_layers), kSlotThreads, 0, st, part, slots, op,
                          scales);
}

cudaError_t launch_opt_step_apply(int n_layers, size_t n_elem, const OptimParams& op,
                                  float* const* D, float* const* s1, float* const* W_master,
                                  void* const* W_out, const float* scales, cudaStream_t st) {
    if (n_layers < 1 || n_layers > kMaxLayers) return cudaErrorInvalidValue;
    if (n_elem == 0) return cudaSuccess;
    const LayerPtrs lp = layer_ptrs(n_layers, D, W_master, W_out, s1, nullptr);
    const dim3 grid(blocks_per_layer(n_layers), n_layers);
    opt_step_apply_kernel<<<grid, kOptThreads, 0, st>>>(lp, n_elem, op, scales),
        ::fpo::note_launch();
    return cudaGetLastError();
}

}  // namespace fpo
