// epilogues.cuh -- per-row epilogues of the tcgen05 GEMM.
//
// Each epilogue thread owns one output row of a 128 x BN tile and receives its
// fp32 accumulator 32 columns at a time: Epi(params, group, row, n0), then
// chunk(params, v[32], col_of_v0, col_offset_in_tile, io) for each 32-column
// chunk in order, then finish(params, n_block).  Rows >= M and columns >= N
// belong to the zero-filled tile overhang and are never written.  Dense
// outputs go through the warp's swizzled staging buffers and TMA stores
// (one 32-row x 128-byte box per store; the TMA engine clips the overhang).
//
// Epilogues that read or update matrices of the output's shape (the update, the
// optimizer's first pass, the cosine, the gate / up signals, plain G) have 8 warps
// (Epi::kWarps) and the form of epilogue_tile's second half: a chunk is staged in shared
// memory and each lane takes 4 columns of 8 of its rows, so that every global access of a
// warp covers 256 bytes of two rows, and the operands of the next chunk (of the first chunk:
// while the mainloop runs) are loaded ahead.  One row per
// thread, as these epilogues had it with 4 warps, made every 16-byte access of a warp
// touch 32 rows and kept 16 KB in flight per SM: AdamW with the step clip at T 4096,
// d 4096, d_ff 11008, 8 layers took 4154 us in the GEMM for 1.5 ms of tensor work.
#pragma once

#include <cuda_bf16.h>
#include <math.h>

#include "error_math.cuh"
#include "optim_math.cuh"
#include "ptx.cuh"
#include "tc_gemm.cuh"

namespace fpo {

// ---------------------------------------------------------------------------
// Logits pass (Sec. 3.1 step 2): per (row, vocabulary tile) the running max and
// sum of exponentials of z = yhat W_U^T over the tile's valid columns, plus the
// target logit z_{t, y_t} when the target falls inside the tile.  With kStoreZ
// the fp32 logits are also written to z [M, ldz] (stored-logits algorithm).
template <bool kStoreZ>
struct EpiLsePartialT {
    static constexpr int kWarps = 4;
    struct Params {
        CUtensorMap zmap;  // fp32 logits [M, N], box 32 x 32 (kStoreZ only)
        float2* part;      // [M, part_ld]: (max, sum exp(z - max)) per vocabulary tile
        int part_ld;
        float* zy;         // [M] target logit, or null
        const int* y;      // [M] targets
        int M, N;
    };
    float m, s, zt;
    int yoff;
    int row;
    bool valid, has_t;

    __device__ __forceinline__ EpiLsePartialT(const Params& p, int, int row_, int n0)
        : m(-INFINITY), s(0.f), zt(0.f), row(row_), has_t(false) {
        valid = row_ < p.M;
        yoff = valid ? __ldg(p.y + row_) - n0 : -1;
    }

    __device__ __forceinline__ void chunk(const Params& p, const float (&v)[32], int col0, int c0,
                                          EpiIO& io) {
        const int lim = p.N - col0;  // valid columns in this chunk (may be <= 0)
        if (lim <= 0) return;
        if constexpr (kStoreZ) {
            if (io.row0 < p.M) {
                const uint32_t buf = out_acquire(io);
                uint32_t w[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) w[j] = __float_as_uint(v[j]);
                out_stage_row(buf, io.lane, w);
                out_commit(io, &p.zmap, buf, col0, io.row0);
            }
        }
        float cm = -INFINITY;
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < lim) cm = fmaxf(cm, v[j]);
        const float nm = fmaxf(m, cm);
        const float nml = nm * kLog2e;
        float acc = (m == -INFINITY) ? 0.f : s * ex2_approx(m * kLog2e - nml);
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < lim) acc += ex2_approx(fmaf(v[j], kLog2e, -nml));
        s = acc;
        m = nm;
        const int r = yoff - c0;
        if (static_cast<unsigned>(r) < 32u) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (j == r) zt = v[j];
            has_t = true;
        }
    }

    __device__ __forceinline__ void finish(const Params& p, int nb) {
        if (!valid) return;
        p.part[static_cast<long long>(row) * p.part_ld + nb] = make_float2(m, s);
        if (has_t && p.zy) p.zy[row] = zt;
    }
};
using EpiLsePartial = EpiLsePartialT<false>;
using EpiLseStoreZ = EpiLsePartialT<true>;

// ---------------------------------------------------------------------------
// Logits pass of the direct algorithm (Sec. 3.1 step 2 rewritten around a
// per-token anchor c_t, the target logit): every valid non-target logit leaves
//   p~_tj = exp(z_tj - c_t)
// rounded to bf16 into P [M, N] (the target column and the overhang are written
// as 0), and per (row, 256-column tile) three sums:
//   su = sum_j p~_tj          (unrounded: lse_t = c_t + log(1 + S_t), the target's
//                              own term being exp(0) = 1)
//   sx = sum_j p^_tj          (p^ the rounded values: the tile's part of S'_t, which
//                              makes the target entry of e the exact negative sum)
//   qz = sum_j p^_tj z_tj     (for the final-norm VJP fused into the projection:
//                              <yhat_t, g_t> = sum_v e_tv z_tv = alpha_t (Qz_t - c_t S'_t))
// No running maximum is kept: a row whose S'_t leaves the window [2^-80, 2^80]
// (where the anchored sums could overflow, or hold no significant digit) is
// recomputed by the fixup path, which takes its lse from a max-based pass
// (EpiFixLse, then EpiFixProb).
// Chunks that hold neither a target nor the vocabulary's ragged end (all but a few
// per row) take a branch-free path on packed f32x2 arithmetic; two 32-column chunks
// fill one 64-column bf16 staging row before each TMA store.
struct EpiAnchorProb {
    static constexpr int kWarps = 4;
    struct Params {
        CUtensorMap pmap;     // bf16 P [M, N], box 64 x 32
        float* su;            // [M, part_ld] sum of p~ over the tile
        float* sx;            // [M, part_ld] sum of the rounded p~ of the tile
        float* qz;            // [M, part_ld] sum of the rounded p~ times z over the tile
        int part_ld;
        const int* y;         // [M] targets
        const float* anchor;  // [M] c_t
        int M, N;
    };
    float2 u0, u1, s0, s1, q0, q1;  // two accumulators each: shorter dependency chains
    float2 nc2;             // (-c_t log2 e) twice
    int yoff, row;
    bool valid, pair_out;
    uint32_t w[32];

    __device__ __forceinline__ EpiAnchorProb(const Params& p, int, int row_, int n0)
        : row(row_), pair_out(false) {
        valid = row_ < p.M;
        yoff = valid ? __ldg(p.y + row_) - n0 : -1;
        const float nc = valid ? -p.anchor[row_] * kLog2e : 0.f;
        nc2 = make_float2(nc, nc);
        u0 = u1 = s0 = s1 = q0 = q1 = make_float2(0.f, 0.f);
    }

    // p^ of the pair (j, j + 1) and its contribution to the sums; kMask: zero the
    // target (position r) and the columns >= lim.
    template <bool kMask>
    __device__ __forceinline__ uint32_t pair(const float (&v)[32], int j, int r, int lim) {
        const float2 z = make_float2(v[j], v[j + 1]);
        const float2 arg = __ffma2_rn(z, make_float2(kLog2e, kLog2e), nc2);
        float pa = ex2_approx(arg.x), pb = ex2_approx(arg.y);
        if constexpr (kMask) {
            pa = (j < lim && j != r) ? pa : 0.f;
            pb = (j + 1 < lim && j + 1 != r) ? pb : 0.f;
        }
        const uint32_t pk = pack_bf16x2(pa, pb);
        const float2 rp = make_float2(__uint_as_float(pk << 16), __uint_as_float(pk & 0xffff0000u));
        if ((j / 2) & 1) {
            u1 = __fadd2_rn(u1, make_float2(pa, pb));
            s1 = __fadd2_rn(s1, rp);
            q1 = __ffma2_rn(rp, z, q1);
        } else {
            u0 = __fadd2_rn(u0, make_float2(pa, pb));
            s0 = __fadd2_rn(s0, rp);
            q0 = __ffma2_rn(rp, z, q0);
        }
        return pk;
    }

    __device__ __forceinline__ void chunk(const Params& p, const float (&v)[32], int col0, int c0,
                                          EpiIO& io) {
        const bool second = (c0 & 32) != 0;
        if (!second) pair_out = col0 >= p.N || io.row0 >= p.M;
        const int lim = p.N - col0;  // valid columns in this chunk (may be <= 0)
        const int r = yoff - c0;     // target position in this chunk, if in [0, 32)
        uint32_t pk[16];
        // warp-uniform: a chunk holding any lane's target, or the ragged end, is masked
        if (lim < 32 || __any_sync(0xffffffffu, static_cast<unsigned>(r) < 32u)) {
#pragma unroll
            for (int j = 0; j < 32; j += 2) pk[j / 2] = pair<true>(v, j, r, lim);
        } else {
#pragma unroll
            for (int j = 0; j < 32; j += 2) pk[j / 2] = pair<false>(v, j, r, lim);
        }
        if (pair_out) return;
        if (!second) {
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = pk[i];
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) w[16 + i] = pk[i];
            const uint32_t buf = out_acquire(io);
            out_stage_row(buf, io.lane, w);
            out_commit(io, &p.pmap, buf, col0 - 32, io.row0);
        }
    }

    __device__ __forceinline__ void finish(const Params& p, int nb) {
        if (!valid) return;
        const long long o = static_cast<long long>(row) * p.part_ld + nb;
        const float2 u = __fadd2_rn(u0, u1), s = __fadd2_rn(s0, s1), q = __fadd2_rn(q0, q1);
        p.su[o] = u.x + u.y;
        p.sx[o] = s.x + s.y;
        p.qz[o] = q.x + q.y;
    }
};

// ---------------------------------------------------------------------------
// Direct algorithm, rows outside the anchor window, first pass: the logits of the
// gathered rows (the GEMM's rows are fix[0, count)) reduced to a running max and
// sum of exponentials per (row, 256-column tile), written to part[row of the chunk,
// tile], from which lse is formed before the second pass (EpiFixProb).
struct EpiFixLse {
    static constexpr int kWarps = 4;
    struct Params {
        float2* part;        // [T, part_ld] (max, sum exp(z - max))
        int part_ld;
        const int* fix;      // gathered row -> row of the chunk
        const int* count;    // gathered rows (device)
        int N;
    };
    float m, s;
    int orig;
    bool valid;

    __device__ __forceinline__ EpiFixLse(const Params& p, int, int row_, int)
        : m(-INFINITY), s(0.f) {
        valid = row_ < *p.count;
        orig = valid ? p.fix[row_] : 0;
    }

    __device__ __forceinline__ void chunk(const Params& p, const float (&v)[32], int col0, int,
                                          EpiIO&) {
        const int lim = p.N - col0;
        if (!valid || lim <= 0) return;
        float cm = -INFINITY;
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < lim) cm = fmaxf(cm, v[j]);
        const float nm = fmaxf(m, cm);
        const float nml = nm * kLog2e;
        float acc = (m == -INFINITY) ? 0.f : s * ex2_approx(m * kLog2e - nml);
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < lim) acc += ex2_approx(fmaf(v[j], kLog2e, -nml));
        s = acc;
        m = nm;
    }

    __device__ __forceinline__ void finish(const Params& p, int nb) {
        if (valid) p.part[static_cast<size_t>(orig) * p.part_ld + nb] = make_float2(m, s);
    }
};

// ---------------------------------------------------------------------------
// Direct algorithm, rows outside the anchor window, second pass (Sec. 3.1 step 2
// with the anchor at lse_t): the GEMM's rows are the yhat rows gathered from
// fix[0, count); each logit z of such a row becomes p~ = exp(z - lse_t), 0 at the
// target, rounded to bf16 and stored into that row of P with plain 16-byte stores;
// the row's sums over the tile of the rounded values and of the rounded values
// times z go to sx[row, tile] and qz[row, tile], as EpiAnchorProb leaves them.
struct EpiFixProb {
    static constexpr int kWarps = 4;
    struct Params {
        __nv_bfloat16* P;    // [T, N] rows of the chunk, row stride N
        float* sx;           // [T, n_tiles]
        float* qz;           // [T, n_tiles]
        const int* fix;      // gathered row -> row of the chunk
        const int* count;    // gathered rows (device)
        const int32_t* y;    // [T] targets
        const float* lse;    // [T]
        int n_tiles, N;
    };
    int orig, yt;
    float lse2, sxs, qs;
    bool valid;

    __device__ __forceinline__ EpiFixProb(const Params& p, int, int row_, int)
        : sxs(0.f), qs(0.f) {
        valid = row_ < *p.count;
        orig = valid ? p.fix[row_] : 0;
        yt = valid ? p.y[orig] : -1;
        lse2 = valid ? p.lse[orig] * kLog2e : 0.f;
    }

    __device__ __forceinline__ void chunk(const Params& p, const float (&v)[32], int col0, int,
                                          EpiIO&) {
        const int lim = p.N - col0;  // valid columns of the chunk
        if (!valid || lim <= 0) return;
        const int r = yt - col0;
        uint32_t w[16];
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
            const float a = (j < lim && j != r) ? ex2_approx(fmaf(v[j], kLog2e, -lse2)) : 0.f;
            const float b =
                (j + 1 < lim && j + 1 != r) ? ex2_approx(fmaf(v[j + 1], kLog2e, -lse2)) : 0.f;
            const uint32_t pk = pack_bf16x2(a, b);
            const float ra = __uint_as_float(pk << 16), rb = __uint_as_float(pk & 0xffff0000u);
            sxs += ra + rb;
            qs = fmaf(ra, v[j], qs);
            qs = fmaf(rb, v[j + 1], qs);
            w[j / 2] = pk;
        }
        uint4* dst = reinterpret_cast<uint4*>(p.P + static_cast<size_t>(orig) * p.N + col0);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q * 8 < lim) dst[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
    }

    __device__ __forceinline__ void finish(const Params& p, int nb) {
        if (valid) {
            p.sx[static_cast<size_t>(orig) * p.n_tiles + nb] = sxs;
            p.qz[static_cast<size_t>(orig) * p.n_tiles + nb] = qs;
        }
    }
};

// ---------------------------------------------------------------------------
// Recompute pass (Sec. 3.1 step 2): e = s (exp(z - lse) - [col == y]) rounded
// to bf16 into the error matrix E [M, N]; two 32-column chunks fill one
// 64-column bf16 staging row before each TMA store.
struct EpiError {
    static constexpr int kWarps = 4;
    struct Params {
        CUtensorMap Emap;  // bf16 E [M, N], box 64 x 32
        const float* lse;  // [M]
        const int* y;      // [M]
        int M, N;
        float s;
    };
    int row, yt;
    float lse2;
    bool pair_out;  // the current 64-column pair lies beyond N
    uint32_t w[32];

    __device__ __forceinline__ EpiError(const Params& p, int, int row_, int) : row(row_) {
        const bool valid = row_ < p.M;
        yt = valid ? __ldg(p.y + row_) : -1;
        lse2 = valid ? p.lse[row_] * kLog2e : 0.f;
        pair_out = false;
    }

    __device__ __forceinline__ void chunk(const Params& p, const float (&v)[32], int col0, int c0,
                                          EpiIO& io) {
        const bool second = (c0 & 32) != 0;
        if (!second) pair_out = col0 >= p.N || io.row0 >= p.M;
        if (pair_out) return;
        if (!second) {
#pragma unroll
            for (int j = 0; j < 32; j += 2)
                w[j / 2] = pack_bf16x2(error_value(v[j], lse2, col0 + j == yt, p.s),
                                       error_value(v[j + 1], lse2, col0 + j + 1 == yt, p.s));
        } else {
#pragma unroll
            for (int j = 0; j < 32; j += 2)
                w[16 + j / 2] = pack_bf16x2(error_value(v[j], lse2, col0 + j == yt, p.s),
                                            error_value(v[j + 1], lse2, col0 + j + 1 == yt, p.s));
            const uint32_t buf = out_acquire(io);
            out_stage_row(buf, io.lane, w);
            out_commit(io, &p.Emap, buf, col0 - 32, io.row0);
        }
    }

    __device__ __forceinline__ void finish(const Params&, int) {}
};

// ---------------------------------------------------------------------------
// Plain fp32 store of C [M, N]: the projection g = E W_U (Eq. gproj).
struct EpiStoreF32 {
    static constexpr int kWarps = 4;
    struct Params {
        CUtensorMap Cmap;  // fp32 C [M, N], box 32 x 32
        int M, N;
    };

    __device__ __forceinline__ EpiStoreF32(const Params&, int, int, int) {}

    __device__ __forceinline__ void chunk(const Params& p, const float (&v)[32], int col0, int,
                                          EpiIO& io) {
        if (col0 >= p.N || io.row0 >= p.M) return;
        const uint32_t buf = out_acquire(io);
        uint32_t w[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) w[j] = __float_as_uint(v[j]);
        out_stage_row(buf, io.lane, w);
        out_commit(io, &p.Cmap, buf, col0, io.row0);
    }

    __device__ __forceinline__ void finish(const Params&, int) {}
};

// ---------------------------------------------------------------------------
// Every tile split over K: the pair kernel stores the parts itself and no tile is whole.
struct EpiParts {
    static constexpr int kWarps = 4;
    struct Params {};
    __device__ __forceinline__ EpiParts(const Params&, int, int, int) {}
    __device__ __forceinline__ void chunk(const Params&, const float (&)[32], int, int, EpiIO&) {}
    __device__ __forceinline__ void finish(const Params&, int) {}
};

// ---------------------------------------------------------------------------
// Projection of the direct algorithm with the final-norm VJP (App. E,
// Eq. rmsnorm-vjp) fused in.  With acc = P W_U (target column of P zero), the
// unnormalised error signal of token t is
//   g_t = alpha_t acc_t + beta_t W_U[y_t],   alpha_t = s exp(c_t - lse_t),
//   beta_t = -alpha_t S'_t,
// which is s (softmax(z_t) - 1_{y_t}) W_U written with the anchor c_t, and the
// epilogue writes, in bf16,
//   g~_t = (w (.) g_t - x^_t k_t) / max(rho_t, rho_min),   x^_t = h_t / rho_t,
// where k_t = <x^_t, w (.) g_t> / d arrives as cv_t / d: cv_t = alpha_t (Qz_t - c_t S'_t)
// from the logits pass (EpiAnchorProb), the same inner product taken through the
// logits (<yhat_t, W_U[v]> = z_tv), so no tile needs the whole row of g.
// A row with alpha_t == 0 is written as zeros (s == 0, or an out-of-range
// target); beta_t == 0 skips the read of the target's W_U row.  The h, w and
// W_U[y] values of the next 32-column chunk are loaded while the current one is
// processed; two chunks fill one 64-column bf16 staging row per TMA store.
struct EpiProjVjp {
    static constexpr int kWarps = 4;
    struct Params {
        CUtensorMap omap;           // bf16 g~ [M, N], box 64 x 32
        const float* alpha;         // [M]
        const float* beta;          // [M]
        const float* cv;            // [M] <yhat_t, g_t>
        const float* rho;           // [M] RMS of h_t (forward pass)
        const int* y;               // [M]
        const __nv_bfloat16* W_U;   // [V, N]
        const __nv_bfloat16* h;     // [M, N] pre-norm residual
        const __nv_bfloat16* w;     // [N] final RMSNorm weight
        float min_rms, inv_d;
        int M, N;
        int tile_n;                 // columns of the kernel's tiles (one epilogue object each)
    };
    float a;
    float2 a2, b2, nk2;  // per row, twice: alpha pref, beta pref, -(cv / d) pref / rho
    const __nv_bfloat16* wy;
    const __nv_bfloat16* hr;
    bool valid, pair_out;
    int n_end;
    uint4 uh[4], uw[4], uy[4];  // h, w, W_U[y] of the chunk the next chunk() call uses
    uint32_t o[32];

    __device__ __forceinline__ void fetch(const Params& p, int col0) {
        const int lim = p.N - col0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool in = q * 8 < lim;
            uh[q] = (valid && in) ? __ldg(reinterpret_cast<const uint4*>(hr + col0) + q)
                                  : make_uint4(0, 0, 0, 0);
            uw[q] = in ? __ldg(reinterpret_cast<const uint4*>(p.w + col0) + q)
                       : make_uint4(0, 0, 0, 0);
            uy[q] = (wy && in) ? __ldg(reinterpret_cast<const uint4*>(wy + col0) + q)
                               : make_uint4(0, 0, 0, 0);
        }
    }

    __device__ __forceinline__ EpiProjVjp(const Params& p, int, int row, int n0)
        : pair_out(false) {
        valid = row < p.M;
        a = valid ? p.alpha[row] : 0.f;
        const float b = valid ? p.beta[row] : 0.f;
        const float r = valid ? p.rho[row] : 1.f;
        const float kd = valid ? p.cv[row] * p.inv_d : 0.f;
        const float pref = 1.0f / fmaxf(r, p.min_rms);
        // g~_j = w_j (a pref acc_j + b pref W_U[y]_j) - h_j (kd pref / rho)
        a2 = make_float2(a * pref, a * pref);
        b2 = make_float2(b * pref, b * pref);
        const float nk = -(kd * (1.0f / r)) * pref;
        nk2 = make_float2(nk, nk);
        wy = (a != 0.f && b != 0.f) ? p.W_U + static_cast<long long>(__ldg(p.y + row)) * p.N
                                    : nullptr;
        hr = p.h + static_cast<long long>(valid ? row : 0) * p.N;
        n_end = min(n0 + p.tile_n, p.N);
        if (n0 < p.N) fetch(p, n0);
    }

    __device__ __forceinline__ void chunk(const Params& p, const float (&v)[32], int col0, int c0,
                                          EpiIO& io) {
        const bool second = (c0 & 32) != 0;
        uint4 ch[4], cw[4], cy[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            ch[q] = uh[q];
            cw[q] = uw[q];
            cy[q] = uy[q];
        }
        if (col0 + 32 < n_end) fetch(p, col0 + 32);
        if (!second) pair_out = col0 >= p.N || io.row0 >= p.M;
        if (pair_out) return;
        uint32_t r[16];
        if (a == 0.f) {  // s == 0 or an out-of-range target: g = 0 and cv = 0, so g~ = 0
#pragma unroll
            for (int i = 0; i < 16; ++i) r[i] = 0u;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t hh[4] = {ch[q].x, ch[q].y, ch[q].z, ch[q].w};
                const uint32_t ww[4] = {cw[q].x, cw[q].y, cw[q].z, cw[q].w};
                const uint32_t yy[4] = {cy[q].x, cy[q].y, cy[q].z, cy[q].w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int j = 8 * q + 2 * k;
                    const float2 hv = make_float2(__uint_as_float(hh[k] << 16),
                                                  __uint_as_float(hh[k] & 0xffff0000u));
                    const float2 wv = make_float2(__uint_as_float(ww[k] << 16),
                                                  __uint_as_float(ww[k] & 0xffff0000u));
                    const float2 uv = make_float2(__uint_as_float(yy[k] << 16),
                                                  __uint_as_float(yy[k] & 0xffff0000u));
                    const float2 t = __ffma2_rn(b2, uv, __fmul2_rn(a2, make_float2(v[j], v[j + 1])));
                    const float2 out = __ffma2_rn(wv, t, __fmul2_rn(nk2, hv));
                    r[j / 2] = pack_bf16x2(out.x, out.y);
                }
            }
        }
        if (!second) {
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = r[i];
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) o[16 + i] = r[i];
            const uint32_t buf = out_acquire(io);
            out_stage_row(buf, io.lane, o);
            out_commit(io, &p.omap, buf, col0 - 32, io.row0);
        }
    }

    __device__ __forceinline__ void finish(const Params&, int) {}
};

// A lane's place in a warp's 32 rows x 64 kCG columns (kCG = 2 or 1 groups of chunk columns,
// of tiles of 256 or 128) of an 8-warp epilogue: the 4 columns of access i of chunk c (numbered
// j = kAcc c + i over the whole block), as element offsets into matrices of row stride ld.
template <int kCG>
struct RowPos {
    using R = RowChunk;
    static constexpr int kChunks = 32 / R::kRows * kCG;
    long long off;    // of the lane's columns in its first row
    int rows, cols;   // rows from the lane's first, columns from its first, inside

    __device__ __forceinline__ RowPos(int M, int N, long long ld, int row0, int n0, int lane) {
        const int r = row0 + lane / R::kLanes, c = n0 + 4 * (lane % R::kLanes);
        off = r * ld + c;
        rows = M - r;
        cols = N - c;
    }
    static __device__ __forceinline__ int row(int j) {
        return j / R::kAcc / kCG * R::kRows + j % R::kAcc * R::kAccRows;
    }
    static __device__ __forceinline__ int col(int j) { return j / R::kAcc % kCG * R::kCols; }
    // Access j is inside the matrix (N is a multiple of 8, so its 4 columns are inside
    // together).
    __device__ __forceinline__ bool in(int j) const { return row(j) < rows && col(j) < cols; }
    __device__ __forceinline__ long long at(long long ld, int j) const {
        return off + row(j) * ld + col(j);
    }
    // That element of a matrix m, or m itself outside the matrix: always readable, so that
    // a batch of loads has no branches between them.
    template <typename TT>
    __device__ __forceinline__ const TT* src(const TT* m, long long ld, int j) const {
        return in(j) ? m + at(ld, j) : m;
    }
};

// Slots of per-warp partial sums per (256-row block, 256 columns): 8 blocks of 32 rows times
// 4 column quarters.  A warp with two column groups keeps their sums apart, so that tiles of
// 128 columns leave the same slots.
constexpr int kColSlots = 32;

template <int N>
__device__ __forceinline__ float* slot_of(float* part, int g, int m256, int n256, int row0, int n0) {
    return part + (((static_cast<long long>(g) * m256 + row0 / 256) * n256 + n0 / 256) * kColSlots +
                   (n0 % 256) / 64 * 8 + (row0 % 256) / 32) * N;
}

// N sums per column group, added chunk by chunk.
template <int N, int kCG>
struct GroupSums {
    float v[kCG][N];
    __device__ __forceinline__ GroupSums() {
#pragma unroll
        for (int k = 0; k < N; ++k) v[0][k] = v[kCG - 1][k] = 0.f;
    }
    __device__ __forceinline__ void add(int chunk, const float (&x)[N]) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            if (chunk % kCG == 0)
                v[0][k] += x[k];
            else
                v[kCG - 1][k] += x[k];
        }
    }
    // The warp's totals (a fixed butterfly) to the slots of its one or two groups.
    __device__ __forceinline__ void store(float* slot, int lane) const;
};

__device__ __forceinline__ float warp_sum_f32(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

template <int N, int kCG>
__device__ __forceinline__ void GroupSums<N, kCG>::store(float* slot, int lane) const {
#pragma unroll
    for (int c = 0; c < kCG; ++c) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const float t = warp_sum_f32(v[c][k]);
            if (lane == 0) slot[8 * c * N + k] = t;
        }
    }
}

// ---------------------------------------------------------------------------
// Pseudogradient update (Eq. w3update, App. A): for group (layer) g,
//   W_master[g] -= lr * G ;  W_out[g] = bf16(W_master[g]) ;  G_out[g] = bf16(G)
// Any of the three pointers may be null for a layer.
//
// The operands of a chunk (here, in the cosine, plain G and gate / up) are loaded as one
// batch when the chunk before is done, with nothing that waits between its loads: loads
// issued one by one between the uses of the batch before shared the warp's few scoreboards
// with it, and each use waited for the newest load (the update of T 512, d 2048, d_ff 8264, 4
// layers: 278 us, 230 of them with the loads alone, 115 without; 195 us with batches, and 176
// with 256 bytes of two rows per access (kRows 16) instead of 128 bytes of four (kRows 32).
// 512 bytes of one row (kRows 8) gave 162 but cost 2% of a T 200 step, as every lane reads the
// accumulator once per row group.  Two batches in flight gave nothing more, nor did 16 warps,
// L2 prefetches of the next tile or streaming cache hints).
struct EpiUpdateBase {
    struct Params {
        float* W_master[kMaxGroups];
        __nv_bfloat16* W_out[kMaxGroups];
        __nv_bfloat16* G_out[kMaxGroups];
        long long ld;
        int M, N;
        float neg_lr;
    };
};

template <int kCG>
struct EpiUpdate : EpiUpdateBase {
    static constexpr int kWarps = 8, kColGroups = kCG;
    using R = RowChunk;
    RowPos<kCG> pos;
    float* wm;
    __nv_bfloat16* wo;
    __nv_bfloat16* go;
    float4 w[R::kAcc];  // master values of the next chunk

    __device__ __forceinline__ void load(const Params& p, int c) {
        if (!wm) return;
#pragma unroll
        for (int i = 0; i < R::kAcc; ++i)
            w[i] = *reinterpret_cast<const float4*>(pos.src(wm, p.ld, R::kAcc * c + i));
    }

    __device__ __forceinline__ EpiUpdate(const Params& p, int g, int row0, int n0, int lane)
        : pos(p.M, p.N, p.ld, row0, n0, lane) {
        wm = p.W_master[g];
        wo = p.W_out[g];
        go = p.G_out[g];
        load(p, 0);
    }

    __device__ __forceinline__ void chunk(const Params& p, uint32_t buf, int lane, int c) {
#pragma unroll
        for (int i = 0; i < R::kAcc; ++i) {
            const float4 v = R::read(buf, lane, i);
            const long long o = pos.at(p.ld, R::kAcc * c + i);
            const bool in = pos.in(R::kAcc * c + i);
            if (wm) {
                float4 a = w[i];
                a.x = fmaf(p.neg_lr, v.x, a.x);
                a.y = fmaf(p.neg_lr, v.y, a.y);
                a.z = fmaf(p.neg_lr, v.z, a.z);
                a.w = fmaf(p.neg_lr, v.w, a.w);
                if (in) {
                    *reinterpret_cast<float4*>(wm + o) = a;
                    if (wo)
                        *reinterpret_cast<uint2*>(wo + o) =
                            make_uint2(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w));
                }
            }
            if (go && in)
                *reinterpret_cast<uint2*>(go + o) =
                    make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
        }
        if (c + 1 < pos.kChunks) load(p, c + 1);
    }

    __device__ __forceinline__ void finish(const Params&, int) {}
};

// ---------------------------------------------------------------------------
// Pseudogradients with the layer-viability diagnostic's cosine (Sec. 2.2 Eq. (cosine),
// Eq. (w3update)): for group (layer) g, G_out[g] = bf16(G), and the three sums of the
// cosine of that stored G against Y[g] (<G, Y>, ||G||^2, ||Y||^2) over the warp's
// block (fp32 per lane, then a fixed butterfly), one triple per slot (slot_of), so the
// cosine needs no second pass over G.
struct EpiGradCosBase {
    struct Params {
        __nv_bfloat16* G_out[kMaxGroups];
        const __nv_bfloat16* Y[kMaxGroups];
        float* part;     // [groups][m256][n_blocks][kColSlots][3]
        long long ld;
        int M, N;
        int m256, n_blocks;
    };
};

template <int kCG>
struct EpiGradCos : EpiGradCosBase {
    static constexpr int kWarps = 8, kColGroups = kCG;
    using R = RowChunk;
    RowPos<kCG> pos;
    int g, row0, n0;
    GroupSums<3, kCG> sums;  // <G, Y>, ||G||^2, ||Y||^2
    uint2 y[R::kAcc];  // Y of the next chunk

    __device__ __forceinline__ void load(const Params& p, int c) {
#pragma unroll
        for (int i = 0; i < R::kAcc; ++i)
            y[i] = __ldg(reinterpret_cast<const uint2*>(pos.src(p.Y[g], p.ld, R::kAcc * c + i)));
    }

    __device__ __forceinline__ EpiGradCos(const Params& p, int g_, int row0_, int n0_, int lane)
        : pos(p.M, p.N, p.ld, row0_, n0_, lane), g(g_), row0(row0_), n0(n0_) {
        load(p, 0);
    }

    __device__ __forceinline__ void chunk(const Params& p, uint32_t buf, int lane, int c) {
        float2 s_gy = make_float2(0.f, 0.f), s_gg = s_gy, s_yy = s_gy;
#pragma unroll
        for (int i = 0; i < R::kAcc; ++i) {
            const float4 v = R::read(buf, lane, i);
            const uint32_t pk[2] = {pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w)};
            if (!pos.in(R::kAcc * c + i)) continue;
            const uint2 yv = y[i];
            const uint32_t yk[2] = {yv.x, yv.y};
            *reinterpret_cast<uint2*>(p.G_out[g] + pos.at(p.ld, R::kAcc * c + i)) =
                make_uint2(pk[0], pk[1]);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float2 gr = make_float2(__uint_as_float(pk[k] << 16),
                                              __uint_as_float(pk[k] & 0xffff0000u));
                const float2 yr = make_float2(__uint_as_float(yk[k] << 16),
                                              __uint_as_float(yk[k] & 0xffff0000u));
                s_gy = __ffma2_rn(gr, yr, s_gy);
                s_gg = __ffma2_rn(gr, gr, s_gg);
                s_yy = __ffma2_rn(yr, yr, s_yy);
            }
        }
        if (c + 1 < pos.kChunks) load(p, c + 1);
        sums.add(c, {s_gy.x + s_gy.y, s_gg.x + s_gg.y, s_yy.x + s_yy.y});
    }

    __device__ __forceinline__ void finish(const Params& p, int lane) {
        sums.store(slot_of<3>(p.part, g, p.m256, p.n_blocks, row0, n0), lane);
    }
};

// ---------------------------------------------------------------------------
// Pseudogradient only, fp32, one output per group (layer): G[g] = g~^T A_l, for
// the optimizers that need the whole G before they step.  With W_master set (the relative
// clip on the gradient) also ||W||^2 and ||G||^2 of the warp's block, one
// pair per slot_of, so that the clip factor needs no pass over W and G of its own
// (448 us of 1823 for 3 layers of 3072 x 23040).
struct EpiStoreGroupF32Base {
    struct Params {
        float* G[kMaxGroups];
        const float* W_master[kMaxGroups];  // or null: no norms
        float* part;                        // [groups][m256][n_blocks][kColSlots][2]
        long long ld;
        int M, N;
        int m256, n_blocks;
    };
};

template <int kCG>
struct EpiStoreGroupF32 : EpiStoreGroupF32Base {
    static constexpr int kWarps = 8, kColGroups = kCG;
    using R = RowChunk;
    RowPos<kCG> pos;
    int g, row0, n0;
    float* G;
    const float* wm;
    GroupSums<2, kCG> sums;  // ||W||^2, ||G||^2
    float4 w[R::kAcc];  // master values of the next chunk

    __device__ __forceinline__ void load(const Params& p, int c) {
        if (!wm) return;
#pragma unroll
        for (int i = 0; i < R::kAcc; ++i)
            w[i] = *reinterpret_cast<const float4*>(pos.src(wm, p.ld, R::kAcc * c + i));
    }

    __device__ __forceinline__ EpiStoreGroupF32(const Params& p, int g_, int row0_, int n0_,
                                                int lane)
        : pos(p.M, p.N, p.ld, row0_, n0_, lane), g(g_), row0(row0_), n0(n0_), G(p.G[g_]),
          wm(p.W_master[g_]) {
        load(p, 0);
    }

    __device__ __forceinline__ void chunk(const Params& p, uint32_t buf, int lane, int c) {
        float s_ww = 0.f, s_gg = 0.f;
#pragma unroll
        for (int i = 0; i < R::kAcc; ++i) {
            const float4 v = R::read(buf, lane, i);
            if (!pos.in(R::kAcc * c + i)) continue;
            *reinterpret_cast<float4*>(G + pos.at(p.ld, R::kAcc * c + i)) = v;
            if (wm) {
                s_gg = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, s_gg))));
                s_ww = fmaf(w[i].x, w[i].x,
                            fmaf(w[i].y, w[i].y, fmaf(w[i].z, w[i].z, fmaf(w[i].w, w[i].w, s_ww))));
            }
        }
        if (c + 1 < pos.kChunks) load(p, c + 1);
        sums.add(c, {s_ww, s_gg});
    }

    __device__ __forceinline__ void finish(const Params& p, int lane) {
        if (wm) sums.store(slot_of<2>(p.part, g, p.m256, p.n_blocks, row0, n0), lane);
    }
};

// ---------------------------------------------------------------------------
// The optimizer's first pass in the pseudogradient GEMM's epilogue, for the relative
// clip on the step (Sec. 3.1: SGD, SGD with momentum, AdamW on the fp32 masters; App. A:
// ||dW|| <= clip_frac ||W||).  With G from the accumulator, each element's optimizer state
// advances and its unclipped step d = opt_step(G, W, s1, s2) is stored (fp32, D[g], null
// for momentum, whose step -lr s1 the state holds; the state sees the unclipped gradient),
// and ||W||^2, ||d||^2 are written as one pair per slot of 32 rows x 64 columns; a kernel
// then scales each layer's steps by min(1, clip_frac ||W|| / ||d||) and applies them (W is
// not written here, so its norm is the pre-step one).  Without a clip the stand-alone passes
// are used: taking the whole step here made the update faster but the power-capped step
// slower (its epilogue then held the tensor pipe back at full draw).
// The operands of the access 4 ahead are loaded as each one is done: its arithmetic hides the
// wait that the batches of the other epilogues avoid (T 4096, d 4096, d_ff 11008, 8 layers,
// AdamW, with 4 rows x 128 bytes per access: 2362 us; batches of a whole or half a chunk
// 3006 and 2500, 2 ahead 2561, 8 ahead 2840, 16 warps 2990).
struct EpiOptStepBase {
    struct Params {
        const float* W_master[kMaxGroups];
        float* s1[kMaxGroups];             // momentum / AdamW first moment (or null)
        float* s2[kMaxGroups];             // AdamW second moment (or null)
        float* D[kMaxGroups];              // the unclipped steps (not for momentum: -lr s1)
        float* part;                       // [groups][m256][n_blocks][kColSlots][2]
        OptimParams op;
        long long ld;
        int M, N;
        int m256, n_blocks;
    };
};

template <int kCG>
struct EpiOptStep : EpiOptStepBase {
    static constexpr int kWarps = 8, kColGroups = kCG;
    using R = RowChunk;
    static constexpr int kAhead = 4;
    RowPos<kCG> pos;
    int g, row0, n0;
    const float* wm;
    float* p1;
    float* p2;
    float* D;
    GroupSums<2, kCG> sums;  // ||W||^2, ||d||^2
    float4 w[kAhead], a[kAhead], b[kAhead];  // of the next kAhead accesses

    __device__ __forceinline__ void load(const Params& p, int k, int j) {
        w[k] = a[k] = b[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!pos.in(j)) return;
        const long long o = pos.at(p.ld, j);
        w[k] = *reinterpret_cast<const float4*>(wm + o);
        if (p1) a[k] = *reinterpret_cast<const float4*>(p1 + o);
        if (p2) b[k] = *reinterpret_cast<const float4*>(p2 + o);
    }

    __device__ __forceinline__ EpiOptStep(const Params& p, int g_, int row0_, int n0_, int lane)
        : pos(p.M, p.N, p.ld, row0_, n0_, lane), g(g_), row0(row0_), n0(n0_) {
        wm = p.W_master[g_];
        p1 = p.s1[g_];
        p2 = p.s2[g_];
        D = p.D[g_];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) load(p, k, k);
    }

    __device__ __forceinline__ void chunk(const Params& p, uint32_t buf, int lane, int c) {
        float s_ww = 0.f, s_dd = 0.f;
#pragma unroll 1
        for (int h = 0; h < R::kAcc; h += kAhead) {
#pragma unroll
            for (int k = 0; k < kAhead; ++k) {
                const int i = h + k;
                const float4 v4 = R::read(buf, lane, i);
                const float v[4] = {v4.x, v4.y, v4.z, v4.w};
                const float wv[4] = {w[k].x, w[k].y, w[k].z, w[k].w};
                float av[4] = {a[k].x, a[k].y, a[k].z, a[k].w};
                float bv[4] = {b[k].x, b[k].y, b[k].z, b[k].w};
                float out[4];
                const bool in = pos.in(R::kAcc * c + i);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    out[e] = opt_step(p.op, v[e], wv[e], av[e], bv[e]);
                    if (in) {
                        s_ww = fmaf(wv[e], wv[e], s_ww);
                        s_dd = fmaf(out[e], out[e], s_dd);
                    }
                }
                if (in) {
                    const long long o = pos.at(p.ld, R::kAcc * c + i);
                    if (D)
                        *reinterpret_cast<float4*>(D + o) =
                            make_float4(out[0], out[1], out[2], out[3]);
                    if (p1) *reinterpret_cast<float4*>(p1 + o) = make_float4(av[0], av[1], av[2], av[3]);
                    if (p2) *reinterpret_cast<float4*>(p2 + o) = make_float4(bv[0], bv[1], bv[2], bv[3]);
                }
                if (R::kAcc * c + i + kAhead < R::kAcc * pos.kChunks) load(p, k, R::kAcc * c + i + kAhead);
            }
        }
        sums.add(c, {s_ww, s_dd});
    }

    __device__ __forceinline__ void finish(const Params& p, int lane) {
        sums.store(slot_of<2>(p.part, g, p.m256, p.n_blocks, row0, n0), lane);
    }
};

// ---------------------------------------------------------------------------
// Gate / up signals of a SwiGLU MLP (Sec. 3.1 step 5, Eq. errh): the GEMM gives
// error_h = g W3_init; with the cached pre-activations a (gate) and b (up),
//   dA = error_h (.) b (.) silu'(a),  dB = error_h (.) silu(a)   (bf16 out)
struct EpiSwigluBase {
    struct Params {
        __nv_bfloat16* dA;       // [M, N]
        __nv_bfloat16* dB;
        const __nv_bfloat16* a;  // [M, N]
        const __nv_bfloat16* b;
        long long ld;
        int M, N;
    };
};

template <int kCG>
struct EpiSwiglu : EpiSwigluBase {
    static constexpr int kWarps = 8, kColGroups = kCG;
    using R = RowChunk;
    RowPos<kCG> pos;
    uint2 ua[R::kAcc], ub[R::kAcc];  // a and b of the next chunk

    __device__ __forceinline__ void load(const Params& p, int c) {
#pragma unroll
        for (int i = 0; i < R::kAcc; ++i) {
            ua[i] = *reinterpret_cast<const uint2*>(pos.src(p.a, p.ld, R::kAcc * c + i));
            ub[i] = *reinterpret_cast<const uint2*>(pos.src(p.b, p.ld, R::kAcc * c + i));
        }
    }

    __device__ __forceinline__ EpiSwiglu(const Params& p, int, int row0, int n0, int lane)
        : pos(p.M, p.N, p.ld, row0, n0, lane) {
        load(p, 0);
    }

    __device__ __forceinline__ void chunk(const Params& p, uint32_t buf, int lane, int c) {
#pragma unroll
        for (int i = 0; i < R::kAcc; ++i) {
            const float4 v4 = R::read(buf, lane, i);
            const float v[4] = {v4.x, v4.y, v4.z, v4.w};
            const uint2 a2 = ua[i], b2 = ub[i];
            const float xa[4] = {__uint_as_float(a2.x << 16), __uint_as_float(a2.x & 0xffff0000u),
                                 __uint_as_float(a2.y << 16), __uint_as_float(a2.y & 0xffff0000u)};
            const float xb[4] = {__uint_as_float(b2.x << 16), __uint_as_float(b2.x & 0xffff0000u),
                                 __uint_as_float(b2.y << 16), __uint_as_float(b2.y & 0xffff0000u)};
            float da[4], db[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                // sigmoid with the fast intrinsic divide: its few-ulp fp32 error is far
                // below the bf16 rounding of dA and dB (for x < -87 it gives 0, as the
                // exact value is below bf16's range there too)
                const float x = xa[k];
                const float sg = __fdividef(1.f, 1.f + __expf(-x));
                da[k] = v[k] * xb[k] * sg * fmaf(x, 1.f - sg, 1.f);
                db[k] = v[k] * x * sg;
            }
            if (pos.in(R::kAcc * c + i)) {
                const long long o = pos.at(p.ld, R::kAcc * c + i);
                *reinterpret_cast<uint2*>(p.dA + o) =
                    make_uint2(pack_bf16x2(da[0], da[1]), pack_bf16x2(da[2], da[3]));
                *reinterpret_cast<uint2*>(p.dB + o) =
                    make_uint2(pack_bf16x2(db[0], db[1]), pack_bf16x2(db[2], db[3]));
            }
        }
        if (c + 1 < pos.kChunks) load(p, c + 1);
    }

    __device__ __forceinline__ void finish(const Params&, int) {}
};

}  // namespace fpo
