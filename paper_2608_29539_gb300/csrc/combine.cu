// combine.cu -- logo_combine / logo_combine_bwd(_gains): ContextNorm (Eq. 9,
// a head-wise RMSNorm over D per branch) fused with the gate-weighted output
// fusion of Eq. 10, the backward of both with z held fixed, and the gradients
// of the two ContextNorm gains.
//
// HBM-bound.  Blocks walk the tokens (grid-stride); a thread owns GPT fixed
// groups of G adjacent 16-byte vectors (8 G bf16 of one head row; G = 2 with
// unit gains, 1 when gains are read) of the token's [H, D] row, issues all of
// a token's loads before any arithmetic (so each thread keeps G*GPT to
// 3*G*GPT loads in flight), sums within its group, and the D/(8 G) lanes of a
// head reduce the sums with warp shuffles.  The backward sums dp_t over
// every head of the token in shared memory, and the gain gradients over the
// block's tokens in shared-memory slots that only the thread owning the vector
// touches, then per block into a workspace that a second kernel sums in a
// fixed order (colsum.cuh: deterministic).  All arithmetic is fp32; inputs
// and outputs bf16.
// The kernels are bound as much by instruction issue as by HBM: without gains
// (both NULL, i.e. 1) a separate instantiation drops the gain loads and the
// unit multiplies and does the elementwise work as f32x2 pairs; with gains,
// token rows of up to 8192 elements have kernels of their own ("gains read"
// below), and these serve the wider ones only.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "colsum.cuh"
#include "host_common.h"
#include "logo_status.cuh"
#include "sm100.cuh"

namespace logo {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxVec = 8 * kThreads;   // H*D/8 vectors per token at most (8 vectors per thread)
constexpr int kMaxVecGains = 4 * kThreads;

struct Vec8 {
    float v[8];
};

__device__ __forceinline__ uint4 ld_vec(const logo_bf16* p) { return *reinterpret_cast<const uint4*>(p); }

__device__ __forceinline__ Vec8 unpack8(const uint4& raw)
{
    Vec8 r;
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float2 f = __bfloat1622float2(h[i]);
        r.v[2 * i] = f.x;
        r.v[2 * i + 1] = f.y;
    }
    return r;
}

__device__ __forceinline__ void store_bf16x8(logo_bf16* p, const Vec8& x)
{
    uint4 raw;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&raw);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(x.v[2 * i], x.v[2 * i + 1]);
    *reinterpret_cast<uint4*>(p) = raw;
}

__device__ __forceinline__ Vec8 load_gain(const float* g, int h, int D, int j)
{
    Vec8 r;
    if (g) {
        const float4* p = reinterpret_cast<const float4*>(g + static_cast<int64_t>(h) * D + j * 8);
        float4 a = p[0], b = p[1];
        r.v[0] = a.x; r.v[1] = a.y; r.v[2] = a.z; r.v[3] = a.w;
        r.v[4] = b.x; r.v[5] = b.y; r.v[6] = b.z; r.v[7] = b.w;
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) r.v[i] = 1.0f;
    }
    return r;
}

// x * a + y * b elementwise (y, b optional), as f32x2 pairs
__device__ __forceinline__ Vec8 axpby8(const Vec8& x, float a, const Vec8* y, float b)
{
    const uint64_t a2 = f2_pack(a, a), b2 = f2_pack(b, b);
    Vec8 r;
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
        uint64_t t = f2_mul(f2_pack(x.v[i], x.v[i + 1]), a2);
        if (y) t = f2_fma(f2_pack(y->v[i], y->v[i + 1]), b2, t);
        f2_unpack(t, r.v[i], r.v[i + 1]);
    }
    return r;
}

// Gain-gradient accumulators of the backward, in shared memory: float4 slot
// (branch * 2 + half) * nvec + s holds elements 4 half .. 4 half + 3 of the
// sums of vector v = 2 (s mod npair) + s / npair (s = e npair + u for vector
// e of pair u).  Only the thread that owns the pair touches its slots, and a
// warp's 32 consecutive pairs are 32 consecutive float4 (no bank conflicts).
// In registers they took 32 more per thread (at Hq*D = 4096), which cut the
// resident blocks per SM, and with them the loads in flight, by half.
__device__ __forceinline__ void acc_add8(float4* sh, int nvec, int branch, int s, const Vec8& c)
{
    float4* p0 = sh + (branch * 2) * nvec + s;
    float4* p1 = p0 + nvec;
    float4 a = *p0, b = *p1;
    a.x += c.v[0]; a.y += c.v[1]; a.z += c.v[2]; a.w += c.v[3];
    b.x += c.v[4]; b.y += c.v[5]; b.z += c.v[6]; b.w += c.v[7];
    *p0 = a;
    *p1 = b;
}

// Sum over W consecutive lanes.
template <int W>
__device__ __forceinline__ float lane_sum(float x)
{
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Sum over the `width` consecutive lanes (a power of two <= 32) of one head.
__device__ __forceinline__ float head_sum(float x, int width)
{
    for (int o = width >> 1; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// A thread owns groups of G adjacent 16-byte vectors of one head row (8 G
// elements).  With G = 2 a head row of D elements is D/16 lanes, so its sums
// take one shuffle level fewer than with a vector per lane and one rsqrt
// serves 16 elements instead of 8: the unit-gain kernels, bound by instruction
// issue as much as by HBM, run with G = 2 when the token row has at least two
// vectors per thread of the block (Hq*D >= 4096: combine 56.7 -> 47.1 us,
// backward 87.9 -> 71.0 us at 16K).  Below that, pairs would leave threads of
// every block idle (4K, Hq*D = 2048: backward 26.5 -> 29.9 us), so G = 1.  The
// kernels that load gains keep G = 1: with two vectors' gains live they
// needed 120-127 registers instead of 72-80.
template <int G>
__device__ __forceinline__ float sumsq_g(const Vec8 (&x)[G])
{
    uint64_t a = 0ull, b = 0ull;
#pragma unroll
    for (int e = 0; e < G; ++e) {
        a = f2_fma(f2_pack(x[e].v[0], x[e].v[1]), f2_pack(x[e].v[0], x[e].v[1]), a);
        b = f2_fma(f2_pack(x[e].v[2], x[e].v[3]), f2_pack(x[e].v[2], x[e].v[3]), b);
        a = f2_fma(f2_pack(x[e].v[4], x[e].v[5]), f2_pack(x[e].v[4], x[e].v[5]), a);
        b = f2_fma(f2_pack(x[e].v[6], x[e].v[7]), f2_pack(x[e].v[6], x[e].v[7]), b);
    }
    float lo, hi;
    f2_unpack(f2_add(a, b), lo, hi);
    return lo + hi;
}

template <int G>
__device__ __forceinline__ float dot_g(const Vec8 (&x)[G], const Vec8 (&y)[G])
{
    uint64_t a = 0ull, b = 0ull;
#pragma unroll
    for (int e = 0; e < G; ++e) {
        a = f2_fma(f2_pack(x[e].v[0], x[e].v[1]), f2_pack(y[e].v[0], y[e].v[1]), a);
        b = f2_fma(f2_pack(x[e].v[2], x[e].v[3]), f2_pack(y[e].v[2], y[e].v[3]), b);
        a = f2_fma(f2_pack(x[e].v[4], x[e].v[5]), f2_pack(y[e].v[4], y[e].v[5]), a);
        b = f2_fma(f2_pack(x[e].v[6], x[e].v[7]), f2_pack(y[e].v[6], y[e].v[7]), b);
    }
    float lo, hi;
    f2_unpack(f2_add(a, b), lo, hi);
    return lo + hi;
}

// dp += dO . (xg r_g - xl r_l) over one vector, as f32x2 pairs
__device__ __forceinline__ uint64_t dp_acc8(uint64_t dp2, const Vec8& g, const Vec8& xl, const Vec8& xg,
                                            uint64_t rl2_neg, uint64_t rg2)
{
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
        const uint64_t t = f2_fma(f2_pack(xl.v[i], xl.v[i + 1]), rl2_neg, f2_mul(f2_pack(xg.v[i], xg.v[i + 1]), rg2));
        dp2 = f2_fma(f2_pack(g.v[i], g.v[i + 1]), t, dp2);
    }
    return dp2;
}

// GPT: groups per thread (group u = vectors G u .. G u + G - 1 of the token's
// [H, D] row; the D/(8 G) lanes of a head reduce its sums with warp shuffles).
template <int GPT, int G, bool UNIT>
__host__ __device__ constexpr int fwd_min_blocks()
{
    return G == 1 && UNIT && GPT == 1 ? 8 : (GPT == 1 || (G == 1 && GPT == 2) ? 5 : 1);
}

template <int GPT, int G, bool UNIT>
__global__ void __launch_bounds__(kThreads, fwd_min_blocks<GPT, G, UNIT>()) combine_fwd_kernel(
    const logo_bf16* __restrict__ o_l, const logo_bf16* __restrict__ o_c, const float* __restrict__ gate_p,
    const uint8_t* __restrict__ z, const int32_t* __restrict__ row_of, const float* __restrict__ gain_l,
    const float* __restrict__ gain_g, float eps, logo_bf16* __restrict__ o, float* __restrict__ rstd_l,
    float* __restrict__ rstd_g, int64_t ntok, int H, int D)
{
    static_assert(G == 1 || (G == 2 && UNIT), "two-vector groups only with unit gains");
    const int vpr = D / 8;               // vectors per head row
    const int gpr = vpr / G;             // groups per head row: the lanes sharing a head
    const int nvec = H * vpr;            // vectors per token
    const int ngrp = nvec / G;
    const float inv_d = 1.0f / static_cast<float>(D);
    for (int64_t bt = blockIdx.x; bt < ntok; bt += gridDim.x) {
        const bool sel = z[bt] != 0;
        const int64_t row = sel ? row_of[bt] : 0;
        const float pt = gate_p[bt];
        uint4 rl[GPT][G], rg[GPT][G];
#pragma unroll
        for (int k = 0; k < GPT; ++k) {
            const int u = threadIdx.x + k * kThreads;
            const bool active = u < ngrp;
#pragma unroll
            for (int e = 0; e < G; ++e) {
                const int v = G * u + e;
                rl[k][e] = active ? ld_vec(o_l + (bt * nvec + v) * 8) : make_uint4(0, 0, 0, 0);
                rg[k][e] = (sel && active) ? ld_vec(o_c + (row * nvec + v) * 8) : make_uint4(0, 0, 0, 0);
            }
        }
#pragma unroll
        for (int k = 0; k < GPT; ++k) {
            const int u = threadIdx.x + k * kThreads;
            const bool active = u < ngrp;
            const int v0 = G * u;
            const int h = active ? v0 / vpr : 0, j0 = active ? v0 % vpr : 0;
            Vec8 xl[G], out[G];
#pragma unroll
            for (int e = 0; e < G; ++e) xl[e] = unpack8(rl[k][e]);
            float r_l, r_g = 0.f;
            if constexpr (UNIT) {
                r_l = rsqrtf(head_sum(sumsq_g<G>(xl), gpr) * inv_d + eps);
                if (sel) {
                    Vec8 xg[G];
#pragma unroll
                    for (int e = 0; e < G; ++e) xg[e] = unpack8(rg[k][e]);
                    r_g = rsqrtf(head_sum(sumsq_g<G>(xg), gpr) * inv_d + eps);
#pragma unroll
                    for (int e = 0; e < G; ++e) out[e] = axpby8(xl[e], (1.0f - pt) * r_l, &xg[e], pt * r_g);
                } else {
#pragma unroll
                    for (int e = 0; e < G; ++e) out[e] = axpby8(xl[e], r_l, nullptr, 0.f);
                }
            } else {  // G = 1
                float ss = 0.f;
#pragma unroll
                for (int i = 0; i < 8; ++i) ss += xl[0].v[i] * xl[0].v[i];
                ss = head_sum(ss, gpr);
                r_l = rsqrtf(ss * inv_d + eps);
                const Vec8 gl = load_gain(gain_l, h, D, j0);
#pragma unroll
                for (int i = 0; i < 8; ++i) out[0].v[i] = xl[0].v[i] * r_l * gl.v[i];
                if (sel) {
                    const Vec8 xg = unpack8(rg[k][0]);
                    float sg = 0.f;
#pragma unroll
                    for (int i = 0; i < 8; ++i) sg += xg.v[i] * xg.v[i];
                    sg = head_sum(sg, gpr);
                    r_g = rsqrtf(sg * inv_d + eps);
                    const Vec8 gg = load_gain(gain_g, h, D, j0);
#pragma unroll
                    for (int i = 0; i < 8; ++i) out[0].v[i] = (1.0f - pt) * out[0].v[i] + pt * (xg.v[i] * r_g * gg.v[i]);
                }
            }
            if (active)
#pragma unroll
                for (int e = 0; e < G; ++e) store_bf16x8(o + (bt * nvec + v0 + e) * 8, out[e]);
            if (active && j0 == 0) {
                if (rstd_l) rstd_l[bt * H + h] = r_l;
                if (sel && rstd_g) rstd_g[row * H + h] = r_g;
            }
        }
    }
}

// Register bound of a backward variant: with unit gains one two-vector group
// per thread is held to 4 blocks per SM (3 with the gain sums in shared
// memory), one one-vector group to 5, with the gain sums up to two of them to 3.
template <int GPT, int G, bool DGAIN, bool UNIT>
__host__ __device__ constexpr int bwd_min_blocks()
{
    return G == 2 ? (GPT == 1 ? (DGAIN ? 3 : 4) : 1)
                  : (DGAIN && GPT <= 2 ? 3 : (UNIT && GPT == 1 ? 5 : 1));
}

// part (DGAIN): [gridDim.x][2][H*D] float32 per-block sums of the local and
// global gain gradients, accumulated in dynamic shared memory (4 * nvec float4,
// see acc_add8) over the block's tokens in increasing order.
template <int GPT, int G, bool DGAIN, bool UNIT>
__global__ void __launch_bounds__(kThreads, bwd_min_blocks<GPT, G, DGAIN, UNIT>()) combine_bwd_kernel(
    const logo_bf16* __restrict__ dO, const logo_bf16* __restrict__ o_l, const logo_bf16* __restrict__ o_c,
    const float* __restrict__ gate_p, const uint8_t* __restrict__ z, const int32_t* __restrict__ row_of,
    const float* __restrict__ gain_l, const float* __restrict__ gain_g, float eps, logo_bf16* __restrict__ dO_l,
    logo_bf16* __restrict__ dO_c, float* __restrict__ dgate_p, float* __restrict__ part, int64_t ntok, int H, int D)
{
    static_assert(UNIT || (G == 1 && !DGAIN), "two-vector groups and gain sums only with unit gains");
    __shared__ float sh_dp[2][kThreads / 32];
    const int vpr = D / 8, gpr = vpr / G;
    const int nvec = H * vpr, ngrp = nvec / G;
    const float inv_d = 1.0f / static_cast<float>(D);
    extern __shared__ float4 sh_acc[];
    if (DGAIN) {
#pragma unroll
        for (int k = 0; k < GPT; ++k) {
            const int u = threadIdx.x + k * kThreads;
            if (u < ngrp)
#pragma unroll
                for (int s = 0; s < 4; ++s)
#pragma unroll
                    for (int e = 0; e < G; ++e) sh_acc[s * nvec + e * ngrp + u] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    int n_sel_seen = 0;
    for (int64_t bt = blockIdx.x; bt < ntok; bt += gridDim.x) {
        const bool sel = z[bt] != 0;
        const int64_t row = sel ? row_of[bt] : 0;
        const float pt = gate_p[bt];
        const float wl = sel ? 1.0f - pt : 1.0f;
        uint4 rd[GPT][G], rl[GPT][G], rg[GPT][G];
#pragma unroll
        for (int k = 0; k < GPT; ++k) {
            const int u = threadIdx.x + k * kThreads;
            const bool active = u < ngrp;
#pragma unroll
            for (int e = 0; e < G; ++e) {
                const int v = G * u + e;
                rd[k][e] = active ? ld_vec(dO + (bt * nvec + v) * 8) : make_uint4(0, 0, 0, 0);
                rl[k][e] = active ? ld_vec(o_l + (bt * nvec + v) * 8) : make_uint4(0, 0, 0, 0);
                rg[k][e] = (sel && active) ? ld_vec(o_c + (row * nvec + v) * 8) : make_uint4(0, 0, 0, 0);
            }
        }
        float dp_acc = 0.f;
        uint64_t dp2 = 0ull;  // UNIT: dp as f32x2 pairs
#pragma unroll
        for (int k = 0; k < GPT; ++k) {
            const int u = threadIdx.x + k * kThreads;
            const bool active = u < ngrp;
            const int v0 = G * u;
            const int h = active ? v0 / vpr : 0, j0 = active ? v0 % vpr : 0;
            Vec8 g[G], xl[G];
#pragma unroll
            for (int e = 0; e < G; ++e) {
                g[e] = unpack8(rd[k][e]);
                xl[e] = unpack8(rl[k][e]);
            }
            if constexpr (UNIT) {
                // gains 1: dx = r dy - x r^3 mean(x dy), dy = w dO
                const float ss = head_sum(sumsq_g<G>(xl), gpr);
                const float xgdy = head_sum(dot_g<G>(xl, g), gpr) * wl;
                const float r_l = rsqrtf(ss * inv_d + eps);
                const float cl = r_l * r_l * r_l * xgdy * inv_d;
#pragma unroll
                for (int e = 0; e < G; ++e) {
                    if (active) store_bf16x8(dO_l + (bt * nvec + v0 + e) * 8, axpby8(g[e], r_l * wl, &xl[e], -cl));
                    if constexpr (DGAIN) {  // d gain_l = dy * x r
                        Vec8 c;
#pragma unroll
                        for (int i = 0; i < 8; ++i) c.v[i] = g[e].v[i] * wl * xl[e].v[i] * r_l;
                        if (active) acc_add8(sh_acc, nvec, 0, e * ngrp + u, c);
                    }
                }
                if (sel) {
                    Vec8 xg[G];
#pragma unroll
                    for (int e = 0; e < G; ++e) xg[e] = unpack8(rg[k][e]);
                    const float sg = head_sum(sumsq_g<G>(xg), gpr);
                    const float xgdyg = head_sum(dot_g<G>(xg, g), gpr) * pt;
                    const float r_g = rsqrtf(sg * inv_d + eps);
                    const float cg = r_g * r_g * r_g * xgdyg * inv_d;
                    const uint64_t rg2 = f2_pack(r_g, r_g), rl2 = f2_pack(-r_l, -r_l);
#pragma unroll
                    for (int e = 0; e < G; ++e) {
                        if (active) store_bf16x8(dO_c + (row * nvec + v0 + e) * 8, axpby8(g[e], r_g * pt, &xg[e], -cg));
                        if constexpr (DGAIN) {
                            Vec8 c;
#pragma unroll
                            for (int i = 0; i < 8; ++i) c.v[i] = g[e].v[i] * pt * xg[e].v[i] * r_g;
                            if (active) acc_add8(sh_acc, nvec, 1, e * ngrp + u, c);
                        }
                        dp2 = dp_acc8(dp2, g[e], xl[e], xg[e], rl2, rg2);  // dp += dO . (xg r_g - xl r_l)
                    }
                }
                continue;
            }
            // gains read (G = 1): local branch dy = dO * wl; dx = r g dy - x r^3 mean(x g dy)
            const Vec8 gl = load_gain(gain_l, h, D, j0);
            float ss = 0.f, xgdy = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                ss += xl[0].v[i] * xl[0].v[i];
                xgdy += xl[0].v[i] * gl.v[i] * g[0].v[i];
            }
            ss = head_sum(ss, gpr);
            xgdy = head_sum(xgdy, gpr) * wl;
            const float r_l = rsqrtf(ss * inv_d + eps);
            const float cl = r_l * r_l * r_l * xgdy * inv_d;
            Vec8 dxl;
#pragma unroll
            for (int i = 0; i < 8; ++i) dxl.v[i] = r_l * gl.v[i] * g[0].v[i] * wl - xl[0].v[i] * cl;
            if (active) store_bf16x8(dO_l + (bt * nvec + v0) * 8, dxl);
            if (sel) {
                const Vec8 xg = unpack8(rg[k][0]);
                const Vec8 gg = load_gain(gain_g, h, D, j0);
                float sg = 0.f, xgdyg = 0.f;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    sg += xg.v[i] * xg.v[i];
                    xgdyg += xg.v[i] * gg.v[i] * g[0].v[i];
                }
                sg = head_sum(sg, gpr);
                xgdyg = head_sum(xgdyg, gpr) * pt;
                const float r_g = rsqrtf(sg * inv_d + eps);
                const float cg = r_g * r_g * r_g * xgdyg * inv_d;
                Vec8 dxg;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    dxg.v[i] = r_g * gg.v[i] * g[0].v[i] * pt - xg.v[i] * cg;
                    dp_acc += g[0].v[i] * (xg.v[i] * r_g * gg.v[i] - xl[0].v[i] * r_l * gl.v[i]);
                }
                if (active) store_bf16x8(dO_c + (row * nvec + v0) * 8, dxg);
            }
        }
        if constexpr (UNIT) {
            float lo, hi;
            f2_unpack(dp2, lo, hi);
            dp_acc = lo + hi;
        }
        // dp_t = z_t * sum_{h,d} dO (o~G - o~L); z_t is uniform over the block
        if (sel) {
            const int buf = n_sel_seen & 1;
            ++n_sel_seen;
            dp_acc = head_sum(dp_acc, 32);
            if ((threadIdx.x & 31) == 0) sh_dp[buf][threadIdx.x >> 5] = dp_acc;
            __syncthreads();
            if (threadIdx.x == 0) {
                float s = 0.f;
#pragma unroll
                for (int w = 0; w < kThreads / 32; ++w) s += sh_dp[buf][w];
                dgate_p[bt] = s;
            }
        } else if (threadIdx.x == 0) {
            dgate_p[bt] = 0.0f;
        }
    }
    if (DGAIN) {
        const int64_t hd = static_cast<int64_t>(nvec) * 8;
        float* pl = part + static_cast<int64_t>(blockIdx.x) * 2 * hd;
#pragma unroll
        for (int k = 0; k < GPT; ++k) {
            const int u = threadIdx.x + k * kThreads;
            if (u < ngrp) {
#pragma unroll
                for (int e = 0; e < G; ++e) {
                    const int v = G * u + e, s = e * ngrp + u;
#pragma unroll
                    for (int br = 0; br < 2; ++br) {
                        float4* dst = reinterpret_cast<float4*>(pl + br * hd + v * 8);
                        dst[0] = sh_acc[(br * 2) * nvec + s];
                        dst[1] = sh_acc[(br * 2 + 1) * nvec + s];
                    }
                }
            }
        }
    }
}

// ------------------------------------------------------------- gains read
// The kernels for trained gains (either gain pointer given), Hq*D <= 8192: one
// 16-byte vector of the token row per thread, and as many rows of threads as
// fill 256 threads when the token row is short.  Each thread copies its
// vectors of the next tokens into shared-memory slots of its own (cp.async, a
// ring of kRing tokens; nothing but the thread itself reads them, so there is
// no barrier), which keeps (kRing - 1) x 16 to 48 bytes a thread in flight at
// no cost in registers: those hold the thread's gains and its sums of the
// gains' gradients for the whole kernel.  The routing (row_of, z, p) of a
// warp's next 32 tokens is loaded at once, one token a lane, 32 steps ahead:
// the tokens of a block lie a grid apart, so each of these loads is a DRAM
// access of its own, and fetched one step ahead they set the pace (2460 clocks
// a step at 16K).  D is a template parameter and addresses advance by adding:
// the first version of this layout ran 200 and 280 instructions a vector and
// was bound by issue.  Before, a thread had one token's loads in flight,
// fetched the gains from L1 for every token and kept the sums in shared
// memory.  16K, 32 heads, d 128, 1/8 selected (kernel times by ncu): forward 70 ->
// 46 us (287 MB, 6.2 TB/s, 91% of the copy rate), backward with gain gradients
// 124 -> 78 us (436 MB, 5.6 TB/s, 82%).
template <int MAXT>
struct GainCfg {
    // The forward runs two blocks of 512 threads an SM at 64 registers, its
    // gains in shared-memory slots of the thread (one block at 80 registers
    // with the gains in them: 54.5 against 48.6 us at 16K).  The backward's
    // gains and sums take 32 registers: one block of 512 threads at up to 128;
    // a token row of more than 512 vectors (Hq*D > 4096) takes a block of 1024
    // at 64, where gains and sums sit in shared memory beside a shorter ring.
    static constexpr int kRingFwd = 3;
    static constexpr bool kInRegs = MAXT <= 512;
    static constexpr int kRingBwd = kInRegs ? 4 : 2;
};

struct Routing {
    int row;  // packed row, -1: not selected (or no such token)
    float p;

    __device__ __forceinline__ void load(const uint8_t* z, const int32_t* row_of, const float* gate_p, int64_t t,
                                         int64_t ntok)
    {
        const bool have = t < ntok;
        const int r = have ? row_of[t] : -1;
        const bool sel = have && z[t] != 0;
        p = have ? gate_p[t] : 0.f;
        row = sel ? r : -1;
    }
};

// Routing of the tokens t0, t0 + step, t0 + 2 step, .. of a warp, handed out in
// order; called by all 32 lanes.
struct RoutingAhead {
    Routing cur, next;  // of this lane's token in the batch of 32, and in the one after
    int k;

    __device__ __forceinline__ RoutingAhead(const uint8_t* z, const int32_t* row_of, const float* gate_p, int64_t t0,
                                            int64_t step, int64_t ntok)
        : k(0)
    {
        const int lane = threadIdx.x & 31;
        cur.load(z, row_of, gate_p, t0 + lane * step, ntok);
        next.load(z, row_of, gate_p, t0 + (lane + 32) * step, ntok);
    }
    // t: the token asked for
    __device__ __forceinline__ Routing get(const uint8_t* z, const int32_t* row_of, const float* gate_p, int64_t t,
                                           int64_t step, int64_t ntok)
    {
        const Routing r{__shfl_sync(0xffffffffu, cur.row, k), __shfl_sync(0xffffffffu, cur.p, k)};
        if (++k == 32) {
            k = 0;
            cur = next;
            next.load(z, row_of, gate_p, t + (33 + (threadIdx.x & 31)) * step, ntok);
        }
        return r;
    }
};

// 8 floats of the thread in shared memory: float4 slot (2 k + half) * n + s.
__device__ __forceinline__ Vec8 slot_load(const float4* sh, int n, int k, int s)
{
    const float4 a = sh[k * 2 * n + s], b = sh[(k * 2 + 1) * n + s];
    return Vec8{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}

__device__ __forceinline__ void slot_store(float4* sh, int n, int k, int s, const Vec8& x)
{
    sh[k * 2 * n + s] = make_float4(x.v[0], x.v[1], x.v[2], x.v[3]);
    sh[(k * 2 + 1) * n + s] = make_float4(x.v[4], x.v[5], x.v[6], x.v[7]);
}

__device__ __forceinline__ Vec8 mul8(const Vec8& x, const Vec8& y)
{
    Vec8 r;
#pragma unroll
    for (int i = 0; i < 8; i += 2)
        f2_unpack(f2_mul(f2_pack(x.v[i], x.v[i + 1]), f2_pack(y.v[i], y.v[i + 1])), r.v[i], r.v[i + 1]);
    return r;
}

// acc += x * y * a
__device__ __forceinline__ void fma8(Vec8& acc, const Vec8& x, const Vec8& y, float a)
{
    const uint64_t a2 = f2_pack(a, a);
#pragma unroll
    for (int i = 0; i < 8; i += 2)
        f2_unpack(f2_fma(f2_mul(f2_pack(x.v[i], x.v[i + 1]), a2), f2_pack(y.v[i], y.v[i + 1]),
                         f2_pack(acc.v[i], acc.v[i + 1])),
                  acc.v[i], acc.v[i + 1]);
}

__device__ __forceinline__ float sumsq8(const Vec8& x)
{
    const Vec8 a[1] = {x};
    return sumsq_g<1>(a);
}

__device__ __forceinline__ float dot8(const Vec8& x, const Vec8& y)
{
    const Vec8 a[1] = {x}, b[1] = {y};
    return dot_g<1>(a, b);
}

// Where thread threadIdx.x stands: its row of threads (tpr of them, a multiple
// of 32) and its vector there.
template <int D>
struct GainPlace {
    int row, v, h, j0;
    bool active;

    __device__ __forceinline__ GainPlace(int tpr, int nvec)
    {
        row = threadIdx.x / tpr;
        v = threadIdx.x - row * tpr;
        active = v < nvec;
        h = active ? v / (D / 8) : 0;
        j0 = active ? v % (D / 8) : 0;
    }
};

template <int D, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 512 ? 2 : 1) combine_gained_fwd_kernel(
    const logo_bf16* __restrict__ o_l, const logo_bf16* __restrict__ o_c, const float* __restrict__ gate_p,
    const uint8_t* __restrict__ z, const int32_t* __restrict__ row_of, const float* __restrict__ gain_l,
    const float* __restrict__ gain_g, float eps, logo_bf16* __restrict__ o, float* __restrict__ rstd_l,
    float* __restrict__ rstd_g, int64_t ntok, int H, int tpr, int rows)
{
    constexpr int S = GainCfg<MAXT>::kRingFwd, VPR = D / 8;
    extern __shared__ float4 sh_dyn[];  // ring [S][o_l, o_c][thread] of 16 bytes, then the gains
    __shared__ Routing sh_rt[S][32];    // per warp
    const int nvec = H * VPR, nthr = blockDim.x, warp = threadIdx.x >> 5;
    const GainPlace<D> me(tpr, nvec);
    float4* sh_gain = sh_dyn + S * 2 * nthr;
    slot_store(sh_gain, nthr, 0, threadIdx.x, load_gain(gain_l, me.h, D, me.j0));
    slot_store(sh_gain, nthr, 1, threadIdx.x, load_gain(gain_g, me.h, D, me.j0));
    const int64_t step = static_cast<int64_t>(gridDim.x) * rows;
    int64_t t = static_cast<int64_t>(blockIdx.x) * rows + me.row, t_issue = t;
    const int64_t step_el = step * nvec * 8;             // elements from one of this thread's tokens to the next
    int64_t off = (t * nvec + me.v) * 8, off_issue = off;
    const logo_bf16* oc_v = o_c + me.v * 8;
    RoutingAhead ahead(z, row_of, gate_p, t, step, ntok);
    const uint32_t ring = smem_u32(sh_dyn + threadIdx.x), stage_bytes = 2 * nthr * 16;
    uint32_t dst = ring;
    Routing* rt_issue = &sh_rt[0][warp];
    int n_issue = 0;
    auto issue = [&]() {
        const Routing nx = ahead.get(z, row_of, gate_p, t_issue, step, ntok);
        if (me.active && t_issue < ntok) {
            cp_async16(dst, o_l + off_issue);
            if (nx.row >= 0) cp_async16(dst + nthr * 16, oc_v + static_cast<int64_t>(nx.row) * (nvec * 8));
        }
        cp_async_commit();
        if ((threadIdx.x & 31) == 0) *rt_issue = nx;
        t_issue += step;
        off_issue += step_el;
        const bool wrap = ++n_issue == S;
        n_issue = wrap ? 0 : n_issue;
        dst = wrap ? ring : dst + stage_bytes;
        rt_issue = wrap ? &sh_rt[0][warp] : rt_issue + 32;
    };
#pragma unroll 1
    for (int i = 0; i < S - 1; ++i) issue();
    int st = 0;
    const float4* slot = sh_dyn + threadIdx.x;
    for (; t < ntok; t += step, off += step_el) {
        __syncwarp();  // every lane has read the routing slot that is written next
        issue();
        cp_async_wait<S - 1>();
        __syncwarp();
        const Routing rt = sh_rt[st][warp];
        const Vec8 x = unpack8(*reinterpret_cast<const uint4*>(slot));
        const float r_l = rsqrtf(lane_sum<VPR>(sumsq8(x)) * (1.0f / D) + eps);
        const bool sel = rt.row >= 0;
        Vec8 out = mul8(axpby8(x, sel ? (1.0f - rt.p) * r_l : r_l, nullptr, 0.f),
                        slot_load(sh_gain, nthr, 0, threadIdx.x));
        if (sel) {
            const Vec8 xg = unpack8(*reinterpret_cast<const uint4*>(slot + nthr));
            const float r_g = rsqrtf(lane_sum<VPR>(sumsq8(xg)) * (1.0f / D) + eps);
            fma8(out, xg, slot_load(sh_gain, nthr, 1, threadIdx.x), rt.p * r_g);
            if (me.active && me.j0 == 0 && rstd_g) rstd_g[static_cast<int64_t>(rt.row) * H + me.h] = r_g;
        }
        if (me.active) {
            store_bf16x8(o + off, out);
            if (me.j0 == 0 && rstd_l) rstd_l[t * H + me.h] = r_l;
        }
        const bool wrap = ++st == S;
        st = wrap ? 0 : st;
        slot = wrap ? sh_dyn + threadIdx.x : slot + 2 * nthr;
    }
    cp_async_wait<0>();
}

// part (DGAIN): [gridDim.x][2][H*D] float32 per-block sums of the local and
// global gain gradients.
template <int D, int MAXT, bool DGAIN>
__global__ void __launch_bounds__(MAXT) combine_gained_bwd_kernel(
    const logo_bf16* __restrict__ dO, const logo_bf16* __restrict__ o_l, const logo_bf16* __restrict__ o_c,
    const float* __restrict__ gate_p, const uint8_t* __restrict__ z, const int32_t* __restrict__ row_of,
    const float* __restrict__ gain_l, const float* __restrict__ gain_g, float eps, logo_bf16* __restrict__ dO_l,
    logo_bf16* __restrict__ dO_c, float* __restrict__ dgate_p, float* __restrict__ part, int64_t ntok, int H, int tpr,
    int rows)
{
    constexpr int S = GainCfg<MAXT>::kRingBwd, VPR = D / 8;
    constexpr bool kInRegs = GainCfg<MAXT>::kInRegs;
    constexpr int kGroup = 8;  // tokens whose dp sums share a barrier
    extern __shared__ float4 sh_dyn[];  // ring [S][dO, o_l, o_c][thread], gains and (DGAIN) sums unless in registers
    __shared__ Routing sh_rt[S][32];    // per warp
    __shared__ float sh_dp[2][kGroup][32];
    const int nvec = H * VPR, nthr = blockDim.x, warp = threadIdx.x >> 5;
    const GainPlace<D> me(tpr, nvec);
    float4* sh_gain = sh_dyn + S * 3 * nthr;
    float4* sh_sum = sh_gain + (kInRegs ? 0 : 4 * nthr);
    const Vec8 gl_r = load_gain(gain_l, me.h, D, me.j0), gg_r = load_gain(gain_g, me.h, D, me.j0);
    Vec8 sum_l{}, sum_g{};
    if (!kInRegs) {
        slot_store(sh_gain, nthr, 0, threadIdx.x, gl_r);
        slot_store(sh_gain, nthr, 1, threadIdx.x, gg_r);
        if (DGAIN) {
            slot_store(sh_sum, nthr, 0, threadIdx.x, sum_l);
            slot_store(sh_sum, nthr, 1, threadIdx.x, sum_g);
        }
    }
    // slots of vectors and tokens that do not exist are never copied to
    for (int i = 0; i < S * 3; ++i) sh_dyn[i * nthr + threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t step = static_cast<int64_t>(gridDim.x) * rows;
    int64_t t = static_cast<int64_t>(blockIdx.x) * rows + me.row, t_issue = t;
    const int64_t step_el = step * nvec * 8;
    int64_t off = (t * nvec + me.v) * 8, off_issue = off;
    const logo_bf16* oc_v = o_c + me.v * 8;
    logo_bf16* dc_v = dO_c + me.v * 8;
    RoutingAhead ahead(z, row_of, gate_p, t, step, ntok);
    const uint32_t ring = smem_u32(sh_dyn + threadIdx.x), stage_bytes = 3 * nthr * 16;
    uint32_t dst = ring;
    Routing* rt_issue = &sh_rt[0][warp];
    int n_issue = 0;
    auto issue = [&]() {
        const Routing nx = ahead.get(z, row_of, gate_p, t_issue, step, ntok);
        if (me.active && t_issue < ntok) {
            cp_async16(dst, dO + off_issue);
            cp_async16(dst + nthr * 16, o_l + off_issue);
            if (nx.row >= 0) cp_async16(dst + nthr * 32, oc_v + static_cast<int64_t>(nx.row) * (nvec * 8));
        }
        cp_async_commit();
        if ((threadIdx.x & 31) == 0) *rt_issue = nx;
        t_issue += step;
        off_issue += step_el;
        const bool wrap = ++n_issue == S;
        n_issue = wrap ? 0 : n_issue;
        dst = wrap ? ring : dst + stage_bytes;
        rt_issue = wrap ? &sh_rt[0][warp] : rt_issue + 32;
    };
#pragma unroll 1
    for (int i = 0; i < S - 1; ++i) issue();
    int st = 0, k = 0, buf = 0;
    const float4* slot = sh_dyn + threadIdx.x;
    // every row of threads makes the same number of steps (the barriers)
    for (int64_t tb = static_cast<int64_t>(blockIdx.x) * rows; tb < ntok; tb += step, t += step, off += step_el) {
        __syncwarp();  // every lane has read the routing slot that is written next
        issue();
        cp_async_wait<S - 1>();
        __syncwarp();
        const Routing rt = sh_rt[st][warp];
        const bool live = me.active && t < ntok;
        const bool sel = rt.row >= 0;
        const float pt = rt.p, wl = sel ? 1.0f - pt : 1.0f;
        const Vec8 g = unpack8(*reinterpret_cast<const uint4*>(slot));
        float dp = 0.f, r_l, xl;  // the local branch's 1 / rms, and this lane's part of x dy / wl
        {  // dy = dO wl; dx = r gain dy - x r^3 mean(x gain dy); d gain = dy x r
            const Vec8 x = unpack8(*reinterpret_cast<const uint4*>(slot + nthr));
            const Vec8 gy = mul8(g, kInRegs ? gl_r : slot_load(sh_gain, nthr, 0, threadIdx.x));
            const float ss = lane_sum<VPR>(sumsq8(x));
            xl = dot8(x, gy);
            const float xd = lane_sum<VPR>(xl);
            const float r = r_l = rsqrtf(ss * (1.0f / D) + eps);
            if (live) store_bf16x8(dO_l + off, axpby8(gy, r * wl, &x, -(r * r * r * (xd * wl) * (1.0f / D))));
            if (DGAIN && kInRegs && live) fma8(sum_l, g, x, wl * r);  // (a slot past the end may hold infinities)
            if (DGAIN && !kInRegs && live) {
                Vec8 a = slot_load(sh_sum, nthr, 0, threadIdx.x);
                fma8(a, g, x, wl * r);
                slot_store(sh_sum, nthr, 0, threadIdx.x, a);
            }
        }
        if (sel) {
            const Vec8 x = unpack8(*reinterpret_cast<const uint4*>(slot + 2 * nthr));
            const Vec8 gy = mul8(g, kInRegs ? gg_r : slot_load(sh_gain, nthr, 1, threadIdx.x));
            const float ss = lane_sum<VPR>(sumsq8(x));
            const float xg = dot8(x, gy), xd = lane_sum<VPR>(xg);
            const float r = rsqrtf(ss * (1.0f / D) + eps);
            if (live)
                store_bf16x8(dc_v + static_cast<int64_t>(rt.row) * (nvec * 8),
                             axpby8(gy, r * pt, &x, -(r * r * r * (xd * pt) * (1.0f / D))));
            if (DGAIN && kInRegs && live) fma8(sum_g, g, x, pt * r);
            if (DGAIN && !kInRegs && live) {
                Vec8 a = slot_load(sh_sum, nthr, 1, threadIdx.x);
                fma8(a, g, x, pt * r);
                slot_store(sh_sum, nthr, 1, threadIdx.x, a);
            }
            // dp_t = z_t sum over heads and d of dO (o~G - o~L), the difference taken
            // of each lane's eight elements: the branches' outputs may nearly agree,
            // and the difference of their heads' sums then had 1.8 times the error
            // (five times where they are equal; these products are rounded alike, not
            // one of them by an FMA, so that equal branches give zero)
            dp = lane_sum<32>(__fsub_rn(__fmul_rn(r, xg), __fmul_rn(r_l, xl)));
        }
        if ((threadIdx.x & 31) == 0) sh_dp[buf][k][warp] = sel ? dp : 0.f;
        if (++k == kGroup || tb + step >= ntok) {  // (two buffers: one barrier a group is enough)
            __syncthreads();
            if (me.v < k) {
                const int64_t tj = t - (k - 1 - me.v) * step;
                if (tj < ntok) {
                    float s = 0.f;
                    for (int w = 0; w < tpr / 32; ++w) s += sh_dp[buf][me.v][me.row * (tpr / 32) + w];
                    dgate_p[tj] = s;
                }
            }
            k = 0;
            buf ^= 1;
        }
        const bool wrap = ++st == S;
        st = wrap ? 0 : st;
        slot = wrap ? sh_dyn + threadIdx.x : slot + 3 * nthr;
    }
    cp_async_wait<0>();
    if (DGAIN) {
        // the block's rows of threads in order, then its partial row
        if (kInRegs) {
            __syncthreads();  // the ring is free
            sh_sum = sh_dyn;
            slot_store(sh_sum, nthr, 0, threadIdx.x, sum_l);
            slot_store(sh_sum, nthr, 1, threadIdx.x, sum_g);
        }
        __syncthreads();
        if (me.row == 0 && me.active) {
            float* pl = part + static_cast<int64_t>(blockIdx.x) * 2 * nvec * 8;
#pragma unroll
            for (int br = 0; br < 2; ++br)
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    float4 a = sh_sum[(br * 2 + half) * nthr + threadIdx.x];
                    for (int r = 1; r < rows; ++r) {
                        const float4 b = sh_sum[(br * 2 + half) * nthr + r * tpr + threadIdx.x];
                        a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
                    }
                    *reinterpret_cast<float4*>(pl + static_cast<int64_t>(br) * nvec * 8 + me.v * 8 + half * 4) = a;
                }
        }
    }
}

// Threads per token row and rows of threads per block of the kernels above.
struct GainShape {
    int tpr, rows, threads;
};

GainShape gain_shape(const logo_dims& d)
{
    const int nvec = d.Hq * (d.D / 8);
    const int tpr = (nvec + 31) / 32 * 32;
    const int rows = tpr >= kThreads ? 1 : kThreads / tpr;
    return GainShape{tpr, rows, tpr * rows};
}

// Vectors per group: two with unit gains when that leaves no thread of the
// block idle (at least 2 x kThreads vectors per token), else one.
int group_vectors(const logo_dims& d, bool unit)
{
    return unit && d.Hq * (d.D / 8) >= 2 * kThreads ? 2 : 1;
}

// Groups of vectors per thread: 1, 2, 4 or 8.
int groups_per_thread(const logo_dims& d, int g)
{
    const int ngrp = d.Hq * (d.D / 8) / g;
    const int need = (ngrp + kThreads - 1) / kThreads;
    return need <= 1 ? 1 : need <= 2 ? 2 : need <= 4 ? 4 : 8;
}

// One wave of resident blocks (the grid-stride loop gives every block the
// same number of tokens), capped by the steps there are.
template <typename K>
int64_t wave_blocks(K kernel, int64_t steps, size_t smem = 0, int threads = kThreads)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    const int64_t cap = static_cast<int64_t>(device_sm_count()) * per_sm;
    return steps < cap ? steps : cap;
}

// Dynamic shared memory of the unit-gain backward with gain sums: its accumulators.
size_t gains_smem(const logo_dims& d) { return static_cast<size_t>(4) * (d.Hq * d.D / 8) * sizeof(float4); }

// The gain variant may need more than the default 48 KB of dynamic shared
// memory (64 KB at Hq*D = 8192); the attribute is set before any occupancy
// query or launch of it.
template <typename K>
bool gains_smem_ok(K kernel, size_t bytes = 4 * kMaxVecGains * sizeof(float4))
{
    return set_smem_limit(kernel, static_cast<int>(bytes)) == cudaSuccess;
}

// A launch of the gains-read kernels; `slots`: float4 of shared memory per thread.
// A kernel's limit is set to what its largest block takes, whatever this call's
// size: calls of other sizes may be under way on other threads.
struct GainLaunch {
    GainShape sh;
    size_t smem;
    int64_t grid;
    bool ok;
};

template <typename K>
GainLaunch gain_launch(K kernel, const logo_dims& d, int slots)
{
    GainLaunch g{gain_shape(d), 0, 0, false};
    g.smem = static_cast<size_t>(slots) * g.sh.threads * sizeof(float4);
    const int max_threads = g.sh.threads > 512 ? 1024 : 512;
    g.ok = gains_smem_ok(kernel, static_cast<size_t>(slots) * max_threads * sizeof(float4));
    const int64_t ntok = static_cast<int64_t>(d.B) * d.T;
    g.grid = wave_blocks(kernel, (ntok + g.sh.rows - 1) / g.sh.rows, g.smem, g.sh.threads);
    return g;
}

// Calls f(kernel, float4 slots per thread) with the backward kernel that runs for these sizes.
template <bool DGAIN, typename F>
auto with_gained_bwd(const logo_dims& d, F f)
{
    constexpr int kSlots = 3 * GainCfg<512>::kRingBwd;
    constexpr int kSlotsBig = 3 * GainCfg<1024>::kRingBwd + (DGAIN ? 8 : 4);
    const bool big = gain_shape(d).threads > 512;
    if (d.D == 128) return big ? f(combine_gained_bwd_kernel<128, 1024, DGAIN>, kSlotsBig)
                               : f(combine_gained_bwd_kernel<128, 512, DGAIN>, kSlots);
    return big ? f(combine_gained_bwd_kernel<64, 1024, DGAIN>, kSlotsBig)
               : f(combine_gained_bwd_kernel<64, 512, DGAIN>, kSlots);
}

// Blocks of the gain-gradient backward (one partial row each): the larger of
// its two variants, so the workspace fits whichever runs.
int64_t gains_blocks(const logo_dims& d)
{
    const int64_t ntok = static_cast<int64_t>(d.B) * d.T;
    const size_t smem = gains_smem(d);
    const int64_t with_gains =
        with_gained_bwd<true>(d, [&](auto kernel, int slots) { return gain_launch(kernel, d, slots).grid; });
    int64_t unit = 0;
    const int gu = group_vectors(d, true), gpt = groups_per_thread(d, gu);
    if (gu == 1 && gpt == 1) {
        gains_smem_ok(combine_bwd_kernel<1, 1, true, true>);
        unit = wave_blocks(combine_bwd_kernel<1, 1, true, true>, ntok, smem);
    } else if (gu == 1) {
        gains_smem_ok(combine_bwd_kernel<2, 1, true, true>);
        unit = wave_blocks(combine_bwd_kernel<2, 1, true, true>, ntok, smem);
    } else if (gpt == 1) {
        gains_smem_ok(combine_bwd_kernel<1, 2, true, true>);
        unit = wave_blocks(combine_bwd_kernel<1, 2, true, true>, ntok, smem);
    } else {
        gains_smem_ok(combine_bwd_kernel<2, 2, true, true>);
        unit = wave_blocks(combine_bwd_kernel<2, 2, true, true>, ntok, smem);
    }
    return std::max(with_gains, unit);
}

int check_combine(const logo_dims& d)
{
    if (d.B < 1 || d.T < 1 || d.Hq < 1) return LOGO_ERR_INVALID_ARG;
    if (d.D != 64 && d.D != 128) return LOGO_ERR_UNSUPPORTED;
    if (static_cast<int64_t>(d.B) * d.T > (1ll << 30)) return LOGO_ERR_UNSUPPORTED;
    if (d.Hq * (d.D / 8) > kMaxVec) return LOGO_ERR_UNSUPPORTED;  // Hq * D <= 16384
    return LOGO_OK;
}

}  // namespace

int combine_tu_status(int clear) { return read_tu_status(clear); }

}  // namespace logo

using namespace logo;

extern "C" int logo_combine(const logo_bf16* o_l, const logo_bf16* o_c, const float* gate_p, const uint8_t* z,
                            const int32_t* row_of, const float* gain_l, const float* gain_g, float eps,
                            logo_bf16* o, float* rstd_l, float* rstd_g, logo_dims dims, void* stream)
{
    int rc = check_combine(dims);
    if (rc != LOGO_OK) return rc;
    if (!o_l || !o_c || !gate_p || !z || !row_of || !o) return LOGO_ERR_INVALID_ARG;
    if (!(eps > 0.0f)) return LOGO_ERR_INVALID_ARG;
    if (!aligned16(o_l) || !aligned16(o_c) || !aligned16(o) || (gain_l && !aligned16(gain_l)) ||
        (gain_g && !aligned16(gain_g)))
        return LOGO_ERR_UNSUPPORTED;
    const int64_t ntok = static_cast<int64_t>(dims.B) * dims.T;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
#define LOGO_COMBINE_FWD(V, G, U)                                                                           \
    combine_fwd_kernel<V, G, U><<<static_cast<unsigned>(wave_blocks(combine_fwd_kernel<V, G, U>, ntok)), kThreads, \
                                  0, st>>>(o_l, o_c, gate_p, z, row_of, gain_l, gain_g, eps, o, rstd_l, rstd_g,      \
                                           ntok, dims.Hq, dims.D)
    const bool unit = !gain_l && !gain_g;
    const int g = group_vectors(dims, unit), gpt = groups_per_thread(dims, g);
    if (g == 2) {
        switch (gpt) {
            case 1: LOGO_COMBINE_FWD(1, 2, true); break;
            case 2: LOGO_COMBINE_FWD(2, 2, true); break;
            default: LOGO_COMBINE_FWD(4, 2, true); break;
        }
    } else if (unit) {  // fewer than 2 x kThreads vectors a token
        if (gpt == 1) { LOGO_COMBINE_FWD(1, 1, true); }
        else { LOGO_COMBINE_FWD(2, 1, true); }
    } else if (dims.Hq * (dims.D / 8) > kMaxVecGains) {  // Hq * D > 8192: more vectors a token than threads
        LOGO_COMBINE_FWD(8, 1, false);
    } else {
        auto run = [&](auto kernel, int slots) {
            const GainLaunch L = gain_launch(kernel, dims, slots);
            if (L.ok)
                kernel<<<static_cast<unsigned>(L.grid), L.sh.threads, L.smem, st>>>(
                    o_l, o_c, gate_p, z, row_of, gain_l, gain_g, eps, o, rstd_l, rstd_g, ntok, dims.Hq, L.sh.tpr,
                    L.sh.rows);
            return L.ok;
        };
        bool ok;
        constexpr int kSlots = 2 * GainCfg<512>::kRingFwd + 4;
        const bool big = gain_shape(dims).threads > 512;
        if (dims.D == 128) {
            ok = big ? run(combine_gained_fwd_kernel<128, 1024>, kSlots) : run(combine_gained_fwd_kernel<128, 512>, kSlots);
        } else {
            ok = big ? run(combine_gained_fwd_kernel<64, 1024>, kSlots) : run(combine_gained_fwd_kernel<64, 512>, kSlots);
        }
        if (!ok) return LOGO_ERR_CUDA;
    }
#undef LOGO_COMBINE_FWD
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}

namespace {
int combine_bwd_common(const logo_bf16* dO, const logo_bf16* o_l, const logo_bf16* o_c, const float* gate_p,
                       const uint8_t* z, const int32_t* row_of, const float* gain_l, const float* gain_g, float eps,
                       logo_bf16* dO_l, logo_bf16* dO_c, float* dgate_p, float* dgain_l, float* dgain_g,
                       void* workspace, size_t workspace_bytes, logo_dims dims, void* stream)
{
    int rc = check_combine(dims);
    if (rc != LOGO_OK) return rc;
    if (!dO || !o_l || !o_c || !gate_p || !z || !row_of || !dO_l || !dO_c || !dgate_p) return LOGO_ERR_INVALID_ARG;
    if (!(eps > 0.0f)) return LOGO_ERR_INVALID_ARG;
    if (!aligned16(dO) || !aligned16(o_l) || !aligned16(o_c) || !aligned16(dO_l) || !aligned16(dO_c) ||
        (gain_l && !aligned16(gain_l)) || (gain_g && !aligned16(gain_g)))
        return LOGO_ERR_UNSUPPORTED;
    const bool gains = dgain_l || dgain_g;
    const bool unit = !gain_l && !gain_g;
    const int g = group_vectors(dims, unit), gpt = groups_per_thread(dims, g);
    if (gains) {
        if (dims.Hq * (dims.D / 8) > kMaxVecGains) return LOGO_ERR_UNSUPPORTED;  // Hq * D <= 8192
        if (!workspace) return LOGO_ERR_INVALID_ARG;
        if (workspace_bytes < logo_combine_bwd_workspace_size(dims)) return LOGO_ERR_WORKSPACE;
        if (!aligned16(workspace)) return LOGO_ERR_WORKSPACE;  // the partial sums go there as float4
    }
    const int64_t ntok = static_cast<int64_t>(dims.B) * dims.T;
    const size_t smem = gains ? gains_smem(dims) : 0;
    unsigned grid = 0;
    float* part = static_cast<float*>(workspace);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
#define LOGO_COMBINE_BWD(V, NV, GN, U)                                                                          \
    if (GN && !gains_smem_ok(combine_bwd_kernel<V, NV, GN, U>)) return LOGO_ERR_CUDA;                             \
    grid = static_cast<unsigned>(wave_blocks(combine_bwd_kernel<V, NV, GN, U>, ntok, smem));                      \
    combine_bwd_kernel<V, NV, GN, U><<<grid, kThreads, smem, st>>>(dO, o_l, o_c, gate_p, z, row_of, gain_l, gain_g,   \
                                                                   eps, dO_l, dO_c, dgate_p, part, ntok, dims.Hq,    \
                                                                   dims.D)
    if (gains && unit) {
        if (g == 1 && gpt == 1) { LOGO_COMBINE_BWD(1, 1, true, true); }
        else if (g == 1) { LOGO_COMBINE_BWD(2, 1, true, true); }  // more than kThreads vectors a token
        else if (gpt == 1) { LOGO_COMBINE_BWD(1, 2, true, true); }
        else { LOGO_COMBINE_BWD(2, 2, true, true); }
    } else if (!unit && dims.Hq * (dims.D / 8) <= kMaxVecGains) {
        auto run = [&](auto kernel, int slots) {
            const GainLaunch L = gain_launch(kernel, dims, slots);
            if (!L.ok) return 0u;
            kernel<<<static_cast<unsigned>(L.grid), L.sh.threads, L.smem, st>>>(
                dO, o_l, o_c, gate_p, z, row_of, gain_l, gain_g, eps, dO_l, dO_c, dgate_p, part, ntok, dims.Hq,
                L.sh.tpr, L.sh.rows);
            return static_cast<unsigned>(L.grid);
        };
        grid = gains ? with_gained_bwd<true>(dims, run) : with_gained_bwd<false>(dims, run);
        if (grid == 0) return LOGO_ERR_CUDA;
    } else if (unit && g == 2) {
        switch (gpt) {
            case 1: LOGO_COMBINE_BWD(1, 2, false, true); break;
            case 2: LOGO_COMBINE_BWD(2, 2, false, true); break;
            default: LOGO_COMBINE_BWD(4, 2, false, true); break;
        }
    } else if (unit) {  // fewer than 2 x kThreads vectors a token
        if (gpt == 1) { LOGO_COMBINE_BWD(1, 1, false, true); }
        else { LOGO_COMBINE_BWD(2, 1, false, true); }
    } else {  // gains read, Hq * D > 8192
        LOGO_COMBINE_BWD(8, 1, false, false);
    }
#undef LOGO_COMBINE_BWD
    if (cudaGetLastError() != cudaSuccess) return LOGO_ERR_CUDA;
    if (gains) {
        const int hd = dims.Hq * dims.D;
        colsum_kernel<<<colsum_blocks(2 * hd), kColSumThreads, 0, st>>>(part, static_cast<int>(grid), 2 * hd, hd,
                                                                        dgain_l, dgain_g);
        if (cudaGetLastError() != cudaSuccess) return LOGO_ERR_CUDA;
    }
    return LOGO_OK;
}
}  // namespace

extern "C" int logo_combine_bwd(const logo_bf16* dO, const logo_bf16* o_l, const logo_bf16* o_c, const float* gate_p,
                                const uint8_t* z, const int32_t* row_of, const float* gain_l, const float* gain_g,
                                float eps, logo_bf16* dO_l, logo_bf16* dO_c, float* dgate_p, logo_dims dims,
                                void* stream)
{
    return combine_bwd_common(dO, o_l, o_c, gate_p, z, row_of, gain_l, gain_g, eps, dO_l, dO_c, dgate_p, nullptr,
                              nullptr, nullptr, 0, dims, stream);
}

extern "C" size_t logo_combine_bwd_workspace_size(logo_dims dims)
{
    if (check_combine(dims) != LOGO_OK) return 0;
    if (dims.Hq * (dims.D / 8) > kMaxVecGains) return 0;
    return static_cast<size_t>(gains_blocks(dims)) * 2 * static_cast<size_t>(dims.Hq) * dims.D * sizeof(float);
}

extern "C" int logo_combine_bwd_gains(const logo_bf16* dO, const logo_bf16* o_l, const logo_bf16* o_c,
                                      const float* gate_p, const uint8_t* z, const int32_t* row_of,
                                      const float* gain_l, const float* gain_g, float eps, logo_bf16* dO_l,
                                      logo_bf16* dO_c, float* dgate_p, float* dgain_l, float* dgain_g,
                                      logo_dims dims, void* workspace, size_t workspace_bytes, void* stream)
{
    if (!dgain_l && !dgain_g) return LOGO_ERR_INVALID_ARG;
    return combine_bwd_common(dO, o_l, o_c, gate_p, z, row_of, gain_l, gain_g, eps, dO_l, dO_c, dgate_p, dgain_l,
                              dgain_g, workspace, workspace_bytes, dims, stream);
}
