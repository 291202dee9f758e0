// transform.cu -- logo_branch_transform / _bwd: the per-head branch transforms
// of Eq. 5 that turn the local branch's Q/K/V into the global branch's,
//   LP: U^G_h = U^L_h A_h   (A_h a d x d matrix per head; the paper's default)
//   SO: U^G_h = U^L_h * s_h + b_h
// on either every row of a [B, T, H, d] tensor (K and V) or only the packed
// selected rows (Q: the global branch reads Q^G on those rows alone, so the
// transform of the other B*T - N rows is never computed).
//
// LP is a contraction of 2 d^2 FLOP per row and head against 4 d bytes moved:
// at d = 128 that is 64 FLOP/byte, more than the CUDA cores can keep up with
// at HBM speed, so it runs on the tensor cores: tcgen05 pipelines over 128-row
// tiles of a head beside that head's A_h in shared memory, one thread issuing
// the MMAs into two TMEM buffers, four warps draining them; tiles of every row
// come by TMA, tiles of the packed selected rows are gathered by four warps with
// cp.async.  The backward computes dU^L = dU^G A_h^T on the same tiles and
// accumulates dA_h = U^L^T dU^G; per-CTA partial dA are reduced in order by a
// second kernel (deterministic).  SO is elementwise; its per-block ds, db are summed by the
// fixed-order column sum of colsum.cuh (deterministic too).
#include <cuda_bf16.h>

#include <cstdint>

#include "colsum.cuh"
#include "attn_common.cuh"
#include "host_common.h"
#include "sm100.cuh"

namespace logo {
namespace {

// Row r of the listed set -> token index b*T + t (all rows: r itself).
struct RowSet {
    const int32_t* pos;    // packed positions, or NULL for every row
    const int32_t* cu_q;
    const int32_t* n_sel;  // device count of packed rows
    int B, T;
};

__device__ __forceinline__ int row_count(const RowSet& R)
{
    return R.pos ? *R.n_sel : R.B * R.T;
}

__device__ __forceinline__ int64_t row_token(const RowSet& R, int r)
{
    if (!R.pos) return r;
    const int b = seq_of_row(R.cu_q, R.B, r);
    return static_cast<int64_t>(b) * R.T + R.pos[r];
}

// out[h][e] = sum over c of part[h][c][e], e < per_head (a multiple of 4).
// Thread (x, g) of a block adds chunks g, g + 4, .. of four columns, then the
// four sums are added in order: a fixed order, and every load in flight.  `out`
// is the caller's and may lie on any 4-byte boundary.
__global__ void __launch_bounds__(256) reduce_parts_kernel(const float* __restrict__ part, int nchunk, int per_head,
                                                           int H, float* __restrict__ out)
{
    __shared__ float4 sh[4][64];
    const int x = threadIdx.x & 63, g = threadIdx.x >> 6;
    const int64_t e = (static_cast<int64_t>(blockIdx.x) * 64 + x) * 4;
    const bool have = e < static_cast<int64_t>(H) * per_head;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (have) {
        const int64_t h = e / per_head;
        const float* src = part + h * nchunk * per_head + e % per_head;
#pragma unroll 4
        for (int c = g; c < nchunk; c += 4) {
            const float4 v = *reinterpret_cast<const float4*>(src + static_cast<int64_t>(c) * per_head);
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
    }
    sh[g][x] = s;
    __syncthreads();
    if (g == 0 && have) {
#pragma unroll
        for (int k = 1; k < 4; ++k) {
            const float4 v = sh[k][x];
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
        if ((reinterpret_cast<uintptr_t>(out) & 15u) == 0) {
            *reinterpret_cast<float4*>(out + e) = s;
        } else {
            out[e] = s.x;
            out[e + 1] = s.y;
            out[e + 2] = s.z;
            out[e + 3] = s.w;
        }
    }
}

// SO forward: u_g = u_l * s + b on the listed rows; a thread per 8-element vector.
__global__ void __launch_bounds__(256) so_fwd_kernel(const logo_bf16* __restrict__ u_l, const float* __restrict__ s,
                                                     const float* __restrict__ b, RowSet R, int H, int D,
                                                     logo_bf16* __restrict__ u_g)
{
    const int nvec = H * D / 8;
    const int64_t total = static_cast<int64_t>(row_count(R)) * nvec;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < total;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int r = static_cast<int>(i / nvec), v = static_cast<int>(i % nvec);
        const int64_t off = row_token(R, r) * H * D + v * 8;
        const uint4 raw = *reinterpret_cast<const uint4*>(u_l + off);
        const __nv_bfloat162* x = reinterpret_cast<const __nv_bfloat162*>(&raw);
        uint4 o;
        uint32_t* ow = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 f = __bfloat1622float2(x[q]);
            const int e = v * 8 + 2 * q;
            ow[q] = pack_bf16x2(fmaf(f.x, s[e], b[e]), fmaf(f.y, s[e + 1], b[e + 1]));
        }
        *reinterpret_cast<uint4*>(u_g + off) = o;
    }
}

// SO backward: du_l (+)= du_g * s; ds += du_g * u_l, db += du_g.  A thread owns
// fixed vectors (VPT of them) of the [H, D] row for all rows of its block.
// part: [gridDim.x][2][H*D] float32 (ds, db).
template <int VPT>
__global__ void __launch_bounds__(256) so_bwd_kernel(const logo_bf16* __restrict__ u_l, const float* __restrict__ s,
                                                     const logo_bf16* __restrict__ du_g, RowSet R, int H, int D,
                                                     logo_bf16* __restrict__ du_l, int accumulate,
                                                     float* __restrict__ part)
{
    const int nvec = H * D / 8;
    float acc_s[VPT][8], acc_b[VPT][8];
#pragma unroll
    for (int k = 0; k < VPT; ++k)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc_s[k][i] = acc_b[k][i] = 0.f;
    const int n = row_count(R);
    for (int r = blockIdx.x; r < n; r += gridDim.x) {
        const int64_t base = row_token(R, r) * H * D;
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
            const int v = threadIdx.x + k * 256;
            if (v >= nvec) continue;
            const uint4 gu = *reinterpret_cast<const uint4*>(du_g + base + v * 8);
            const uint4 uu = *reinterpret_cast<const uint4*>(u_l + base + v * 8);
            const __nv_bfloat162* g2 = reinterpret_cast<const __nv_bfloat162*>(&gu);
            const __nv_bfloat162* u2 = reinterpret_cast<const __nv_bfloat162*>(&uu);
            uint4 prev = make_uint4(0u, 0u, 0u, 0u);
            if (accumulate) prev = *reinterpret_cast<const uint4*>(du_l + base + v * 8);
            const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&prev);
            uint4 o;
            uint32_t* ow = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 g = __bfloat1622float2(g2[q]), u = __bfloat1622float2(u2[q]);
                const int e = v * 8 + 2 * q;
                float x0 = g.x * s[e], x1 = g.y * s[e + 1];
                if (accumulate) {
                    const float2 pv = __bfloat1622float2(p2[q]);
                    x0 += pv.x;
                    x1 += pv.y;
                }
                ow[q] = pack_bf16x2(x0, x1);
                acc_s[k][2 * q] = fmaf(g.x, u.x, acc_s[k][2 * q]);
                acc_s[k][2 * q + 1] = fmaf(g.y, u.y, acc_s[k][2 * q + 1]);
                acc_b[k][2 * q] += g.x;
                acc_b[k][2 * q + 1] += g.y;
            }
            *reinterpret_cast<uint4*>(du_l + base + v * 8) = o;
        }
    }
    const int64_t hd = static_cast<int64_t>(H) * D;
#pragma unroll
    for (int k = 0; k < VPT; ++k) {
        const int v = threadIdx.x + k * 256;
        if (v >= nvec) continue;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            part[static_cast<int64_t>(blockIdx.x) * 2 * hd + v * 8 + i] = acc_s[k][i];
            part[static_cast<int64_t>(blockIdx.x) * 2 * hd + hd + v * 8 + i] = acc_b[k][i];
        }
    }
}

// ------------------------------------------------------------------------
// LP forward with tcgen05, on every row (K, V) or on the packed selected rows
// (Q): a tile is 128 rows of one head.  Roles: one warp (every row: TMA) or four
// (selected rows, gathered by cp.async one tile ahead) bring U tiles through a
// 2-deep ring, after A_h once; the next warp issues the MMAs (D[128 x D] =
// U_tile A_h into one of two TMEM buffers); four warps drain them (bf16).  A CTA
// keeps one head; the row tiles of that head are strided over gridDim.x CTAs.
// Shared memory: A_h as 64-column halves of [D rows][64] (128-byte swizzle), read
// as the MN-major B operand; U tiles as 64-column halves of [128 rows][64], the
// K-major A operand.  Memory bounds it on every row; on few selected rows the
// chain of dependent loads at a CTA's start (count, positions, rows) does:
// T 8192, an eighth of the rows of 32 heads of 128 (17 MB) 8.5 us (a kernel of
// mma.sync tiles of 64 rows took 10.2).
struct LpTcParams {
    CUtensorMap tm_u;   // u_l [B,T,H,D] as (d, h, t, b), box {64, 1, 128, 1}
    CUtensorMap tm_a;   // a [H*D rows][D] as (j, 1, row, 1), box {64, 1, D, 1}
    const logo_bf16* u_l;
    logo_bf16* u_g;
    RowSet rows;        // selected rows (GATHER)
    int B, T, H;
};

template <int D>
struct LpTcCfg {
    static constexpr int kHalfA = D * 128;                 // [D rows][64] bf16
    static constexpr int kABytes = (D / 64) * kHalfA;
    static constexpr int kHalfU = 128 * 128;               // [128 rows][64] bf16
    static constexpr int kUBytes = (D / 64) * kHalfU;
    static constexpr int kOffA = 0;
    static constexpr int kOffU = kABytes;                  // 2 stages
    static constexpr int kSmemBytes = kOffU + 2 * kUBytes + 1024;
    static constexpr uint32_t kTmemCols = D == 128 ? 256 : 128;  // two D-column result buffers
};

template <bool GATHER>
constexpr int kLpProducers = GATHER ? 4 : 1;  // warps

template <int D, bool GATHER>
__global__ void __launch_bounds__(32 * (kLpProducers<GATHER> + 5), 1) lp_tc_fwd_kernel(const __grid_constant__ LpTcParams p)
{
    using C = LpTcCfg<D>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t bar_a, bar_u_full[2], bar_u_empty[2], bar_t_full[2], bar_t_empty[2], bar_drain;
    __shared__ uint32_t tmem_sh;
    __shared__ volatile int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kMma = kLpProducers<GATHER>;  // the MMA issuer; the warps before it are producers
    const int h = blockIdx.y;
    const int tiles_per_seq = (p.T + 127) / 128;
    const int n = GATHER ? row_count(p.rows) : 0;  // packed rows
    const int ntiles = GATHER ? (n + 127) / 128 : p.B * tiles_per_seq;
    const uint32_t sA = smem_u32(smem + C::kOffA), sU = smem_u32(smem + C::kOffU);
    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(smem_u32(&bar_a), 1);
        mbar_init(smem_u32(&bar_drain), 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bar_u_full[s]), GATHER ? 128 : 1);
            mbar_init(smem_u32(&bar_u_empty[s]), 1);
            mbar_init(smem_u32(&bar_t_full[s]), 1);
            mbar_init(smem_u32(&bar_t_empty[s]), 128);
        }
        fence_mbar_init();
    }
    if (warp == kMma) {
        tmem_alloc(smem_u32(&tmem_sh), C::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    if (warp < kMma) {
        if (warp == 0 && lane == 0) {
            tma_prefetch_desc(&p.tm_a);
            mbar_arrive_expect_tx(smem_u32(&bar_a), C::kABytes);
            for (int s = 0; s < D / 64; ++s)
                tma_load_4d(sA + s * C::kHalfA, &p.tm_a, smem_u32(&bar_a), 64 * s, 0, h * D, 0, policy_evict_last());
        }
        bool ok = true;
        int k = 0;
        if (!GATHER) {
            // -------------------------------------------------------- producer (TMA)
            if (warp == 0 && lane == 0) {
                tma_prefetch_desc(&p.tm_u);
                const uint64_t pol_u = policy_evict_first();
                for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
                    const int st = k & 1;
                    if (!(ok = mbar_wait(smem_u32(&bar_u_empty[st]), ((k >> 1) & 1) ^ 1, &abort_flag))) break;
                    const int b = tile / tiles_per_seq, t0 = (tile % tiles_per_seq) * 128;
                    mbar_arrive_expect_tx(smem_u32(&bar_u_full[st]), C::kUBytes);
                    for (int s = 0; s < D / 64; ++s)
                        tma_load_4d(sU + st * C::kUBytes + s * C::kHalfU, &p.tm_u, smem_u32(&bar_u_full[st]), 64 * s, h,
                                    t0, b, pol_u);
                }
                if (!ok) {  // let the copies already issued land before the CTA exits
                    for (int j = k - 2 > 0 ? k - 2 : 0; j < k; ++j)
                        mbar_wait_drain(smem_u32(&bar_u_full[j & 1]), (j >> 1) & 1);
                }
            }
        } else {
            // -------------------------------------------------------- producers (gathered rows)
            // warp w copies rows 32w .. 32w + 31 of a tile, whole rows side by side in
            // a step; rows that do not exist are zero
            constexpr int kChunks = D / 8, kStep = 32 / kChunks;  // lanes a row, rows a step
            const int c = lane % kChunks;
            const logo_bf16* src = p.u_l + h * D + c * 8;
            for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
                const int st = k & 1;
                const int r = tile * 128 + warp * 32 + lane;
                const int64_t tok = r < n ? row_token(p.rows, r) : -1;
                ok = mbar_wait_warp(smem_u32(&bar_u_empty[st]), ((k >> 1) & 1) ^ 1, &abort_flag);
                if (!ok) break;
                const uint32_t base = sU + st * C::kUBytes + (c >> 3) * C::kHalfU;
#pragma unroll 8
                for (int i = 0; i < 32; i += kStep) {
                    const int row = i + lane / kChunks;
                    const int64_t t = __shfl_sync(0xffffffffu, tok, row);
                    const uint32_t dst = base + sw128_offset(warp * 32 + row, c & 7);
                    if (t >= 0) cp_async16(dst, src + t * p.H * D);
                    else st_shared_v4(dst, 0u, 0u, 0u, 0u);
                }
                cp_async_commit();
                if (k > 0) {  // tile k-1 has landed while tile k was issued
                    cp_async_wait<1>();
                    fence_proxy_async_smem();
                    mbar_arrive(smem_u32(&bar_u_full[st ^ 1]));
                }
            }
            cp_async_wait<0>();
            if (ok && k > 0) {
                fence_proxy_async_smem();
                mbar_arrive(smem_u32(&bar_u_full[(k - 1) & 1]));
            }
        }
        if (!ok && warp == 0 && lane == 0) mbar_wait_drain(smem_u32(&bar_a), 0);
    } else if (warp == kMma) {
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16_f32(128, D, false, true);
            bool ok = mbar_wait(smem_u32(&bar_a), 0, &abort_flag);
            int k = 0;
            for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x, ++k) {
                const int st = k & 1;
                if (!(ok = mbar_wait(smem_u32(&bar_u_full[st]), (k >> 1) & 1, &abort_flag))) break;
                if (!(ok = mbar_wait(smem_u32(&bar_t_empty[st]), ((k >> 1) & 1) ^ 1, &abort_flag))) break;
                tc_fence_after();
                const uint32_t ub = sU + st * C::kUBytes;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    const uint32_t ka = (ks >> 2) * C::kHalfU + (ks & 3) * 32;  // U: K-major halves of 64
                    umma_bf16_ss(tmem + st * D, sdesc_sw128(ub + ka, 16, 1024),
                                 sdesc_sw128(sA + ks * 2048, C::kHalfA, 1024), idesc, ks > 0 ? 1u : 0u);
                }
                umma_commit(smem_u32(&bar_u_empty[st]));
                umma_commit(smem_u32(&bar_t_full[st]));
            }
            if (!ok) {
                umma_commit(smem_u32(&bar_drain));
                mbar_wait_drain(smem_u32(&bar_drain), 0);
            }
        }
    } else {
        // epilogue: warp w reads TMEM lanes 32 (w % 4) .. (its rows of the tile)
        const int quad = warp & 3;
        const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
        int k = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
            const int st = k & 1;
            const bool ok = mbar_wait_warp(smem_u32(&bar_t_full[st]), (k >> 1) & 1, &abort_flag);
            if (!ok) break;
            tc_fence_after();
            // 16 x 256-bit pieces, four lanes trading bf16 pairs (quad_gather8): a warp
            // store is 8 rows of 64 contiguous bytes, not 32 rows of 16
            const int b = tile / tiles_per_seq, t0 = (tile % tiles_per_seq) * 128 + quad * 32;
            logo_bf16* dst = p.u_g + h * D + (lane & 3) * 8;
            logo_bf16* at[2][2];  // GATHER: this lane's rows t / 4, + 8, + 16, + 24 (null: no such row)
            if constexpr (GATHER) {
                const int r = tile * 128 + quad * 32 + lane;
                const int64_t tok = r < n ? row_token(p.rows, r) : -1;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int64_t t = __shfl_sync(0xffffffffu, tok, x * 8 + (lane >> 2));
                    at[x >> 1][x & 1] = t >= 0 ? dst + t * p.H * D : nullptr;
                }
            } else {
                dst += (static_cast<int64_t>(b) * p.T + t0) * p.H * D;
            }
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
                uint32_t v[2][16];
#pragma unroll
                for (int hf = 0; hf < 2; ++hf)
                    tmem_ld_16x256b_x4(tmem + lane_off + (static_cast<uint32_t>(hf * 16) << 16) + st * D + c * 32, v[hf]);
                tmem_wait_ld();
                if (c == D / 32 - 1) {
                    tc_fence_before();
                    mbar_arrive(smem_u32(&bar_t_empty[st]));
                }
#pragma unroll
                for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                    for (int ab = 0; ab < 2; ++ab) {
                        uint32_t w[4];
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4)
                            w[k4] = cvt_bf16x2(__uint_as_float(v[hf][4 * k4 + 2 * ab]),
                                               __uint_as_float(v[hf][4 * k4 + 2 * ab + 1]));
                        const uint4 o = quad_gather8(w, lane);
                        if constexpr (GATHER) {
                            if (at[hf][ab]) *reinterpret_cast<uint4*>(at[hf][ab] + c * 32) = o;
                        } else {
                            const int row = hf * 16 + ab * 8 + (lane >> 2);
                            if (t0 + row < p.T) *reinterpret_cast<uint4*>(dst + static_cast<int64_t>(row) * p.H * D + c * 32) = o;
                        }
                    }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMma) {
        tc_fence_after();
        tmem_dealloc(tmem, C::kTmemCols);
    }
}

template <int D, bool GATHER>
int launch_lp_tc_fwd(const logo_bf16* u_l, const logo_bf16* a, const RowSet& rows, const logo_dims& d, logo_bf16* u_g,
                     cudaStream_t st)
{
    LpTcParams prm{};
    if (!encode_bf16_4d(&prm.tm_u, u_l, D, d.Hq, d.T, d.B, 64, 128) ||
        !encode_bf16_4d(&prm.tm_a, a, D, 1, static_cast<uint64_t>(d.Hq) * D, 1, 64, D))
        return LOGO_ERR_CUDA;
    prm.u_l = u_l;
    prm.u_g = u_g;
    prm.rows = rows;
    prm.B = d.B;
    prm.T = d.T;
    prm.H = d.Hq;
    if (set_smem_limit(lp_tc_fwd_kernel<D, GATHER>, LpTcCfg<D>::kSmemBytes) != cudaSuccess) return LOGO_ERR_CUDA;
    const int ntiles = GATHER ? (d.B * d.T + 127) / 128 : d.B * ((d.T + 127) / 128);  // at most
    int per_head = (2 * device_sm_count()) / d.Hq;
    per_head = per_head < 1 ? 1 : (per_head > ntiles ? ntiles : per_head);
    lp_tc_fwd_kernel<D, GATHER><<<dim3(per_head, d.Hq), 32 * (kLpProducers<GATHER> + 5), LpTcCfg<D>::kSmemBytes, st>>>(prm);
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}

// LP backward with tcgen05, on every row (K, V) or on the packed selected rows
// (Q).  A tile is 128 rows of 128 columns: one head of d = 128, or two
// adjacent heads of d = 64 (a CTA keeps its heads and walks a strided share of
// the row tiles).  Per tile: dU = dG A_h^T (A_h read as the K-major B operand:
// its rows are the output dimension i, its columns the contracted j), per head,
// into one of two TMEM buffers, drained to du_l by the epilogue warps; and
// dA += U^T dG (both tiles read as MN-major operands: rows are the contracted
// dimension), accumulated in TMEM over all the CTA's tiles and written as its
// partial at the end (d = 64: the two 64 x 64 blocks on the diagonal; the
// cross products of the two heads cost nothing that is in short supply).
// Every row: tiles come by TMA.  Selected rows: four producer warps copy the
// rows, wherever their tokens are, into the same swizzled layout (cp.async, one
// tile ahead).  What dU is added to (accumulate) comes in the same way, as a
// third tile; an epilogue warp adds its rows in place (a row a lane), reads them
// back two whole rows a step and stores those.  (Reading and storing global
// memory from the accumulator's layout, even as 64-byte pieces, left the load
// latency and the lane exchange on the tile's path.)  With 3 tiles a stage only
// one CTA fits an SM; memory bounds it.  T8192 d128, dA's sum over the partials
// included: every row of 8 heads, added to dU (67 MB), 24 + 5 us when stored
// from the accumulator's layout, now 17.5 + 4.2; an eighth of the rows of 32
// heads (34 MB), 34 + 8 us with mma.sync tiles, now 15 + 5.6.
constexpr int kMaxChunks = 32;  // partial dA per head at most

struct LpBwdParams {
    CUtensorMap tm_u, tm_g, tm_a, tm_d;
    const logo_bf16* u_l;
    const logo_bf16* du_g;
    logo_bf16* du_l;
    float* part;  // [H][gridDim.x][D][D]
    RowSet rows;  // selected rows (GATHER)
    int B, T, H, accumulate;
};

template <int D>
struct LpBwdCfg {
    static constexpr int kHeads = 128 / D;           // heads per CTA
    static constexpr int kHalf = 128 * 128;          // [128 rows][64] bf16
    static constexpr int kTile = 2 * kHalf;          // 128 rows x 128 columns
    static constexpr int kHalfA = D * 128;           // [D rows][64] bf16
    static constexpr int kOffA = 0;
    static constexpr int kOffU = 2 * kHalfA;         // 2 stages of (U, G, dU)
    static constexpr int kStage = 3 * kTile;
    static constexpr int kSmemBytes = kOffU + 2 * kStage + 1024;
    static constexpr uint32_t kColDA = 256;          // dU buffers at 0 and 128
    static constexpr uint32_t kTmemCols = 512;
};
constexpr int kLpBwdThreads = 288;  // warps 0..3 producers (TMA: one thread), 4 MMA issuer, 5..8 epilogue

template <int D, bool GATHER>
__global__ void __launch_bounds__(kLpBwdThreads, 1) lp_tc_bwd_kernel(const __grid_constant__ LpBwdParams p)
{
    using C = LpBwdCfg<D>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t bar_a, bar_in_full[2], bar_in_empty[2], bar_t_full[2], bar_t_empty[2];
    __shared__ __align__(8) uint64_t bar_d_empty[2], bar_da, bar_drain;
    __shared__ uint32_t tmem_sh;
    __shared__ volatile int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int h0 = blockIdx.y * C::kHeads, heads = min(C::kHeads, p.H - h0);
    const int cols = heads * D;                      // columns that exist (64 at an odd last head of d = 64)
    const int row_elems = p.H * D;
    const int tiles_per_seq = (p.T + 127) / 128;
    const int n = GATHER ? row_count(p.rows) : 0;    // packed rows
    const int ntiles = GATHER ? (n + 127) / 128 : p.B * tiles_per_seq;
    const uint32_t sA = smem_u32(smem + C::kOffA), sIn = smem_u32(smem + C::kOffU);
    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(smem_u32(&bar_a), 1);
        mbar_init(smem_u32(&bar_da), 1);
        mbar_init(smem_u32(&bar_drain), 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bar_in_full[s]), GATHER ? 128 : 1);
            mbar_init(smem_u32(&bar_in_empty[s]), 1);
            mbar_init(smem_u32(&bar_t_full[s]), 1);
            mbar_init(smem_u32(&bar_t_empty[s]), 128);
            mbar_init(smem_u32(&bar_d_empty[s]), 128);
        }
        fence_mbar_init();
    }
    if (warp == 4) {
        tmem_alloc(smem_u32(&tmem_sh), C::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    if (warp < 4) {
        if (warp == 0 && lane == 0) {  // A_h of the CTA's heads, once
            tma_prefetch_desc(&p.tm_a);
            mbar_arrive_expect_tx(smem_u32(&bar_a), heads * D * D * 2);
            if (D == 128) {
                for (int s = 0; s < 2; ++s)
                    tma_load_4d(sA + s * C::kHalfA, &p.tm_a, smem_u32(&bar_a), 64 * s, 0, h0 * D, 0, policy_evict_last());
            } else {
                for (int s = 0; s < heads; ++s)
                    tma_load_4d(sA + s * C::kHalfA, &p.tm_a, smem_u32(&bar_a), 0, 0, (h0 + s) * D, 0, policy_evict_last());
            }
        }
        bool ok = true;
        if (!GATHER) {
            // -------------------------------------------------------- producer (TMA)
            if (warp == 0 && lane == 0) {
                tma_prefetch_desc(&p.tm_u);
                tma_prefetch_desc(&p.tm_g);
                const uint64_t pol = policy_evict_first();
                int k = 0;
                for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
                    const int st = k & 1;
                    if (!(ok = mbar_wait(smem_u32(&bar_in_empty[st]), ((k >> 1) & 1) ^ 1, &abort_flag))) break;
                    if (!(ok = mbar_wait(smem_u32(&bar_d_empty[st]), ((k >> 1) & 1) ^ 1, &abort_flag))) break;
                    const int b = tile / tiles_per_seq, t0 = (tile % tiles_per_seq) * 128;
                    const uint32_t bar = smem_u32(&bar_in_full[st]);
                    const uint32_t ub = sIn + st * C::kStage, gb = ub + C::kTile, db = gb + C::kTile;
                    // (a head past the last one of d = 64 reads as zeros)
                    mbar_arrive_expect_tx(bar, (p.accumulate ? 3 : 2) * C::kTile);
                    for (int s = 0; s < 2; ++s) {
                        const int c0 = D == 128 ? 64 * s : 0, hh = D == 128 ? h0 : h0 + s;
                        tma_load_4d(ub + s * C::kHalf, &p.tm_u, bar, c0, hh, t0, b, pol);
                        tma_load_4d(gb + s * C::kHalf, &p.tm_g, bar, c0, hh, t0, b, pol);
                        if (p.accumulate) tma_load_4d(db + s * C::kHalf, &p.tm_d, bar, c0, hh, t0, b, pol);
                    }
                }
                if (!ok) {
                    for (int j = k - 2 > 0 ? k - 2 : 0; j < k; ++j)
                        mbar_wait_drain(smem_u32(&bar_in_full[j & 1]), (j >> 1) & 1);
                }
            }
        } else {
            // -------------------------------------------------------- producers (gathered rows)
            // warp w copies rows 32w .. 32w + 31 of a tile: a row a step, lanes 0..15
            // its U, lanes 16..31 its G; rows and columns that do not exist are zero
            // (dU's rows, when added to, two a step)
            const logo_bf16* src = (lane < 16 ? p.u_l : p.du_g) + h0 * D + (lane & 15) * 8;
            const bool have = (lane & 15) * 8 < cols;
            int k = 0;
            for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
                const int st = k & 1;
                const int r = tile * 128 + warp * 32 + lane;
                const int tok = r < n ? static_cast<int>(row_token(p.rows, r)) : -1;
                ok = mbar_wait_warp(smem_u32(&bar_in_empty[st]), ((k >> 1) & 1) ^ 1, &abort_flag) &&
                     mbar_wait_warp(smem_u32(&bar_d_empty[st]), ((k >> 1) & 1) ^ 1, &abort_flag);
                if (!ok) break;
                const uint32_t half = sIn + st * C::kStage + ((lane & 15) >> 3) * C::kHalf;
                const uint32_t base = half + (lane < 16 ? 0 : C::kTile);
#pragma unroll 8
                for (int i = 0; i < 32; ++i) {
                    const int t = __shfl_sync(0xffffffffu, tok, i);
                    const uint32_t dst = base + sw128_offset(warp * 32 + i, lane & 7);
                    if (t >= 0 && have) cp_async16(dst, src + static_cast<int64_t>(t) * row_elems);
                    else st_shared_v4(dst, 0u, 0u, 0u, 0u);
                }
                if (p.accumulate) {
#pragma unroll 8
                    for (int i = 0; i < 16; ++i) {
                        const int row = 2 * i + (lane >> 4), t = __shfl_sync(0xffffffffu, tok, row);
                        if (t >= 0 && have)
                            cp_async16(half + 2 * C::kTile + sw128_offset(warp * 32 + row, lane & 7),
                                       p.du_l + static_cast<int64_t>(t) * row_elems + h0 * D + (lane & 15) * 8);
                    }
                }
                cp_async_commit();
                if (k > 0) {  // tile k-1 has landed while tile k was issued
                    cp_async_wait<1>();
                    fence_proxy_async_smem();
                    mbar_arrive(smem_u32(&bar_in_full[st ^ 1]));
                }
            }
            cp_async_wait<0>();
            if (ok && k > 0) {
                fence_proxy_async_smem();
                mbar_arrive(smem_u32(&bar_in_full[(k - 1) & 1]));
            }
        }
        if (!ok && warp == 0 && lane == 0) mbar_wait_drain(smem_u32(&bar_a), 0);
    } else if (warp == 4) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            constexpr uint32_t id_du = idesc_bf16_f32(128, D, false, false);  // G K-major x A_h K-major
            constexpr uint32_t id_da = idesc_bf16_f32(128, 128, true, true);  // U^T, G: both MN-major
            bool ok = mbar_wait(smem_u32(&bar_a), 0, &abort_flag);
            int k = 0;
            for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x, ++k) {
                const int st = k & 1;
                if (!(ok = mbar_wait(smem_u32(&bar_in_full[st]), (k >> 1) & 1, &abort_flag))) break;
                if (!(ok = mbar_wait(smem_u32(&bar_t_empty[st]), ((k >> 1) & 1) ^ 1, &abort_flag))) break;
                tc_fence_after();
                const uint32_t ub = sIn + st * C::kStage, gb = ub + C::kTile;
#pragma unroll
                for (int s = 0; s < C::kHeads; ++s)
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {  // contracted: j
                        const uint32_t half = ks >> 2, in = (ks & 3) * 32;
                        umma_bf16_ss(tmem + st * 128 + s * D, sdesc_sw128(gb + (s + half) * C::kHalf + in, 16, 1024),
                                     sdesc_sw128(sA + (s + half) * C::kHalfA + in, 16, 1024), id_du, ks > 0 ? 1u : 0u);
                    }
#pragma unroll
                for (int ks = 0; ks < 128 / 16; ++ks) {  // contracted: the tile's rows
                    umma_bf16_ss(tmem + C::kColDA, sdesc_sw128(ub + ks * 2048, C::kHalf, 1024),
                                 sdesc_sw128(gb + ks * 2048, C::kHalf, 1024), id_da, (k > 0 || ks > 0) ? 1u : 0u);
                }
                umma_commit(smem_u32(&bar_in_empty[st]));
                umma_commit(smem_u32(&bar_t_full[st]));
            }
            // dA complete (every MMA of this thread before the commit); also on a
            // CTA with no tile, so that the epilogue's final wait ends
            if (ok) umma_commit(smem_u32(&bar_da));
            if (!ok) {
                umma_commit(smem_u32(&bar_drain));
                mbar_wait_drain(smem_u32(&bar_drain), 0);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int quad = warp & 3;
        const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
        logo_bf16* out = p.du_l + h0 * D + (lane & 15) * 8;
        int k = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
            const int st = k & 1;
            const uint32_t db = sIn + st * C::kStage + 2 * C::kTile;
            // token of this lane's row (-1: no such row)
            int tok;
            if (GATHER) {
                const int r = tile * 128 + quad * 32 + lane;
                tok = r < n ? static_cast<int>(row_token(p.rows, r)) : -1;
            } else {
                const int b = tile / tiles_per_seq, t = (tile % tiles_per_seq) * 128 + quad * 32 + lane;
                tok = t < p.T ? b * p.T + t : -1;
            }
            // the tile's dU has landed (with U and G), and the product is there
            ok = mbar_wait_warp(smem_u32(&bar_in_full[st]), (k >> 1) & 1, &abort_flag) &&
                 mbar_wait_warp(smem_u32(&bar_t_full[st]), (k >> 1) & 1, &abort_flag);
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t v[32];
                tmem_ld32(tmem + lane_off + st * 128 + c * 32, v);
                tmem_wait_ld();
                if (c == 3) {
                    tc_fence_before();
                    mbar_arrive(smem_u32(&bar_t_empty[st]));
                }
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) {
                    const int chunk = c * 4 + q4;
                    const uint32_t at = db + (chunk >> 3) * C::kHalf + sw128_offset(quad * 32 + lane, chunk & 7);
                    float x[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = __uint_as_float(v[8 * q4 + e]);
                    if (p.accumulate) {
                        const uint4 old = ld_shared_v4(at);
                        const __nv_bfloat162* o2 = reinterpret_cast<const __nv_bfloat162*>(&old);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 f = __bfloat1622float2(o2[e]);
                            x[2 * e] += f.x;
                            x[2 * e + 1] += f.y;
                        }
                    }
                    st_shared_v4(at, cvt_bf16x2(x[0], x[1]), cvt_bf16x2(x[2], x[3]), cvt_bf16x2(x[4], x[5]),
                                 cvt_bf16x2(x[6], x[7]));
                }
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 16; ++i) {  // two whole rows (of this warp's) a store
                const int row = 2 * i + (lane >> 4), t = __shfl_sync(0xffffffffu, tok, row);
                const uint4 w = ld_shared_v4(db + ((lane & 15) >> 3) * C::kHalf + sw128_offset(quad * 32 + row, lane & 7));
                if (t >= 0 && (lane & 15) * 8 < cols)
                    *reinterpret_cast<uint4*>(out + static_cast<int64_t>(t) * row_elems) = w;
            }
            fence_proxy_async_smem();  // the stage's next copies come after these reads and writes
            mbar_arrive(smem_u32(&bar_d_empty[st]));
        }
        // the CTA's dA partial: lane r holds row i = r % D of head h0 + r / D
        const int r = quad * 32 + lane, s = r / D, i = r % D;
        float* pp = p.part + ((static_cast<int64_t>(h0 + s) * gridDim.x + blockIdx.x) * D + i) * D;
        if (ok && k == 0) {  // no tile: a zero partial
            if (s < heads)
                for (int j = 0; j < D; j += 4) *reinterpret_cast<float4*>(pp + j) = make_float4(0.f, 0.f, 0.f, 0.f);
        } else if (ok && mbar_wait_warp(smem_u32(&bar_da), 0, &abort_flag)) {
            tc_fence_after();
            const int first = (quad * 32 / D) * D;  // the head's columns (the same for the warp)
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
                uint32_t v[32];
                tmem_ld32(tmem + lane_off + C::kColDA + first + c * 32, v);
                tmem_wait_ld();
                if (s < heads) {
#pragma unroll
                    for (int e = 0; e < 32; e += 4)
                        *reinterpret_cast<float4*>(pp + c * 32 + e) =
                            make_float4(__uint_as_float(v[e]), __uint_as_float(v[e + 1]), __uint_as_float(v[e + 2]),
                                        __uint_as_float(v[e + 3]));
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4) {
        tc_fence_after();
        tmem_dealloc(tmem, C::kTmemCols);
    }
}

// CTAs a head (d = 64: a pair of heads) at most: one an SM.  As many partial dA
// a head are in the workspace.
int lp_bwd_chunks(const logo_dims& d)
{
    const int groups = d.D == 64 ? (d.Hq + 1) / 2 : d.Hq;
    const int per_group = device_sm_count() / groups;
    return per_group < 1 ? 1 : (per_group > kMaxChunks ? kMaxChunks : per_group);
}

template <int D, bool GATHER>
int launch_lp_tc_bwd(const logo_bf16* u_l, const logo_bf16* a, const logo_bf16* du_g, const RowSet& rows,
                     const logo_dims& d, logo_bf16* du_l, int accumulate, float* da, float* part, cudaStream_t st)
{
    using C = LpBwdCfg<D>;
    LpBwdParams prm{};
    if (!encode_bf16_4d(&prm.tm_u, u_l, D, d.Hq, d.T, d.B, 64, 128) ||
        !encode_bf16_4d(&prm.tm_g, du_g, D, d.Hq, d.T, d.B, 64, 128) ||
        !encode_bf16_4d(&prm.tm_d, du_l, D, d.Hq, d.T, d.B, 64, 128) ||
        !encode_bf16_4d(&prm.tm_a, a, D, 1, static_cast<uint64_t>(d.Hq) * D, 1, 64, D))
        return LOGO_ERR_CUDA;
    prm.u_l = u_l;
    prm.du_g = du_g;
    prm.du_l = du_l;
    prm.part = part;
    prm.rows = rows;
    prm.B = d.B;
    prm.T = d.T;
    prm.H = d.Hq;
    prm.accumulate = accumulate;
    if (set_smem_limit(lp_tc_bwd_kernel<D, GATHER>, C::kSmemBytes) != cudaSuccess) return LOGO_ERR_CUDA;
    // selected rows: the tiles are not known here, every row is the most
    const int groups = (d.Hq + C::kHeads - 1) / C::kHeads;
    const int ntiles = GATHER ? (d.B * d.T + 127) / 128 : d.B * ((d.T + 127) / 128);
    int per_group = lp_bwd_chunks(d);
    per_group = per_group > ntiles ? ntiles : per_group;
    const int rounds = (ntiles + per_group - 1) / per_group;
    per_group = (ntiles + rounds - 1) / rounds;  // the fewest partial dA for as many rounds
    lp_tc_bwd_kernel<D, GATHER><<<dim3(per_group, groups), kLpBwdThreads, C::kSmemBytes, st>>>(prm);
    if (cudaGetLastError() != cudaSuccess) return LOGO_ERR_CUDA;
    const int64_t vecs = static_cast<int64_t>(d.Hq) * D * D / 4;
    reduce_parts_kernel<<<static_cast<unsigned>((vecs + 63) / 64), 256, 0, st>>>(part, per_group, D * D, d.Hq, da);
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}

int so_vpt(const logo_dims& d)
{
    const int nvec = d.Hq * d.D / 8;
    const int need = (nvec + 255) / 256;
    return need <= 1 ? 1 : need <= 2 ? 2 : 4;
}

int so_bwd_blocks(const logo_dims& d)
{
    const int64_t rows = static_cast<int64_t>(d.B) * d.T;
    const int64_t cap = static_cast<int64_t>(device_sm_count()) * 4;
    return static_cast<int>(rows < cap ? rows : cap);
}

// Every row: no row depends on where its sequence begins, so the batch is taken as
// one sequence and a 128-row tile goes on across the ends (a tile a sequence at
// least: 600 sequences of 10 rows, 16 heads of 64, forward and backward
// 25.8 -> 6.6 and 47.5 -> 12.8 us).
void every_row(logo_dims* d)
{
    d->T *= d->B;
    d->B = 1;
}

int check_transform(const logo_dims& d, const void* u, const void* out)
{
    if (d.B < 1 || d.T < 1 || d.Hq < 1) return LOGO_ERR_INVALID_ARG;
    if (d.D != 64 && d.D != 128) return LOGO_ERR_UNSUPPORTED;
    if (static_cast<int64_t>(d.B) * d.T > (1ll << 30)) return LOGO_ERR_UNSUPPORTED;
    if (d.Hq * d.D > 8192) return LOGO_ERR_UNSUPPORTED;
    if (!aligned16(u) || !aligned16(out)) return LOGO_ERR_UNSUPPORTED;
    return LOGO_OK;
}

}  // namespace
int transform_tu_status(int clear) { return read_tu_status(clear); }

}  // namespace logo

using namespace logo;

extern "C" int logo_branch_transform(const logo_bf16* u_l, const logo_bf16* a_lp, const float* s_so,
                                     const float* b_so, const int32_t* pos, const int32_t* cu_q,
                                     const int32_t* n_sel_total, logo_bf16* u_g, logo_dims dims, void* stream)
{
    int rc = check_transform(dims, u_l, u_g);
    if (rc != LOGO_OK) return rc;
    if (!u_l || !u_g) return LOGO_ERR_INVALID_ARG;
    if ((a_lp != nullptr) == (s_so != nullptr || b_so != nullptr)) return LOGO_ERR_INVALID_ARG;  // exactly one form
    if (!a_lp && (!s_so || !b_so)) return LOGO_ERR_INVALID_ARG;
    if (pos && (!cu_q || !n_sel_total)) return LOGO_ERR_INVALID_ARG;
    if (a_lp && !aligned16(a_lp)) return LOGO_ERR_UNSUPPORTED;
    if (!pos) every_row(&dims);
    const RowSet R{pos, cu_q, n_sel_total, dims.B, dims.T};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (a_lp && !pos) {
        return dims.D == 128 ? launch_lp_tc_fwd<128, false>(u_l, a_lp, R, dims, u_g, st)
                             : launch_lp_tc_fwd<64, false>(u_l, a_lp, R, dims, u_g, st);
    }
    if (a_lp) {  // the packed selected rows (Q)
        return dims.D == 128 ? launch_lp_tc_fwd<128, true>(u_l, a_lp, R, dims, u_g, st)
                             : launch_lp_tc_fwd<64, true>(u_l, a_lp, R, dims, u_g, st);
    }
    const int64_t work = static_cast<int64_t>(dims.B) * dims.T * dims.Hq * dims.D / 8;
    const int64_t cap = static_cast<int64_t>(device_sm_count()) * 8;
    const int64_t blocks = (work + 255) / 256;
    so_fwd_kernel<<<static_cast<unsigned>(blocks < cap ? blocks : cap), 256, 0, st>>>(u_l, s_so, b_so, R, dims.Hq,
                                                                                       dims.D, u_g);
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}

extern "C" size_t logo_branch_transform_bwd_workspace_size(logo_dims dims)
{
    if (dims.B < 1 || dims.T < 1 || dims.Hq < 1 || (dims.D != 64 && dims.D != 128) || dims.Hq * dims.D > 8192)
        return 0;
    const size_t lp = static_cast<size_t>(dims.Hq) * lp_bwd_chunks(dims) * dims.D * dims.D * sizeof(float);
    const size_t so = static_cast<size_t>(so_bwd_blocks(dims)) * 2 * dims.Hq * dims.D * sizeof(float);
    return lp > so ? lp : so;
}

extern "C" int logo_branch_transform_bwd(const logo_bf16* u_l, const logo_bf16* a_lp, const float* s_so,
                                         const int32_t* pos, const int32_t* cu_q, const int32_t* n_sel_total,
                                         const logo_bf16* du_g, logo_bf16* du_l, int accumulate, float* da_lp,
                                         float* ds_so, float* db_so, logo_dims dims, void* workspace,
                                         size_t workspace_bytes, void* stream)
{
    int rc = check_transform(dims, u_l, du_l);
    if (rc != LOGO_OK) return rc;
    if (!u_l || !du_g || !du_l) return LOGO_ERR_INVALID_ARG;
    if ((a_lp != nullptr) == (s_so != nullptr)) return LOGO_ERR_INVALID_ARG;  // exactly one form
    if (a_lp && !da_lp) return LOGO_ERR_INVALID_ARG;
    if (accumulate != 0 && accumulate != 1) return LOGO_ERR_INVALID_ARG;
    if (pos && (!cu_q || !n_sel_total)) return LOGO_ERR_INVALID_ARG;
    if (!aligned16(du_g) || (a_lp && !aligned16(a_lp))) return LOGO_ERR_UNSUPPORTED;
    if (!workspace || workspace_bytes < logo_branch_transform_bwd_workspace_size(dims)) return LOGO_ERR_WORKSPACE;
    if (a_lp && !aligned16(workspace)) return LOGO_ERR_WORKSPACE;  // the partial dA go there as float4
    if (!pos) every_row(&dims);
    const RowSet R{pos, cu_q, n_sel_total, dims.B, dims.T};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    float* part = static_cast<float*>(workspace);
    if (a_lp && dims.D == 128)
        return pos ? launch_lp_tc_bwd<128, true>(u_l, a_lp, du_g, R, dims, du_l, accumulate, da_lp, part, st)
                   : launch_lp_tc_bwd<128, false>(u_l, a_lp, du_g, R, dims, du_l, accumulate, da_lp, part, st);
    if (a_lp)
        return pos ? launch_lp_tc_bwd<64, true>(u_l, a_lp, du_g, R, dims, du_l, accumulate, da_lp, part, st)
                   : launch_lp_tc_bwd<64, false>(u_l, a_lp, du_g, R, dims, du_l, accumulate, da_lp, part, st);
    const int grid = so_bwd_blocks(dims);
    switch (so_vpt(dims)) {
        case 1: so_bwd_kernel<1><<<grid, 256, 0, st>>>(u_l, s_so, du_g, R, dims.Hq, dims.D, du_l, accumulate, part); break;
        case 2: so_bwd_kernel<2><<<grid, 256, 0, st>>>(u_l, s_so, du_g, R, dims.Hq, dims.D, du_l, accumulate, part); break;
        default: so_bwd_kernel<4><<<grid, 256, 0, st>>>(u_l, s_so, du_g, R, dims.Hq, dims.D, du_l, accumulate, part); break;
    }
    if (cudaGetLastError() != cudaSuccess) return LOGO_ERR_CUDA;
    const int hd = dims.Hq * dims.D;
    colsum_kernel<<<colsum_blocks(2 * hd), kColSumThreads, 0, st>>>(part, grid, 2 * hd, hd, ds_so, db_so);
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}
