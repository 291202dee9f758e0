// attn_bwd.cu -- backward of both attention branches on tcgen05 tensor cores.
//
//   logo_local_attn_bwd          gradients of Eq. 6 (window W, every token)
//   logo_global_sparse_attn_bwd  row-sparse gradients of Eq. 8 (Sec. 3.3, App. B)
//
// With P = softmax(scale * Q K^T) over the visible keys, dO the upstream
// gradient and Dsum = rowsum(dO * O):
//   dV = P^T dO,  dP = dO V^T,  dS = P * (dP - Dsum),
//   dQ = scale * dS K,  dK = scale * dS^T Q.
// Both kernels are persistent and KV-block-major: a work item is one block of
// 128 keys of one KV head of one sequence, and it walks every (query head of
// the KV head's group) x (query tile that can see the block).  dK and dV stay
// in TMEM for the whole item (one CTA owns the block for every query head of
// its group, so they need no atomics); dQ is reduced across items in fp32.
// Five MMAs per (query tile, KV block), the minimum: the paper's separate dQ
// and dK/dV kernels recompute S and dP and take seven.
//
// d = 128, attn_bwd2_kernel (16 warps, query tiles of 64 rows):
//   warp 0       TMA: K/V once per item, Q/dO tiles through a 4-deep ring
//   warp 1       MMA issuer A: S^T = K Q^T, dP^T = V dO^T (M = 128 keys,
//                N = 64 queries) into one TMEM buffer that the softmax warps
//                release as soon as they have loaded it
//   warps 2..9   two warpgroups, one per 32-query half of the tile; thread =
//                key row: P^T (back to TMEM as bf16 pairs, two buffers) and
//                dS^T (bf16, to shared memory, two buffers)
//   warp 15      MMA issuer B: dV += P^T dO (P^T as the TMEM operand),
//                dK += dS^T Q, dQ^T = K^T dS^T into a TMEM buffer of its own
//   warps 10..13 dQ^T out of TMEM (thread = head-dim row), coalesced fp32
//                reductions into the dQ accumulator (one 128-byte row segment
//                per warp instruction), converted to bf16 by a pass after the
//                kernel; dK/dV epilogue at the end of each item
//   warp 14      global branch: zero rows of the dense dQ for unselected tokens
// Global query tiles are 64-row slices of the packed selected rows, starting
// at the first packed row whose position reaches the block, read from a table
// the pre-pass builds once per call (App. B's precomputed search); the same
// pre-pass gathers the selected Q rows and computes Dsum.
//
// d = 64, attn_bwd64_kernel (16 warps, query tiles of 128 rows): the same
// split of the work over two MMA issuers, two softmax-backward warpgroups and
// a drain warpgroup, laid out for 64-wide rows (below).
#include <cuda_bf16.h>

#include <cstdint>
#include <type_traits>

#include "attn_common.cuh"
#include "host_common.h"
#include "sm100.cuh"

namespace logo {
namespace {

struct BwdParams {
    CUtensorMap tm_q;   // local: Q [B,T,Hq,D]; global: packed [1,cap+128,Hq,D]
    CUtensorMap tm_do;  // same layout as tm_q
    CUtensorMap tm_k;   // [B,T,Hkv,D]
    CUtensorMap tm_v;
    CUtensorMap tm_dq;  // d = 64: dq_acc, for the bulk reductions
    const float* lse;   // d = 128: local [B,Hq,T]; global [Hq,cap]
    const float* dsum;  // same layout as lse
    const float4* stats;  // d = 64: local [B,Hq][stat_rows / 2], global [Hq][stat_rows / 2] (RowStats)
    const float4* stats0; // d = 64, local: zeros, for the rows of a tile past the sequence's end
    const int32_t* pos_c; // d = 64, global: pos, on a 16-byte boundary
    int64_t stat_rows;
    float* dq_acc;      // local [B,T,Hq,D]; global [cap+128,Hq,D]
    logo_bf16* dk;      // [B,T,Hkv,D]
    logo_bf16* dv;
    const int32_t* pos;
    const int32_t* cu_q;
    const int32_t* first_row;  // global: [B, nblk] first packed row of sequence b whose position reaches block j
    logo_bf16* dq_fill;        // global: dense dQ [B, T, Hq, D] whose unselected rows this kernel zeroes
    int B, T, Hq, Hkv, window, cap, nblk;
    float scale, scale_log2;
};

struct BwdItem {
    int b, j, kvh;
    int i_lo, ntiles;   // query tiles visited: i_lo .. i_lo + ntiles - 1
    int row_lo, row_hi; // global: packed rows of sequence b
};

// BQ: query rows per tile
template <int BQ, bool GLOBAL>
__device__ __forceinline__ BwdItem decode_bwd2(const BwdParams& p, int k)
{
    BwdItem it;
    it.kvh = k % p.Hkv;
    const int t = k / p.Hkv;
    it.b = t % p.B;
    it.j = t / p.B;
    const int k0 = it.j * kBN;
    if (!GLOBAL) {
        it.i_lo = k0 / BQ;
        const int i_hi = min((p.T + BQ - 1) / BQ - 1, (k0 + kBN - 1 + p.window - 1) / BQ);
        it.ntiles = i_hi - it.i_lo + 1;
        it.row_lo = it.row_hi = 0;
    } else {
        it.row_lo = p.cu_q[it.b];
        it.row_hi = p.cu_q[it.b + 1];
        const int lo = p.first_row[it.b * p.nblk + it.j];  // precomputed search (App. B)
        if (lo >= it.row_hi) {
            it.i_lo = 0;
            it.ntiles = 0;
        } else {
            it.i_lo = lo / BQ;
            it.ntiles = (it.row_hi - 1) / BQ - it.i_lo + 1;
        }
    }
    return it;
}

// One warp of each CTA: zero the dense dQ rows of the tokens that were not
// selected (the conversion after the kernel writes only the selected rows).
// The backward kernels leave nearly all of HBM's bandwidth idle; a separate
// pass writing the whole dense tensor would not.
__device__ __forceinline__ void zero_unselected_dq(const BwdParams& p, int D, int lane)
{
    const int64_t ntok = static_cast<int64_t>(p.B) * p.T;
    const int64_t per = (ntok + gridDim.x - 1) / gridDim.x;
    const int64_t t_begin = static_cast<int64_t>(blockIdx.x) * per;
    const int64_t t_end = t_begin + per < ntok ? t_begin + per : ntok;
    const int row_vecs = p.Hq * D / 8;  // 16-byte vectors per token row
    int cur_b = -1, r = 0, r_hi = 0;
    for (int64_t bt = t_begin; bt < t_end; ++bt) {
        const int b = static_cast<int>(bt / p.T), t = static_cast<int>(bt % p.T);
        if (b != cur_b) {  // first packed row of sequence b at or after position t
            cur_b = b;
            int lo = p.cu_q[b], hi = p.cu_q[b + 1];
            r_hi = hi;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (p.pos[mid] < t) lo = mid + 1;
                else hi = mid;
            }
            r = lo;
        }
        if (r < r_hi && p.pos[r] == t) {  // selected: converted later
            ++r;
            continue;
        }
        uint4* dst = reinterpret_cast<uint4*>(p.dq_fill + bt * p.Hq * D);
        for (int v = lane; v < row_vecs; v += 32) dst[v] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// ---------------------------------------------------------------- d = 128
// Overlapped variant for D = 128: query tiles of 64 rows.  S^T and dP^T of a
// tile share one TMEM buffer that the softmax warps release as soon as they
// have loaded it, so the MMAs of tile u+1 run while the softmax works on tile
// u.  P^T goes back to TMEM (two buffers; dV reads it as the TMEM operand),
// dS^T to shared memory (two buffers; dK and dQ^T read it), and dQ is produced
// transposed (dQ^T = K^T dS^T, one TMEM lane per head-dim row).  Roles:
//   warp 0       TMA: K/V per item, Q/dO tiles through a 4-deep ring
//   warp 1       MMA issuer A: S^T, dP^T (M=128 keys, N=64 queries)
//   warp 15      MMA issuer B: once P^T/dS^T of a tile are in shared memory,
//                dV += P^T dO, dK += dS^T Q, dQ^T = K^T dS^T
//   warps 2..9   two warpgroups, one per 32-query half of the tile; thread =
//                key row: P^T and dS^T (bf16) from S^T and dP^T
//   warps 10..13 dQ^T out of TMEM (thread = head-dim row), coalesced fp32
//                atomics into the dQ accumulator (one 128-byte row segment per
//                warp instruction); dK/dV epilogue at the end of each item
//   warp 14      global branch: zero rows of the dense dQ for unselected tokens
// Shared memory's bandwidth bounds it where items are long.  In a tile the MMAs
// read 192 KB (an N = 64 product reads its whole 4 KB A step: 48 clocks by itself,
// 64 for N = 128), the copies write 32, dS^T 16, the statistics 16, and the
// reductions move 32 through L1: 2300 clocks at 128 bytes each, beside barriers
// and the items' K, V, dK and dV.  16K, window 1024: 2590 clocks of the kernel's
// time a tile, of which ncu counts 2570 as data-bank cycles (99%; the global call
// at 16K 100%).  At 4K, with 9 (local) and 4.5 (global) tiles an item, they are
// busy 83% and 72%: the item switches.  Tiles of 128 rows move a sixth less, but
// leave no TMEM for anything to overlap (5250 clocks and more).
struct Bwd2Cfg {
    static constexpr int D = 128;
    static constexpr int kBQ = 64;                 // queries per tile
    static constexpr int kStages = 4;              // Q/dO ring depth
    static constexpr int kKVBytes = kBN * D * 2;   // K or V block: 32 KB
    static constexpr int kQBytes = kBQ * D * 2;    // Q or dO tile: 16 KB (two 8 KB halves of d)
    static constexpr int kPBytes = kBN * kBQ * 2;  // dS^T: 16 KB
    static constexpr int kOffK = 0;
    static constexpr int kOffV = kOffK + kKVBytes;
    static constexpr int kOffQ = kOffV + kKVBytes;
    static constexpr int kOffDO = kOffQ + kStages * kQBytes;
    static constexpr int kOffDS = kOffDO + kStages * kQBytes;  // 2 buffers
    static constexpr int kSmemBytes = kOffDS + 2 * kPBytes + 1024;
    static constexpr uint32_t kColDK = 0;
    static constexpr uint32_t kColDV = 128;
    static constexpr uint32_t kColS = 256;    // S^T (64 cols), dP^T at +64
    static constexpr uint32_t kColDQ = 384;   // dQ^T (64 cols)
    static constexpr uint32_t kColP = 448;    // P^T buffer b (bf16 pairs) at 448 + 32b
    static constexpr uint32_t kTmemCols = 512;
    static constexpr int kThreads = 512;
};

template <bool GLOBAL>
__global__ void __launch_bounds__(Bwd2Cfg::kThreads, 1) attn_bwd2_kernel(const __grid_constant__ BwdParams p)
{
    using C = Bwd2Cfg;
    constexpr int D = C::D, BQ = C::kBQ, NS = C::kStages;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t bar_kv_full, bar_kv_empty, bar_dkv_full, bar_dkv_empty, bar_drain, bar_stage;
    __shared__ __align__(8) uint64_t bar_drain_b;
    __shared__ __align__(8) uint64_t bar_qdo_full[NS], bar_qdo_empty[NS];
    __shared__ __align__(8) uint64_t bar_st_full, bar_st_empty;
    __shared__ __align__(8) uint64_t bar_ds_full[2], bar_dq_full[2], bar_dq_empty[2];
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_flag;
    __shared__ int sh_pos[2][BQ];
    // per pair of query columns (2c, 2c+1): (-lse_2c, -lse_2c+1, -Dsum_2c, -Dsum_2c+1), lse in log2 units
    __shared__ float4 sh_pair[2][BQ / 2];
    __shared__ int sh_open[2][2];       // per staging warp: every column sees every key of the block

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sK = smem_u32(smem + C::kOffK), sV = smem_u32(smem + C::kOffV);
    const uint32_t sQ = smem_u32(smem + C::kOffQ), sDO = smem_u32(smem + C::kOffDO);
    const uint32_t sDS = smem_u32(smem + C::kOffDS);
    const int group = p.Hq / p.Hkv;
    const int n_items = p.B * p.nblk * p.Hkv;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(smem_u32(&bar_kv_full), 1);
        mbar_init(smem_u32(&bar_kv_empty), 1);
        mbar_init(smem_u32(&bar_dkv_full), 1);
        mbar_init(smem_u32(&bar_dkv_empty), 128);
        mbar_init(smem_u32(&bar_drain), 1);
        mbar_init(smem_u32(&bar_drain_b), 1);
        mbar_init(smem_u32(&bar_stage), 256);
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&bar_qdo_full[s]), 1);
            mbar_init(smem_u32(&bar_qdo_empty[s]), 1);
        }
        mbar_init(smem_u32(&bar_st_full), 1);
        mbar_init(smem_u32(&bar_st_empty), 256);
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&bar_ds_full[b]), 256);
            mbar_init(smem_u32(&bar_dq_full[b]), 1);
            mbar_init(smem_u32(&bar_dq_empty[b]), 128);
        }
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&tmem_base_sh), C::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            tma_prefetch_desc(&p.tm_q);
            tma_prefetch_desc(&p.tm_do);
            tma_prefetch_desc(&p.tm_k);
            tma_prefetch_desc(&p.tm_v);
            const uint64_t pol_q = policy_evict_last();
            const uint64_t pol_kv = policy_evict_first();
            int u = 0, kv_items = 0;
            bool ok = true;
            for (int k = blockIdx.x; k < n_items && ok; k += gridDim.x) {
                const BwdItem it = decode_bwd2<BQ, GLOBAL>(p, k);
                if (it.ntiles == 0) continue;
                if (!(ok = mbar_wait(smem_u32(&bar_kv_empty), (kv_items & 1) ^ 1, &abort_flag))) break;
                const uint32_t kvb = smem_u32(&bar_kv_full);
                mbar_arrive_expect_tx(kvb, 2 * C::kKVBytes);
                for (int s = 0; s < 2; ++s) {
                    tma_load_4d(sK + s * 16384, &p.tm_k, kvb, 64 * s, it.kvh, it.j * kBN, it.b, pol_kv);
                    tma_load_4d(sV + s * 16384, &p.tm_v, kvb, 64 * s, it.kvh, it.j * kBN, it.b, pol_kv);
                }
                ++kv_items;
                const int n_it = group * it.ntiles;
                for (int x = 0; x < n_it; ++x, ++u) {
                    const int h = it.kvh * group + x / it.ntiles;
                    const int i = it.i_lo + x % it.ntiles;
                    const int st = u % NS, f = u / NS;
                    if (!(ok = mbar_wait(smem_u32(&bar_qdo_empty[st]), (f & 1) ^ 1, &abort_flag))) break;
                    const uint32_t qb = smem_u32(&bar_qdo_full[st]);
                    mbar_arrive_expect_tx(qb, 2 * C::kQBytes);
                    const int cb = GLOBAL ? 0 : it.b;
                    for (int s = 0; s < 2; ++s) {
                        tma_load_4d(sQ + st * C::kQBytes + s * 8192, &p.tm_q, qb, 64 * s, h, i * BQ, cb, pol_q);
                        tma_load_4d(sDO + st * C::kQBytes + s * 8192, &p.tm_do, qb, 64 * s, h, i * BQ, cb, pol_q);
                    }
                }
            }
            if (!ok) {  // let copies already issued land before the CTA exits
                if (kv_items > 0) mbar_wait_drain(smem_u32(&bar_kv_full), (kv_items - 1) & 1);
                for (int v = u - NS > 0 ? u - NS : 0; v < u; ++v)
                    mbar_wait_drain(smem_u32(&bar_qdo_full[v % NS]), (v / NS) & 1);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer A: S^T, dP^T
        // The tile's second half (dV, dK, dQ^T) comes from warp 15: two issuing
        // threads keep the tensor pipe fed while either waits for its inputs
        // (the issue queue is short, so one thread that stops to wait starves it).
        if (lane == 0) {
            constexpr uint32_t idS = idesc_bf16_f32(kBN, BQ, false, false);  // S^T, dP^T: 128 x 64
            int u = 0, kv_items = 0;
            bool ok = true;
            for (int k = blockIdx.x; k < n_items && ok; k += gridDim.x) {
                const BwdItem it = decode_bwd2<BQ, GLOBAL>(p, k);
                if (it.ntiles == 0) continue;
                if (!(ok = mbar_wait(smem_u32(&bar_kv_full), kv_items & 1, &abort_flag))) break;
                const int n_it = group * it.ntiles;
                for (int x = 0; x < n_it; ++x, ++u) {
                    const int st = u % NS;
                    if (!(ok = mbar_wait(smem_u32(&bar_qdo_full[st]), (u / NS) & 1, &abort_flag))) break;
                    // the softmax warps have loaded S^T, dP^T of tile u-1
                    if (!(ok = mbar_wait(smem_u32(&bar_st_empty), (u & 1) ^ 1, &abort_flag))) break;
                    tc_fence_after();
                    const uint32_t qb = sQ + st * C::kQBytes, ob = sDO + st * C::kQBytes;
                    const uint32_t scol = tmem + C::kColS;
                    // S^T and dP^T k-steps alternate (two accumulators, both
                    // needed before the softmax can start)
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        const uint32_t ka = (ks >> 2) * 16384 + (ks & 3) * 32;
                        const uint32_t kb = (ks >> 2) * 8192 + (ks & 3) * 32;
                        umma_bf16_ss(scol, sdesc_sw128(sK + ka, 16, 1024), sdesc_sw128(qb + kb, 16, 1024), idS,
                                     ks > 0 ? 1u : 0u);
                        umma_bf16_ss(scol + 64, sdesc_sw128(sV + ka, 16, 1024), sdesc_sw128(ob + kb, 16, 1024), idS,
                                     ks > 0 ? 1u : 0u);
                    }
                    umma_commit(smem_u32(&bar_st_full));
                }
                if (!ok) break;
                ++kv_items;
            }
            if (!ok) {
                umma_commit(smem_u32(&bar_drain));
                mbar_wait_drain(smem_u32(&bar_drain), 0);
            }
        }
    } else if (warp == 15) {
        // ------------------------------------------------------------ MMA issuer B: dV, dK, dQ^T
        if (lane == 0) {
            constexpr uint32_t idKV = idesc_bf16_f32(kBN, D, false, true);  // dV, dK: 128 x 128
            constexpr uint32_t idQ = idesc_bf16_f32(D, BQ, true, true);     // dQ^T: 128 x 64
            int u = 0, kv_items = 0;
            bool ok = true;
            for (int k = blockIdx.x; k < n_items && ok; k += gridDim.x) {
                const BwdItem it = decode_bwd2<BQ, GLOBAL>(p, k);
                if (it.ntiles == 0) continue;
                const int n_it = group * it.ntiles;
                for (int x = 0; x < n_it; ++x, ++u) {
                    const int b = u & 1, st = u % NS;
                    if (!(ok = mbar_wait(smem_u32(&bar_ds_full[b]), (u >> 1) & 1, &abort_flag))) break;
                    if (x == 0 && !(ok = mbar_wait(smem_u32(&bar_dkv_empty), (kv_items & 1) ^ 1, &abort_flag))) break;
                    tc_fence_after();
                    const uint32_t db = sDS + b * C::kPBytes;
                    const uint32_t qb = sQ + st * C::kQBytes, ob = sDO + st * C::kQBytes;
#pragma unroll
                    for (int ks = 0; ks < BQ / 16; ++ks) {
                        const uint32_t acc = (x > 0 || ks > 0) ? 1u : 0u;
                        umma_bf16_ts(tmem + C::kColDV, tmem + C::kColP + 32 * b + 8 * ks,
                                     sdesc_sw128(ob + ks * 2048, 8192, 1024), idKV, acc);
                        umma_bf16_ss(tmem + C::kColDK, sdesc_sw128(db + ks * 32, 16, 1024),
                                     sdesc_sw128(qb + ks * 2048, 8192, 1024), idKV, acc);
                    }
                    // Q, dO of tile u are read: release the ring stage before dQ^T
                    // (which reads K and dS^T only), so the next load starts earlier
                    umma_commit(smem_u32(&bar_qdo_empty[st]));
                    // dQ^T: the drain warps have read tile u-1's.  Waited for only
                    // now, so that dV and dK never queue behind the drain.
                    if (u > 0 && !(ok = mbar_wait(smem_u32(&bar_dq_empty[b ^ 1]), ((u - 1) >> 1) & 1, &abort_flag)))
                        break;
                    tc_fence_after();
#pragma unroll
                    for (int ks = 0; ks < kBN / 16; ++ks) {
                        umma_bf16_ss(tmem + C::kColDQ, sdesc_sw128(sK + ks * 2048, 16384, 1024),
                                     sdesc_sw128(db + ks * 2048, 16384, 1024), idQ, ks > 0 ? 1u : 0u);
                    }
                    umma_commit(smem_u32(&bar_dq_full[b]));
                }
                if (!ok) break;
                // the item's last reads of K and V (S^T, dP^T of issuer A finished before ds_full)
                umma_commit(smem_u32(&bar_kv_empty));
                umma_commit(smem_u32(&bar_dkv_full));
                ++kv_items;
            }
            if (!ok) {
                umma_commit(smem_u32(&bar_drain_b));
                mbar_wait_drain(smem_u32(&bar_drain_b), 0);
            }
        }
    } else if (warp < 10) {
        // ------------------------------------------------------------ P^T, dS^T
        const int quad = warp & 3;
        const int half = (warp - 2) >> 2;   // query columns half*32 .. half*32+31
        const int t = quad * 32 + lane;     // key row of the block
        const int tw = threadIdx.x - 64;    // 0..255 across both warpgroups
        const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
        const int window = GLOBAL ? kNoWindow : p.window;
        int u = 0;
        bool ok = true;
        for (int k = blockIdx.x; k < n_items && ok; k += gridDim.x) {
            const BwdItem it = decode_bwd2<BQ, GLOBAL>(p, k);
            if (it.ntiles == 0) continue;
            const int k0 = it.j * kBN;
            const int key = k0 + t;
            const int n_it = group * it.ntiles;
            // staging values of tile x (query position, lse, Dsum; -1 / 0 / 0
            // outside the tile's rows): loaded one tile ahead and used only at
            // the next tile, so no instruction waits for the loads while the
            // current tile is computed
            int pf_pos = -1;
            float pf_lse = 0.f, pf_dsum = 0.f;
            auto load_stage = [&](int x) {
                const int h = it.kvh * group + x / it.ntiles;
                const int i = it.i_lo + x % it.ntiles;
                pf_pos = -1;
                pf_lse = pf_dsum = 0.f;
                if (!GLOBAL) {
                    const int q = i * BQ + tw;
                    if (q < p.T) {
                        const int64_t idx = (static_cast<int64_t>(it.b) * p.Hq + h) * p.T + q;
                        pf_pos = q;
                        pf_lse = p.lse[idx];
                        pf_dsum = p.dsum[idx];
                    }
                } else {
                    const int row = i * BQ + tw;
                    if (row >= it.row_lo && row < it.row_hi) {
                        const int64_t idx = static_cast<int64_t>(h) * p.cap + row;
                        pf_pos = p.pos[row];
                        pf_lse = p.lse[idx];
                        pf_dsum = p.dsum[idx];
                    }
                }
            };
            if (tw < BQ) load_stage(0);
            for (int x = 0; x < n_it; ++x, ++u) {
                const int b = u & 1;
                if (tw < BQ) {
                    // lse in log2 units; "sees every key of the block"
                    const bool pf_open = pf_pos >= k0 + kBN - 1 && (GLOBAL || pf_pos - k0 < window);
                    sh_pos[b][tw] = pf_pos;
                    float* pr = reinterpret_cast<float*>(&sh_pair[b][tw >> 1]);
                    pr[tw & 1] = -(pf_lse * kLog2e);
                    pr[2 + (tw & 1)] = -pf_dsum;
                    const bool all_open = __all_sync(0xffffffffu, pf_open);
                    if (lane == 0) sh_open[b][tw >> 5] = all_open ? 1 : 0;
                }
                mbar_arrive(smem_u32(&bar_stage));
                mbar_wait(smem_u32(&bar_stage), u & 1, &abort_flag);  // (if it gave up, so will the next wait)
                if (tw < BQ && x + 1 < n_it) load_stage(x + 1);
                const bool open = sh_open[b][0] && sh_open[b][1];
                ok = mbar_wait(smem_u32(&bar_st_full), u & 1, &abort_flag);
                __syncwarp();
                ok = warp_all(ok);
                if (!ok) break;
                tc_fence_after();
                uint32_t sv[32], dpv[32];
                tmem_ld32(tmem + lane_off + C::kColS + half * 32, sv);
                tmem_ld32(tmem + lane_off + C::kColS + 64 + half * 32, dpv);
                tmem_wait_ld();
                tc_fence_before();
                mbar_arrive(smem_u32(&bar_st_empty));  // S^T, dP^T of tile u+1 may now be written
                uint32_t pk[16], dk2[16];
                // P = 2^(S*scale*log2e - lse), dS = P (dP - Dsum), two columns per
                // f32x2 instruction.  Two branch-free copies of the loop (open
                // tiles skip the visibility test) so that the iterations overlap.
                const uint64_t scale2 = f2_pack(p.scale_log2, p.scale_log2);
                auto columns = [&](auto masked) {
                    constexpr bool kMasked = decltype(masked)::value;
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        const int c = half * 32 + e;
                        const float4 q = sh_pair[b][c >> 1];
                        float x0, x1;
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(sv[e]), __uint_as_float(sv[e + 1])), scale2,
                                         f2_pack(q.x, q.y)),
                                  x0, x1);
                        float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
                        if constexpr (kMasked) {
                            p0 = key_visible(key, sh_pos[b][c], window) ? p0 : 0.f;
                            p1 = key_visible(key, sh_pos[b][c + 1], window) ? p1 : 0.f;
                        }
                        const uint64_t pp = f2_pack(p0, p1);
                        const uint64_t t2 =
                            f2_add(f2_pack(__uint_as_float(dpv[e]), __uint_as_float(dpv[e + 1])), f2_pack(q.z, q.w));
                        float d0, d1;
                        f2_unpack(f2_mul(pp, t2), d0, d1);
                        pk[e / 2] = cvt_bf16x2(p0, p1);
                        dk2[e / 2] = cvt_bf16x2(d0, d1);
                    }
                };
                if (open) columns(std::false_type{});
                else columns(std::true_type{});
                // P^T (TMEM) / dS^T (shared) buffer b is free once the MMAs of tile
                // u-2 are done.  Waiting here rather than before the loads lets
                // S^T, dP^T of tile u+1 enter the MMA queue earlier.
                ok = warp_all(mbar_wait(smem_u32(&bar_dq_full[b]), ((u >> 1) & 1) ^ 1, &abort_flag));
                if (!ok) break;
                tc_fence_after();
                // P^T row t: query columns half*32.. as 16 bf16 pairs, the TMEM
                // operand layout (column c holds queries 2c, 2c+1)
                tmem_st16(tmem + lane_off + C::kColP + 32 * b + half * 16, pk);
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) {
                    const uint32_t off = sw128_offset(t, half * 4 + q4);
                    st_shared_v4(sDS + b * C::kPBytes + off, dk2[4 * q4], dk2[4 * q4 + 1], dk2[4 * q4 + 2],
                                 dk2[4 * q4 + 3]);
                }
                tmem_wait_st();
                fence_proxy_async_smem();
                tc_fence_before();
                mbar_arrive(smem_u32(&bar_ds_full[b]));
            }
        }
    } else if (warp < 14) {
        // ------------------------------------------------------------ dQ drain, dK/dV epilogue
        const int quad = warp & 3;
        const int t = quad * 32 + lane;  // head-dim row of dQ^T
        const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
        int u = 0, kv_items = 0;
        bool ok = true;
        for (int k = blockIdx.x; k < n_items && ok; k += gridDim.x) {
            const BwdItem it = decode_bwd2<BQ, GLOBAL>(p, k);
            const int64_t kv_off =
                ((static_cast<int64_t>(it.b) * p.T + it.j * kBN + quad * 32) * p.Hkv + it.kvh) * D;  // this warp's first key
            const int keys = p.T - (it.j * kBN + quad * 32);  // keys of the warp that exist (may exceed 32, or be negative)
            if (it.ntiles == 0) {
                // no selected query sees the block: zero dK, dV rows, two whole
                // rows (16 lanes x 16 bytes each) per warp store, this warp's 32 keys
                static_assert(D == 128, "two rows of 16 vectors per warp store");
                for (int r = quad * 32 + (lane >> 4); r < quad * 32 + 32; r += 2) {
                    const int kr = it.j * kBN + r;
                    if (kr < p.T) {
                        const int64_t off =
                            ((static_cast<int64_t>(it.b) * p.T + kr) * p.Hkv + it.kvh) * D + (lane & 15) * 8;
                        *reinterpret_cast<uint4*>(p.dk + off) = make_uint4(0, 0, 0, 0);
                        *reinterpret_cast<uint4*>(p.dv + off) = make_uint4(0, 0, 0, 0);
                    }
                }
                continue;
            }
            const int n_it = group * it.ntiles;
            for (int x = 0; x < n_it; ++x, ++u) {
                const int h = it.kvh * group + x / it.ntiles;
                const int i = it.i_lo + x % it.ntiles;
                const int b = u & 1;
                ok = warp_all(mbar_wait(smem_u32(&bar_dq_full[b]), (u >> 1) & 1, &abort_flag));
                if (!ok) break;
                tc_fence_after();
                uint32_t v0[32], v1[32];
                tmem_ld32(tmem + lane_off + C::kColDQ, v0);
                tmem_ld32(tmem + lane_off + C::kColDQ + 32, v1);
                tmem_wait_ld();
                tc_fence_before();
                mbar_arrive(smem_u32(&bar_dq_empty[b]));
                // column c of dQ^T is query row c of the tile: rows outside the
                // tile's valid range carry exact zeros (dS = 0 there) and land in
                // padded or neighbouring accumulator rows
                float* base;
                if (GLOBAL) base = p.dq_acc + static_cast<int64_t>(i * BQ) * p.Hq * D + h * D + t;
                else base = p.dq_acc + (static_cast<int64_t>(it.b) * p.T + i * BQ) * p.Hq * D + h * D + t;
                const int64_t rs = static_cast<int64_t>(p.Hq) * D;
#pragma unroll
                for (int c = 0; c < 32; ++c) atomicAdd(base + c * rs, __uint_as_float(v0[c]) * p.scale);
#pragma unroll
                for (int c = 0; c < 32; ++c) atomicAdd(base + (32 + c) * rs, __uint_as_float(v1[c]) * p.scale);
            }
            if (!ok) break;
            ok = warp_all(mbar_wait(smem_u32(&bar_dkv_full), kv_items & 1, &abort_flag));
            if (!ok) break;
            tc_fence_after();
            // 16 x 256-bit pieces, four lanes trading bf16 pairs (quad_gather8): a warp
            // store is 8 rows of 64 contiguous bytes, not 32 rows of 16, which took
            // 5800 clocks an item behind the reductions, with every role waiting
            // (2 x 4K, 16 heads, 1/8 selected: the kernel 78 -> 71 us)
#pragma unroll
            for (int which = 0; which < 2; ++which) {
                const uint32_t col = which == 0 ? C::kColDK : C::kColDV;
                const float mul = which == 0 ? p.scale : 1.0f;
                logo_bf16* dst = (which == 0 ? p.dk : p.dv) + kv_off + (lane & 3) * 8;
#pragma unroll
                for (int cc = 0; cc < D / 32; ++cc) {
                    uint32_t v[2][16];
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf)
                        tmem_ld_16x256b_x4(tmem + lane_off + (static_cast<uint32_t>(hf * 16) << 16) + col + cc * 32, v[hf]);
                    tmem_wait_ld();
                    if (which == 1 && cc == D / 32 - 1) {
                        tc_fence_before();
                        mbar_arrive(smem_u32(&bar_dkv_empty));
                    }
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                        for (int ab = 0; ab < 2; ++ab) {
                            uint32_t w[4];
#pragma unroll
                            for (int k4 = 0; k4 < 4; ++k4)
                                w[k4] = cvt_bf16x2(__uint_as_float(v[hf][4 * k4 + 2 * ab]) * mul,
                                                   __uint_as_float(v[hf][4 * k4 + 2 * ab + 1]) * mul);
                            const uint4 o = quad_gather8(w, lane);
                            const int r = hf * 16 + ab * 8 + (lane >> 2);
                            if (r < keys) *reinterpret_cast<uint4*>(dst + static_cast<int64_t>(r) * p.Hkv * D + cc * 32) = o;
                        }
                }
            }
            ++kv_items;
        }
    } else if (GLOBAL) {
        // ------------------------------------------------------------ dQ zero fill
        zero_unselected_dq(p, D, lane);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, C::kTmemCols);
    }
}

// ---------------------------------------------------------------- d = 64
// Query tiles of 128 rows: S^T and dP^T are 128 x 128, so a tile has twice the
// elements per MMA instruction, per barrier and per reduced byte that 64-row
// tiles would have (dQ has to be computed as queries x d: d x queries would be
// an M = 64 product).  Per tile 4 + 4 MMAs of N = 128 (S^T, dP^T) and 8 + 8 + 8
// of N = 64 (dV with P^T as the TMEM operand, dK, dQ).  Roles:
//   warp 0       TMA: K/V of an item into one of two buffers (the next item's
//                land during this one: an item has only a few tiles), Q/dO
//                tiles and their rows' lse and Dsum through a 3-deep ring
//   warp 1       MMA issuer A: S^T, dP^T
//   warp 2       MMA issuer B: dV, dK, dQ
//   warp 3       global branch: zero rows of the dense dQ for unselected tokens
//   warps 4..11  two warpgroups, one per 64-query half of the tile; thread =
//                key row: P^T (to TMEM as bf16 pairs) and dS^T (to shared
//                memory) from S^T and dP^T, which it loads whole so that the
//                MMAs of tile u+1 can overwrite them while it computes
//   warps 12..15 dQ out of TMEM (thread = query row), staged 32 columns at a
//                time and added to the fp32 accumulator by bulk tensor
//                reductions, a warp's 32 rows by itself; dK/dV epilogue
// P^T and dS^T are single buffers: TMEM is full (dK, dV, dQ 64 columns each,
// S^T, dP^T 128 each, P^T 64), and the next tile's are only written once its
// arithmetic is done, when the MMAs that read this tile's have ended.
// The kernel before it ran the stages of a tile one after the other (one MMA
// thread, one warpgroup for softmax and dQ atomics, no second tile in flight):
// 2 x 8K, 16 heads, 1/8 selected 299 -> 139 us (131 since the statistics come by
// bulk copy), 3 x 2987, 12/4 heads, window 300 111 -> 53 us.
struct Bwd64Cfg {
    static constexpr int D = 64;
    static constexpr int kBQ = 128;
    static constexpr int kStages = 3;              // Q/dO ring depth
    static constexpr int kTileBytes = 128 * D * 2; // K, V, Q or dO: 16 KB
    static constexpr int kWarpStage = 32 * 128;    // dQ staging of one warp: 32 rows x 32 fp32
    static constexpr int kOffKV = 0;               // 2 buffers of K, V
    static constexpr int kOffQ = kOffKV + 4 * kTileBytes;              // stages of Q, dO
    static constexpr int kOffDS = kOffQ + kStages * 2 * kTileBytes;    // [2 query halves][128 keys][64] bf16
    static constexpr int kOffDQ = kOffDS + 128 * 128 * 2;
    static constexpr int kSmemBytes = kOffDQ + 4 * kWarpStage + 1024;
    static constexpr uint32_t kColDK = 0;
    static constexpr uint32_t kColDV = 64;
    static constexpr uint32_t kColDQ = 128;
    static constexpr uint32_t kColP = 192;   // P^T, bf16 pairs
    static constexpr uint32_t kColS = 256;   // S^T
    static constexpr uint32_t kColDP = 384;  // dP^T
    static constexpr uint32_t kTmemCols = 512;
    static constexpr int kThreads = 512;
    // launched at 128 registers a thread (512 x 128 = 65,536); the softmax
    // warpgroups hold 64 columns of S^T and dP^T a thread (of the splits this one
    // spills least, four words): 128 x (64 + 176 + 176 + 96) = 65,536
    static constexpr uint32_t kRegsControl = 64;
    static constexpr uint32_t kRegsSoftmax = 176;
    static constexpr uint32_t kRegsDrain = 96;
};

template <bool GLOBAL>
__global__ void __launch_bounds__(Bwd64Cfg::kThreads, 1) attn_bwd64_kernel(const __grid_constant__ BwdParams p)
{
    using C = Bwd64Cfg;
    constexpr int D = C::D, BQ = C::kBQ, NS = C::kStages;
    static_assert(128 * (2 * C::kRegsSoftmax + C::kRegsDrain + C::kRegsControl) <= 512 * 128,
                  "register split exceeds the launch allocation");
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t bar_kv_full[2], bar_kv_empty[2], bar_dkv_full, bar_dkv_empty, bar_drain, bar_drain_b;
    __shared__ __align__(8) uint64_t bar_qdo_full[NS], bar_qdo_empty[NS];
    __shared__ __align__(8) uint64_t bar_st_full, bar_st_empty, bar_ds_full, bar_dq_full, bar_dq_empty;
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_flag;
    // of a stage's query columns (2c, 2c+1): (-lse_2c, -lse_2c+1, -Dsum_2c, -Dsum_2c+1),
    // lse in log2 units, and (global) their positions
    __shared__ __align__(16) float4 sh_pair[NS][BQ / 2];
    __shared__ __align__(16) int sh_pos[NS][BQ];
    constexpr uint32_t kStageBytes = 2 * C::kTileBytes + sizeof(sh_pair[0]) + (GLOBAL ? sizeof(sh_pos[0]) : 0);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sKV = smem_u32(smem + C::kOffKV), sQ = smem_u32(smem + C::kOffQ), sDS = smem_u32(smem + C::kOffDS);
    const int group = p.Hq / p.Hkv;
    const int n_items = p.B * p.nblk * p.Hkv;

    // no divisions in the roles' loops: the next tile of an item (head by head),
    // the next stage of the ring and the parity of its turn
    auto next_tile = [](const BwdItem& it, int& h, int& i) {
        if (++i == it.i_lo + it.ntiles) {
            i = it.i_lo;
            ++h;
        }
    };
    auto next_stage = [](int& st, int& turn) {
        if (++st == NS) {
            st = 0;
            turn ^= 1;
        }
    };

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&bar_kv_full[b]), 1);
            mbar_init(smem_u32(&bar_kv_empty[b]), 1);
        }
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&bar_qdo_full[s]), 1);
            mbar_init(smem_u32(&bar_qdo_empty[s]), 1);
        }
        mbar_init(smem_u32(&bar_dkv_full), 1);
        mbar_init(smem_u32(&bar_dkv_empty), 128);
        mbar_init(smem_u32(&bar_drain), 1);
        mbar_init(smem_u32(&bar_drain_b), 1);
        mbar_init(smem_u32(&bar_st_full), 1);
        mbar_init(smem_u32(&bar_st_empty), 256);
        mbar_init(smem_u32(&bar_ds_full), 256);
        mbar_init(smem_u32(&bar_dq_full), 1);
        mbar_init(smem_u32(&bar_dq_empty), 128);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&tmem_base_sh), C::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;

    if (warp < 4) {
        setmaxnreg_dec<C::kRegsControl>();
        if (warp == 0) {
            // -------------------------------------------------------- producer
            if (lane == 0) {
                tma_prefetch_desc(&p.tm_q);
                tma_prefetch_desc(&p.tm_do);
                tma_prefetch_desc(&p.tm_k);
                tma_prefetch_desc(&p.tm_v);
                const uint64_t pol_q = policy_evict_last();
                const uint64_t pol_kv = policy_evict_first();
                int u = 0, st = 0, turn = 0, kv_items = 0;
                bool ok = true;
                for (int k = blockIdx.x; k < n_items && ok; k += gridDim.x) {
                    const BwdItem it = decode_bwd2<BQ, GLOBAL>(p, k);
                    if (it.ntiles == 0) continue;
                    const int kb = kv_items & 1;
                    if (!(ok = mbar_wait(smem_u32(&bar_kv_empty[kb]), ((kv_items >> 1) & 1) ^ 1, &abort_flag))) break;
                    const uint32_t kvb = smem_u32(&bar_kv_full[kb]);
                    mbar_arrive_expect_tx(kvb, 2 * C::kTileBytes);
                    tma_load_4d(sKV + kb * 2 * C::kTileBytes, &p.tm_k, kvb, 0, it.kvh, it.j * kBN, it.b, pol_kv);
                    tma_load_4d(sKV + (kb * 2 + 1) * C::kTileBytes, &p.tm_v, kvb, 0, it.kvh, it.j * kBN, it.b, pol_kv);
                    ++kv_items;
                    const int n_it = group * it.ntiles;
                    for (int x = 0, h = it.kvh * group, i = it.i_lo; x < n_it; ++x, ++u) {
                        if (!(ok = mbar_wait(smem_u32(&bar_qdo_empty[st]), turn ^ 1, &abort_flag))) break;
                        const uint32_t qb = smem_u32(&bar_qdo_full[st]);
                        mbar_arrive_expect_tx(qb, kStageBytes);
                        const int cb = GLOBAL ? 0 : it.b;
                        const int64_t plane = GLOBAL ? h : static_cast<int64_t>(it.b) * p.Hq + h;
                        const float4* stats = p.stats + (plane * p.stat_rows + i * BQ) / 2;
                        if (GLOBAL) {
                            bulk_load(smem_u32(sh_pair[st]), stats, sizeof(sh_pair[0]), qb);
                            bulk_load(smem_u32(sh_pos[st]), p.pos_c + i * BQ, sizeof(sh_pos[0]), qb);
                        } else {
                            const uint32_t have = min(BQ, static_cast<int>(p.stat_rows) - i * BQ) / 2 * sizeof(float4);
                            bulk_load(smem_u32(sh_pair[st]), stats, have, qb);
                            if (have < sizeof(sh_pair[0]))
                                bulk_load(smem_u32(sh_pair[st]) + have, p.stats0, sizeof(sh_pair[0]) - have, qb);
                        }
                        tma_load_4d(sQ + st * 2 * C::kTileBytes, &p.tm_q, qb, 0, h, i * BQ, cb, pol_q);
                        tma_load_4d(sQ + (st * 2 + 1) * C::kTileBytes, &p.tm_do, qb, 0, h, i * BQ, cb, pol_q);
                        next_tile(it, h, i);
                        next_stage(st, turn);
                    }
                }
                if (!ok) {  // let copies already issued land before the CTA exits
                    for (int v = max(0, kv_items - 2); v < kv_items; ++v)
                        mbar_wait_drain(smem_u32(&bar_kv_full[v & 1]), (v >> 1) & 1);
                    for (int v = max(0, u - NS); v < u; ++v)
                        mbar_wait_drain(smem_u32(&bar_qdo_full[v % NS]), (v / NS) & 1);
                }
            }
        } else if (warp == 1) {
            // -------------------------------------------------------- MMA issuer A: S^T, dP^T
            if (lane == 0) {
                constexpr uint32_t idS = idesc_bf16_f32(kBN, BQ, false, false);
                int u = 0, st = 0, turn = 0, kv_items = 0;
                bool ok = true;
                for (int k = blockIdx.x; k < n_items && ok; k += gridDim.x) {
                    const BwdItem it = decode_bwd2<BQ, GLOBAL>(p, k);
                    if (it.ntiles == 0) continue;
                    const uint32_t sK = sKV + (kv_items & 1) * 2 * C::kTileBytes, sV = sK + C::kTileBytes;
                    if (!(ok = mbar_wait(smem_u32(&bar_kv_full[kv_items & 1]), (kv_items >> 1) & 1, &abort_flag))) break;
                    const int n_it = group * it.ntiles;
                    for (int x = 0; x < n_it; ++x, ++u) {
                        if (!(ok = mbar_wait(smem_u32(&bar_qdo_full[st]), turn, &abort_flag))) break;
                        // the softmax warps have loaded S^T, dP^T of tile u-1
                        if (!(ok = mbar_wait(smem_u32(&bar_st_empty), (u & 1) ^ 1, &abort_flag))) break;
                        tc_fence_after();
                        const uint32_t qb = sQ + st * 2 * C::kTileBytes, ob = qb + C::kTileBytes;
#pragma unroll
                        for (int ks = 0; ks < D / 16; ++ks) {
                            umma_bf16_ss(tmem + C::kColS, sdesc_sw128(sK + ks * 32, 16, 1024),
                                         sdesc_sw128(qb + ks * 32, 16, 1024), idS, ks > 0 ? 1u : 0u);
                            umma_bf16_ss(tmem + C::kColDP, sdesc_sw128(sV + ks * 32, 16, 1024),
                                         sdesc_sw128(ob + ks * 32, 16, 1024), idS, ks > 0 ? 1u : 0u);
                        }
                        umma_commit(smem_u32(&bar_st_full));
                        next_stage(st, turn);
                    }
                    if (!ok) break;
                    ++kv_items;
                }
                if (!ok) {
                    umma_commit(smem_u32(&bar_drain));
                    mbar_wait_drain(smem_u32(&bar_drain), 0);
                }
            }
        } else if (warp == 2) {
            // -------------------------------------------------------- MMA issuer B: dV, dK, dQ
            if (lane == 0) {
                constexpr uint32_t idKV = idesc_bf16_f32(kBN, D, false, true);  // dV, dK: keys x d
                constexpr uint32_t idQ = idesc_bf16_f32(BQ, D, true, true);     // dQ: queries x d
                int u = 0, st = 0, turn = 0, kv_items = 0;
                bool ok = true;
                for (int k = blockIdx.x; k < n_items && ok; k += gridDim.x) {
                    const BwdItem it = decode_bwd2<BQ, GLOBAL>(p, k);
                    if (it.ntiles == 0) continue;
                    const uint32_t sK = sKV + (kv_items & 1) * 2 * C::kTileBytes;
                    const int n_it = group * it.ntiles;
                    for (int x = 0; x < n_it; ++x, ++u) {
                        if (!(ok = mbar_wait(smem_u32(&bar_ds_full), u & 1, &abort_flag))) break;
                        if (x == 0 && !(ok = mbar_wait(smem_u32(&bar_dkv_empty), (kv_items & 1) ^ 1, &abort_flag))) break;
                        tc_fence_after();
                        const uint32_t qb = sQ + st * 2 * C::kTileBytes, ob = qb + C::kTileBytes;
#pragma unroll
                        for (int ks = 0; ks < BQ / 16; ++ks) {
                            const uint32_t acc = (x > 0 || ks > 0) ? 1u : 0u;
                            umma_bf16_ts(tmem + C::kColDV, tmem + C::kColP + 8 * ks,
                                         sdesc_sw128(ob + ks * 2048, 16384, 1024), idKV, acc);
                            umma_bf16_ss(tmem + C::kColDK, sdesc_sw128(sDS + (ks >> 2) * 16384 + (ks & 3) * 32, 16, 1024),
                                         sdesc_sw128(qb + ks * 2048, 16384, 1024), idKV, acc);
                        }
                        // Q, dO of tile u are read: the ring stage is free before dQ
                        umma_commit(smem_u32(&bar_qdo_empty[st]));
                        // the drain warps have read tile u-1's dQ
                        if (u > 0 && !(ok = mbar_wait(smem_u32(&bar_dq_empty), (u - 1) & 1, &abort_flag))) break;
                        tc_fence_after();
#pragma unroll
                        for (int ks = 0; ks < kBN / 16; ++ks)
                            umma_bf16_ss(tmem + C::kColDQ, sdesc_sw128(sDS + ks * 2048, 16384, 1024),
                                         sdesc_sw128(sK + ks * 2048, 16384, 1024), idQ, ks > 0 ? 1u : 0u);
                        umma_commit(smem_u32(&bar_dq_full));
                        next_stage(st, turn);
                    }
                    if (!ok) break;
                    umma_commit(smem_u32(&bar_kv_empty[kv_items & 1]));
                    umma_commit(smem_u32(&bar_dkv_full));
                    ++kv_items;
                }
                if (!ok) {
                    umma_commit(smem_u32(&bar_drain_b));
                    mbar_wait_drain(smem_u32(&bar_drain_b), 0);
                }
            }
        } else if (GLOBAL) {
            zero_unselected_dq(p, D, lane);
        }
    } else if (warp < 12) {
        // ------------------------------------------------------------ P^T, dS^T
        setmaxnreg_inc<C::kRegsSoftmax>();
        const int quad = warp & 3;
        const int half = (warp - 4) >> 2;  // query columns half*64 .. half*64+63
        const int t = quad * 32 + lane;    // key row of the block
        const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
        int u = 0, st = 0, turn = 0;
        bool ok = true;
        for (int k = blockIdx.x; k < n_items && ok; k += gridDim.x) {
            const BwdItem it = decode_bwd2<BQ, GLOBAL>(p, k);
            if (it.ntiles == 0) continue;
            const int k0 = it.j * kBN;
            const int key = k0 + t;
            const int row_first = it.i_lo * BQ, row_end = row_first + it.ntiles * BQ;
            int row0 = row_first;
            for (int left = group * it.ntiles; left > 0; --left, ++u) {
                mbar_wait(smem_u32(&bar_qdo_full[st]), turn, &abort_flag);  // (if it gave up, so will the next wait)
                // every column of the half sees every key of the block
                bool open;
                {
                    const int r0 = row0 + half * 64, r1 = r0 + 63;
                    if (!GLOBAL) open = r0 >= k0 + kBN - 1 && r1 < p.T && r1 - k0 < p.window;
                    else open = r0 >= it.row_lo && r1 < it.row_hi && sh_pos[st][half * 64] >= k0 + kBN - 1;
                }
                // the columns that see this key are adjacent: [lo, hi] of this half
                int lo = 0, hi = 63;
                if (!open) {
                    if (!GLOBAL) {
                        lo = key - row0;
                        hi = min(lo + p.window - 1, p.T - 1 - row0);
                    } else {  // positions ascend over the sequence's rows of the tile
                        int a = max(0, it.row_lo - row0), e = min(BQ, it.row_hi - row0);
                        hi = e - 1;
                        while (a < e) {
                            const int mid = (a + e) >> 1;
                            if (sh_pos[st][mid] < key) a = mid + 1;
                            else e = mid;
                        }
                        lo = a;
                    }
                    lo -= half * 64;
                    hi -= half * 64;
                }
                ok = mbar_wait_warp(smem_u32(&bar_st_full), u & 1, &abort_flag);
                __syncwarp();
                if (!ok) break;
                tc_fence_after();
                uint32_t sv[2][32], dpv[2][32];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    tmem_ld32(tmem + lane_off + C::kColS + half * 64 + c * 32, sv[c]);
                    tmem_ld32(tmem + lane_off + C::kColDP + half * 64 + c * 32, dpv[c]);
                }
                tmem_wait_ld();
                tc_fence_before();
                mbar_arrive(smem_u32(&bar_st_empty));  // S^T, dP^T of tile u+1 may now be written
                // P = 2^(S*scale*log2e - lse), dS = P (dP - Dsum), two columns per
                // f32x2 instruction; two branch-free copies of the loop (open tiles
                // skip the visibility selects)
                uint32_t pk[32], dk2[32];
                const uint64_t scale2 = f2_pack(p.scale_log2, p.scale_log2);
                auto columns = [&](auto masked) {
                    constexpr bool kMasked = decltype(masked)::value;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t m = 0xffffffffu;
                        if constexpr (kMasked) m = column_mask(lo - 32 * c, hi - 32 * c);
#pragma unroll
                        for (int e = 0; e < 32; e += 2) {
                            const float4 q = sh_pair[st][(half * 64 + c * 32 + e) >> 1];
                            float x0, x1;
                            f2_unpack(f2_fma(f2_pack(__uint_as_float(sv[c][e]), __uint_as_float(sv[c][e + 1])), scale2,
                                             f2_pack(q.x, q.y)),
                                      x0, x1);
                            float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
                            if constexpr (kMasked) {
                                p0 = (m & (1u << e)) ? p0 : 0.f;
                                p1 = (m & (2u << e)) ? p1 : 0.f;
                            }
                            const uint64_t t2 = f2_add(
                                f2_pack(__uint_as_float(dpv[c][e]), __uint_as_float(dpv[c][e + 1])), f2_pack(q.z, q.w));
                            float d0, d1;
                            f2_unpack(f2_mul(f2_pack(p0, p1), t2), d0, d1);
                            pk[c * 16 + e / 2] = cvt_bf16x2(p0, p1);
                            dk2[c * 16 + e / 2] = cvt_bf16x2(d0, d1);
                        }
                    }
                };
                if (open) columns(std::false_type{});
                else columns(std::true_type{});
                // P^T (TMEM) and dS^T (shared) are free once the MMAs of tile u-1 are done
                if (u > 0) {
                    ok = mbar_wait_warp(smem_u32(&bar_dq_full), (u - 1) & 1, &abort_flag);
                    __syncwarp();
                    if (!ok) break;
                }
                tc_fence_after();
                tmem_st32(tmem + lane_off + C::kColP + half * 32, pk);
#pragma unroll
                for (int q4 = 0; q4 < 8; ++q4)
                    st_shared_v4(sDS + half * 16384 + sw128_offset(t, q4), dk2[4 * q4], dk2[4 * q4 + 1], dk2[4 * q4 + 2],
                                 dk2[4 * q4 + 3]);
                tmem_wait_st();
                fence_proxy_async_smem();
                tc_fence_before();
                mbar_arrive(smem_u32(&bar_ds_full));
                row0 = row0 + BQ == row_end ? row_first : row0 + BQ;
                next_stage(st, turn);
            }
        }
    } else {
        // ------------------------------------------------------------ dQ drain, dK/dV epilogue
        setmaxnreg_dec<C::kRegsDrain>();
        const int quad = warp & 3;
        const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
        const uint32_t stage = smem_u32(smem + C::kOffDQ) + quad * C::kWarpStage;
        int u = 0, kv_items = 0;
        bool ok = true;
        for (int k = blockIdx.x; k < n_items && ok; k += gridDim.x) {
            const BwdItem it = decode_bwd2<BQ, GLOBAL>(p, k);
            const int64_t kv_off =
                ((static_cast<int64_t>(it.b) * p.T + it.j * kBN + quad * 32) * p.Hkv + it.kvh) * D;  // this warp's first key
            const int keys = p.T - (it.j * kBN + quad * 32);  // keys of the warp that exist (may exceed 32, or be negative)
            if (it.ntiles == 0) {
                // no selected query sees the block: zero dK, dV rows, four whole
                // rows (8 lanes x 16 bytes each) per warp store
                for (int r = lane >> 3; r < 32; r += 4) {
                    if (r < keys) {
                        const int64_t off = kv_off + static_cast<int64_t>(r) * p.Hkv * D + (lane & 7) * 8;
                        *reinterpret_cast<uint4*>(p.dk + off) = make_uint4(0, 0, 0, 0);
                        *reinterpret_cast<uint4*>(p.dv + off) = make_uint4(0, 0, 0, 0);
                    }
                }
                continue;
            }
            const int n_it = group * it.ntiles;
            for (int x = 0, h = it.kvh * group, i = it.i_lo; x < n_it; ++x, ++u, next_tile(it, h, i)) {
                const int row0 = i * BQ + quad * 32;  // this warp's first query row
                ok = mbar_wait_warp(smem_u32(&bar_dq_full), u & 1, &abort_flag);
                __syncwarp();
                if (!ok) break;
                tc_fence_after();
                uint32_t v[2][32];
                tmem_ld32(tmem + lane_off + C::kColDQ, v[0]);
                tmem_ld32(tmem + lane_off + C::kColDQ + 32, v[1]);
                tmem_wait_ld();
                tc_fence_before();
                mbar_arrive(smem_u32(&bar_dq_empty));
                // rows of other sequences or past the end add zero
                const int row = row0 + lane;
                const float mul = (!GLOBAL || (row >= it.row_lo && row < it.row_hi)) ? p.scale : 0.f;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    // the reduction before has read the staging rows
                    if (lane == 0) bulk_wait_read();
                    __syncwarp();
#pragma unroll
                    for (int q4 = 0; q4 < 8; ++q4) {
                        uint32_t w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            w[e] = mul != 0.f ? __float_as_uint(__uint_as_float(v[c][4 * q4 + e]) * mul) : 0u;
                        st_shared_v4(stage + sw128_offset(lane, q4), w[0], w[1], w[2], w[3]);
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0 && (GLOBAL || row0 < p.T)) {
                        tma_reduce_add_4d(&p.tm_dq, stage, 32 * c, h, row0, GLOBAL ? 0 : it.b);
                        bulk_commit();
                    }
                }
            }
            if (!ok) break;
            ok = mbar_wait_warp(smem_u32(&bar_dkv_full), kv_items & 1, &abort_flag);
            __syncwarp();
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int which = 0; which < 2; ++which) {
                const uint32_t col = which == 0 ? C::kColDK : C::kColDV;
                const float mul = which == 0 ? p.scale : 1.0f;
                logo_bf16* dst = (which == 0 ? p.dk : p.dv) + kv_off + (lane & 3) * 8;
#pragma unroll
                for (int cc = 0; cc < D / 32; ++cc) {
                    uint32_t v[2][16];
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf)
                        tmem_ld_16x256b_x4(tmem + lane_off + (static_cast<uint32_t>(hf * 16) << 16) + col + cc * 32, v[hf]);
                    tmem_wait_ld();
                    if (which == 1 && cc == D / 32 - 1) {
                        tc_fence_before();
                        mbar_arrive(smem_u32(&bar_dkv_empty));
                    }
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                        for (int ab = 0; ab < 2; ++ab) {
                            uint32_t w[4];
#pragma unroll
                            for (int k4 = 0; k4 < 4; ++k4)
                                w[k4] = cvt_bf16x2(__uint_as_float(v[hf][4 * k4 + 2 * ab]) * mul,
                                                   __uint_as_float(v[hf][4 * k4 + 2 * ab + 1]) * mul);
                            const uint4 o = quad_gather8(w, lane);
                            const int r = hf * 16 + ab * 8 + (lane >> 2);
                            if (r < keys) *reinterpret_cast<uint4*>(dst + static_cast<int64_t>(r) * p.Hkv * D + cc * 32) = o;
                        }
                }
            }
            ++kv_items;
        }
        if (lane == 0) bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, C::kTmemCols);
    }
}

// ---------------------------------------------------------------- pre / post
// Per (row, head): Dsum = sum_d dO * O (fp32); zero the dQ accumulator rows.
// Global branch: also copy dO_c into the workspace and gather the selected
// rows of the dense Q into the packed layout (App. B), zero-padding the 128
// rows after the last selected one so that partial tiles read finite values;
// and build, for every sequence b and KV block j, the first packed row of b
// whose position reaches the block's first key (App. B's precomputed search
// that lets the backward skip every query tile before it).
// For d = 64 the pass writes what the backward kernel needs of a row as the
// kernel's shared memory holds it, (-lse, -lse, -Dsum, -Dsum) of two adjacent
// rows with lse in log2 units, and with the positions beside them: a tile's are
// then two bulk copies that come with its Q and dO.  Rows of a tile that do not
// exist are zero: the packed rows' plane is filled to a multiple of 128, the
// local branch's planes (one a sequence and head, perhaps of a single row) to an
// even length only, and the rest of a last tile comes from one block of zeros.  (Loaded, converted and stored by the
// softmax warps with a barrier of all 256 threads, and divisions in the roles'
// loops: 2 x 8K, 16 heads, 1/8 selected, all kernels of the call 158 -> 149 us.)
struct RowStats {
    const float* lse;  // local [B,H,T]; global [H,cap]
    float* out;        // null: d = 128, dsum is written instead
    int32_t* pos;      // global
    int64_t rows;      // of a plane
    float4* zeros;     // local: the statistics of kBM rows that do not exist
};

__host__ __device__ constexpr int64_t packed_stat_rows(int64_t rows) { return (rows + kBM - 1) / kBM * kBM; }
__host__ __device__ constexpr int64_t local_stat_rows(int64_t T) { return (T + 1) / 2 * 2; }
constexpr size_t kStatZeros = kBM / 2 * sizeof(float4);

struct GlobalPrep {
    const logo_bf16* q;   // dense [B, T, H, D]
    const int32_t* pos;
    const int32_t* cu_q;
    logo_bf16* qc;        // packed [cap + 128, H, D]
    int32_t* first_row;   // [B, nblk]
    int B, nblk;
};

template <bool GLOBAL>
__global__ void __launch_bounds__(128) bwd_pre_kernel(const logo_bf16* __restrict__ o, const logo_bf16* __restrict__ dO,
                                                      const int32_t* __restrict__ n_sel, int rows_host, int T, int H,
                                                      int D, int cap, float* __restrict__ dsum,
                                                      logo_bf16* __restrict__ do_copy, float* __restrict__ dq_acc,
                                                      GlobalPrep gp, RowStats rst)
{
    const int n = GLOBAL ? *n_sel : rows_host;
    const int rows = GLOBAL ? n + kBM : rows_host;
    const int vpr = D / 8, nvec = H * vpr;
    if (GLOBAL) {
        for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < gp.B * gp.nblk; idx += gridDim.x * blockDim.x) {
            const int b = idx / gp.nblk, j = idx % gp.nblk;
            int lo = gp.cu_q[b], hi = gp.cu_q[b + 1];
            const int k0 = j * kBN;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (gp.pos[mid] < k0) lo = mid + 1;
                else hi = mid;
            }
            gp.first_row[idx] = lo;
        }
    }
    auto put_stats = [&](int64_t plane, int64_t r, float nlse, float ndsum) {
        float* at = rst.out + (plane * rst.rows + (r & ~static_cast<int64_t>(1))) * 2 + (r & 1);
        at[0] = nlse;
        at[2] = ndsum;
    };
    if (!GLOBAL && rst.out && blockIdx.x == 0)
        for (int i = threadIdx.x; i < kBM / 2; i += blockDim.x) rst.zeros[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int row = blockIdx.x; row < rows; row += gridDim.x) {
        const bool live = row < n;
        if (GLOBAL && rst.out && threadIdx.x == 0) rst.pos[row] = live ? gp.pos[row] : 0;
        const int64_t base = static_cast<int64_t>(row) * H * D;
        if (GLOBAL) {
            uint4* dst = reinterpret_cast<uint4*>(gp.qc + base);
            if (live) {
                const int b = seq_of_row(gp.cu_q, gp.B, row);
                const uint4* src = reinterpret_cast<const uint4*>(gp.q + (static_cast<int64_t>(b) * T + gp.pos[row]) * H * D);
                for (int v = threadIdx.x; v < nvec; v += blockDim.x) dst[v] = src[v];
            } else {
                for (int v = threadIdx.x; v < nvec; v += blockDim.x) dst[v] = make_uint4(0, 0, 0, 0);
            }
        }
        for (int v0 = 0; v0 < nvec; v0 += blockDim.x) {
            const int v = v0 + threadIdx.x;
            const bool active = v < nvec;
            const int h = active ? v / vpr : 0, jj = active ? v % vpr : 0;
            float acc = 0.f;
            uint4 graw = make_uint4(0, 0, 0, 0);
            if (active && live) {
                graw = *reinterpret_cast<const uint4*>(dO + base + h * D + jj * 8);
                const uint4 oraw = *reinterpret_cast<const uint4*>(o + base + h * D + jj * 8);
                const __nv_bfloat162* g2 = reinterpret_cast<const __nv_bfloat162*>(&graw);
                const __nv_bfloat162* o2 = reinterpret_cast<const __nv_bfloat162*>(&oraw);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 a = __bfloat1622float2(g2[e]), b = __bfloat1622float2(o2[e]);
                    acc = fmaf(a.x, b.x, acc);
                    acc = fmaf(a.y, b.y, acc);
                }
            }
            for (int off = vpr >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (active) {
                if (GLOBAL) *reinterpret_cast<uint4*>(do_copy + base + h * D + jj * 8) = graw;
                float4* z = reinterpret_cast<float4*>(dq_acc + base + h * D + jj * 8);
                z[0] = make_float4(0.f, 0.f, 0.f, 0.f);
                z[1] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (jj == 0 && rst.out) {
                    const int b = GLOBAL ? 0 : row / T, tt = GLOBAL ? row : row % T;
                    const int64_t lse_row = GLOBAL ? static_cast<int64_t>(h) * cap + row
                                                   : (static_cast<int64_t>(b) * H + h) * T + tt;
                    const int64_t plane = static_cast<int64_t>(b) * H + h;
                    put_stats(plane, tt, live ? -(rst.lse[lse_row] * kLog2e) : 0.f, -acc);
                    if (!GLOBAL && tt + 1 == T && tt + 1 < rst.rows) put_stats(plane, tt + 1, 0.f, 0.f);
                } else if (live && jj == 0) {
                    if (GLOBAL) dsum[static_cast<int64_t>(h) * cap + row] = acc;
                    else {
                        const int b = row / T, tt = row % T;
                        dsum[(static_cast<int64_t>(b) * H + h) * T + tt] = acc;
                    }
                }
            }
        }
    }
}

// Global branch: dQ accumulator rows of the selected tokens -> their
// rows of the dense dq (the backward kernel zeroed the others); blocks stride
// over the packed rows below the selected count.
__global__ void __launch_bounds__(128) bwd_post_selected_kernel(const float* __restrict__ dq_acc,
                                                                const int32_t* __restrict__ pos,
                                                                const int32_t* __restrict__ cu_q,
                                                                const int32_t* __restrict__ n_sel, int B, int T, int H,
                                                                int D, logo_bf16* __restrict__ dq)
{
    const int n = *n_sel;
    const int row_elems = H * D;
    for (int r = blockIdx.x; r < n; r += gridDim.x) {
        const int b = seq_of_row(cu_q, B, r);
        const int64_t dst_row = static_cast<int64_t>(b) * T + pos[r];
        for (int v = threadIdx.x; v < row_elems / 8; v += blockDim.x) {
            const float4* s = reinterpret_cast<const float4*>(dq_acc + static_cast<int64_t>(r) * row_elems + v * 8);
            const float4 a = s[0], c = s[1];
            uint4 w;
            w.x = pack_bf16x2(a.x, a.y);
            w.y = pack_bf16x2(a.z, a.w);
            w.z = pack_bf16x2(c.x, c.y);
            w.w = pack_bf16x2(c.z, c.w);
            *reinterpret_cast<uint4*>(dq + dst_row * row_elems + v * 8) = w;
        }
    }
}

// Local branch: dQ accumulator (fp32) -> dq (bf16).
__global__ void __launch_bounds__(128) bwd_post_kernel(const float* __restrict__ dq_acc, int row_elems,
                                                       logo_bf16* __restrict__ dq)
{
    const int64_t bt = blockIdx.x;
    for (int v = threadIdx.x; v < row_elems / 8; v += blockDim.x) {
        const float4* s = reinterpret_cast<const float4*>(dq_acc + bt * row_elems + v * 8);
        const float4 a = s[0], c = s[1];
        uint4 w;
        w.x = pack_bf16x2(a.x, a.y);
        w.y = pack_bf16x2(a.z, a.w);
        w.z = pack_bf16x2(c.x, c.y);
        w.w = pack_bf16x2(c.z, c.w);
        *reinterpret_cast<uint4*>(dq + bt * row_elems + v * 8) = w;
    }
}

struct BwdWs {
    logo_bf16* qc;
    logo_bf16* doc;
    float* dsum;  // d = 128; d = 64: the row stats
    float4* zeros;
    int32_t* pos_c;
    float* dq_acc;
    int32_t* first_row;
};

size_t local_bwd_ws_layout(const logo_dims& d, char* base, BwdWs* ws)
{
    const size_t rows = static_cast<size_t>(d.B) * d.T;
    size_t off = 0;
    const size_t o_ds = off;
    const size_t stats = d.D == 64 ? static_cast<size_t>(d.B) * local_stat_rows(d.T) * 2 : rows;
    off = round_up(off + stats * d.Hq * sizeof(float), 256);
    const size_t o_zr = off;
    if (d.D == 64) off = round_up(off + kStatZeros, 256);
    const size_t o_dq = off;
    off = round_up(off + (rows + kBM) * d.Hq * d.D * sizeof(float), 256);
    if (ws) {
        ws->qc = ws->doc = nullptr;
        ws->pos_c = nullptr;
        ws->zeros = reinterpret_cast<float4*>(base + o_zr);
        ws->dsum = reinterpret_cast<float*>(base + o_ds);
        ws->dq_acc = reinterpret_cast<float*>(base + o_dq);
        ws->first_row = nullptr;
    }
    return off;
}

size_t global_bwd_ws_layout(const logo_dims& d, char* base, BwdWs* ws)
{
    const size_t cap = static_cast<size_t>(d.B) * d.T;
    const size_t rows = cap + kBM;
    size_t off = 0;
    const size_t o_qc = off;
    off = round_up(off + rows * d.Hq * d.D * 2, 256);
    const size_t o_do = off;
    off = round_up(off + rows * d.Hq * d.D * 2, 256);
    const size_t o_ds = off;
    const size_t stats = d.D == 64 ? static_cast<size_t>(packed_stat_rows(rows)) * 2 : cap;
    off = round_up(off + stats * d.Hq * sizeof(float), 256);
    const size_t o_pc = off;
    if (d.D == 64) off = round_up(off + packed_stat_rows(rows) * sizeof(int32_t), 256);
    const size_t o_dq = off;
    off = round_up(off + rows * d.Hq * d.D * sizeof(float), 256);
    const size_t o_fr = off;
    off = round_up(off + static_cast<size_t>(d.B) * ((d.T + kBN - 1) / kBN) * sizeof(int32_t), 256);
    if (ws) {
        ws->first_row = reinterpret_cast<int32_t*>(base + o_fr);
        ws->zeros = nullptr;
        ws->pos_c = reinterpret_cast<int32_t*>(base + o_pc);
        ws->qc = reinterpret_cast<logo_bf16*>(base + o_qc);
        ws->doc = reinterpret_cast<logo_bf16*>(base + o_do);
        ws->dsum = reinterpret_cast<float*>(base + o_ds);
        ws->dq_acc = reinterpret_cast<float*>(base + o_dq);
    }
    return off;
}

template <int D, bool GLOBAL>
int launch_bwd(const BwdParams& prm, cudaStream_t st)
{
    static bool attr_done = false;  // benign race: setting the attribute twice is harmless
    const int n_items = prm.B * prm.nblk * prm.Hkv;
    const int grid = max(1, min(n_items, device_sm_count()));
    if (D == 128) {
        if (!attr_done) {
            if (set_smem_limit(attn_bwd2_kernel<GLOBAL>, Bwd2Cfg::kSmemBytes) != cudaSuccess) return LOGO_ERR_CUDA;
            attr_done = true;
        }
        attn_bwd2_kernel<GLOBAL><<<grid, Bwd2Cfg::kThreads, Bwd2Cfg::kSmemBytes, st>>>(prm);
    } else {
        if (!attr_done) {
            if (set_smem_limit(attn_bwd64_kernel<GLOBAL>, Bwd64Cfg::kSmemBytes) != cudaSuccess) return LOGO_ERR_CUDA;
            attr_done = true;
        }
        attn_bwd64_kernel<GLOBAL><<<grid, Bwd64Cfg::kThreads, Bwd64Cfg::kSmemBytes, st>>>(prm);
    }
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}

int check_bwd_ptrs(const void* const* ptrs, int n)
{
    for (int i = 0; i < n; ++i) {
        if (!ptrs[i]) return LOGO_ERR_INVALID_ARG;
        if (!aligned16(ptrs[i])) return LOGO_ERR_UNSUPPORTED;
    }
    return LOGO_OK;
}

}  // namespace

int attn_bwd_tu_status(int clear) { return read_tu_status(clear); }

}  // namespace logo

using namespace logo;

extern "C" size_t logo_local_attn_bwd_workspace_size(logo_dims dims)
{
    if (check_dims(dims) != LOGO_OK) return 0;
    return local_bwd_ws_layout(dims, nullptr, nullptr);
}

extern "C" int logo_local_attn_bwd(const logo_bf16* q, const logo_bf16* k, const logo_bf16* v, const logo_bf16* o,
                                   const float* lse, const logo_bf16* dO, logo_bf16* dq, logo_bf16* dk,
                                   logo_bf16* dv, logo_dims dims, int window, float scale, void* workspace,
                                   size_t workspace_bytes, void* stream)
{
    int rc = check_dims(dims);
    if (rc != LOGO_OK) return rc;
    const void* ptrs[] = {q, k, v, o, dO, dq, dk, dv};
    if ((rc = check_bwd_ptrs(ptrs, 8)) != LOGO_OK) return rc;
    if (!lse || window < 1) return LOGO_ERR_INVALID_ARG;
    if (!(scale >= 0.0f)) return LOGO_ERR_INVALID_ARG;
    if (scale == 0.0f) scale = 1.0f / sqrtf(static_cast<float>(dims.D));
    const size_t need = local_bwd_ws_layout(dims, nullptr, nullptr);
    if (!workspace || workspace_bytes < need || !aligned16(workspace)) return LOGO_ERR_WORKSPACE;
    BwdWs ws;
    local_bwd_ws_layout(dims, static_cast<char*>(workspace), &ws);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int rows = dims.B * dims.T;
    const int pre_grid = max(1, min(rows, device_sm_count() * 16));
    const RowStats rst{lse, dims.D == 64 ? ws.dsum : nullptr, nullptr, local_stat_rows(dims.T), ws.zeros};
    bwd_pre_kernel<false><<<pre_grid, 128, 0, st>>>(o, dO, nullptr, rows, dims.T, dims.Hq, dims.D, 0, ws.dsum,
                                                    nullptr, ws.dq_acc, GlobalPrep{}, rst);
    BwdParams prm{};
    prm.stats = reinterpret_cast<const float4*>(rst.out);
    prm.stats0 = rst.zeros;
    prm.stat_rows = rst.rows;
    const uint32_t qrows = dims.D == 128 ? Bwd2Cfg::kBQ : Bwd64Cfg::kBQ;
    if (!encode_bf16_4d(&prm.tm_q, q, dims.D, dims.Hq, dims.T, dims.B, 64, qrows) ||
        !encode_bf16_4d(&prm.tm_do, dO, dims.D, dims.Hq, dims.T, dims.B, 64, qrows) ||
        !encode_bf16_4d(&prm.tm_k, k, dims.D, dims.Hkv, dims.T, dims.B, 64, kBN) ||
        !encode_bf16_4d(&prm.tm_v, v, dims.D, dims.Hkv, dims.T, dims.B, 64, kBN) ||
        (dims.D == 64 && !encode_f32_4d(&prm.tm_dq, ws.dq_acc, dims.D, dims.Hq, dims.T, dims.B, 32, 32)))
        return LOGO_ERR_CUDA;
    prm.lse = lse;
    prm.dsum = ws.dsum;
    prm.dq_acc = ws.dq_acc;
    prm.dk = dk;
    prm.dv = dv;
    prm.B = dims.B;
    prm.T = dims.T;
    prm.Hq = dims.Hq;
    prm.Hkv = dims.Hkv;
    prm.window = window > dims.T ? dims.T : window;
    prm.cap = rows;
    prm.nblk = (dims.T + kBN - 1) / kBN;
    prm.scale = scale;
    prm.scale_log2 = scale * kLog2e;
    rc = dims.D == 128 ? launch_bwd<128, false>(prm, st) : launch_bwd<64, false>(prm, st);
    if (rc != LOGO_OK) return rc;
    bwd_post_kernel<<<rows, 128, 0, st>>>(ws.dq_acc, dims.Hq * dims.D, dq);
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}

extern "C" size_t logo_global_attn_bwd_workspace_size(logo_dims dims)
{
    if (check_dims(dims) != LOGO_OK) return 0;
    return global_bwd_ws_layout(dims, nullptr, nullptr);
}

extern "C" int logo_global_sparse_attn_bwd(const logo_bf16* q, const logo_bf16* k, const logo_bf16* v,
                                           const int32_t* pos, const int32_t* cu_q, const int32_t* n_sel_total,
                                           const logo_bf16* o_c, const float* lse_c, const logo_bf16* dO_c,
                                           logo_bf16* dq, logo_bf16* dk, logo_bf16* dv, logo_dims dims, float scale,
                                           void* workspace, size_t workspace_bytes, void* stream)
{
    int rc = check_dims(dims);
    if (rc != LOGO_OK) return rc;
    const void* ptrs[] = {q, k, v, o_c, dO_c, dq, dk, dv};
    if ((rc = check_bwd_ptrs(ptrs, 8)) != LOGO_OK) return rc;
    if (!pos || !cu_q || !n_sel_total || !lse_c) return LOGO_ERR_INVALID_ARG;
    if (!(scale >= 0.0f)) return LOGO_ERR_INVALID_ARG;
    if (scale == 0.0f) scale = 1.0f / sqrtf(static_cast<float>(dims.D));
    const size_t need = global_bwd_ws_layout(dims, nullptr, nullptr);
    if (!workspace || workspace_bytes < need || !aligned16(workspace)) return LOGO_ERR_WORKSPACE;
    BwdWs ws;
    global_bwd_ws_layout(dims, static_cast<char*>(workspace), &ws);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int cap = dims.B * dims.T;
    const int grid_rows = max(1, min(cap + kBM, device_sm_count() * 16));
    const int nblk = (dims.T + kBN - 1) / kBN;
    const GlobalPrep gp{q, pos, cu_q, ws.qc, ws.first_row, dims.B, nblk};
    const RowStats rst{lse_c, dims.D == 64 ? ws.dsum : nullptr, ws.pos_c, packed_stat_rows(static_cast<int64_t>(cap) + kBM),
                       nullptr};
    bwd_pre_kernel<true><<<grid_rows, 128, 0, st>>>(o_c, dO_c, n_sel_total, 0, dims.T, dims.Hq, dims.D, cap, ws.dsum,
                                                    ws.doc, ws.dq_acc, gp, rst);
    if (cudaGetLastError() != cudaSuccess) return LOGO_ERR_CUDA;
    BwdParams prm{};
    prm.stats = reinterpret_cast<const float4*>(rst.out);
    prm.pos_c = rst.pos;
    prm.stat_rows = rst.rows;
    const uint32_t qrows = dims.D == 128 ? Bwd2Cfg::kBQ : Bwd64Cfg::kBQ;
    if (!encode_bf16_4d(&prm.tm_q, ws.qc, dims.D, dims.Hq, static_cast<uint64_t>(cap) + kBM, 1, 64, qrows) ||
        !encode_bf16_4d(&prm.tm_do, ws.doc, dims.D, dims.Hq, static_cast<uint64_t>(cap) + kBM, 1, 64, qrows) ||
        !encode_bf16_4d(&prm.tm_k, k, dims.D, dims.Hkv, dims.T, dims.B, 64, kBN) ||
        !encode_bf16_4d(&prm.tm_v, v, dims.D, dims.Hkv, dims.T, dims.B, 64, kBN) ||
        (dims.D == 64 &&
         !encode_f32_4d(&prm.tm_dq, ws.dq_acc, dims.D, dims.Hq, static_cast<uint64_t>(cap) + kBM, 1, 32, 32)))
        return LOGO_ERR_CUDA;
    prm.lse = lse_c;
    prm.dsum = ws.dsum;
    prm.dq_acc = ws.dq_acc;
    prm.dk = dk;
    prm.dv = dv;
    prm.pos = pos;
    prm.cu_q = cu_q;
    prm.first_row = ws.first_row;
    prm.dq_fill = dq;
    prm.B = dims.B;
    prm.T = dims.T;
    prm.Hq = dims.Hq;
    prm.Hkv = dims.Hkv;
    prm.window = kNoWindow;
    prm.cap = cap;
    prm.nblk = (dims.T + kBN - 1) / kBN;
    prm.scale = scale;
    prm.scale_log2 = scale * kLog2e;
    rc = dims.D == 128 ? launch_bwd<128, true>(prm, st) : launch_bwd<64, true>(prm, st);
    if (rc != LOGO_OK) return rc;
    bwd_post_selected_kernel<<<grid_rows, 128, 0, st>>>(ws.dq_acc, pos, cu_q, n_sel_total, dims.B, dims.T, dims.Hq,
                                                        dims.D, dq);
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}
