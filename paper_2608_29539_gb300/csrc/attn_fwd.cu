// attn_fwd.cu -- forward of both attention branches on tcgen05 tensor cores.
//
//   logo_local_attn_fwd          O^L = SoftmaxAttn_W(Q^L, K^L, V^L)   (Eq. 6)
//   logo_global_sparse_attn_fwd  O^G_I = SoftmaxAttn_inf(Q^G_I, K^G, V^G) (Eq. 8)
//
// One persistent kernel template serves both.  A CTA (16 warps) loops over
// work items = (128-row query tile, query head):
//   warp 12     TMA producer: Q tile once per item, then K blocks through a
//               ring of shared-memory stages (128-byte swizzle)
//   warp 15     V blocks through a ring of their own
//   warp 13     S issuer (one thread): S = Q K^T into one of two TMEM S buffers
//   warp 14     P.V issuer (one thread): O += P V into the TMEM O accumulator
//               with P read straight from TMEM.  Two issuing threads keep the
//               tensor pipe fed while either waits for its inputs: the issue
//               queue is short, so a single thread that stops to wait starves
//               the pipe (measured: 1728 vs 2427 TFLOP/s on the same MMA stream).
//   warps 0..3  softmax of the even KV blocks (S and P buffer 0), warps 4..7 of
//               the odd ones (buffer 1); one thread per query row (its TMEM
//               lane).  Online softmax in the log2 domain with conditional
//               rescaling of O (only when the running max grows by more than
//               2^8); P goes back to TMEM as bf16 pairs.  The running max is
//               the one thing the blocks of a row share: the thread of block n
//               reads the one block n-1 left in shared memory, right after its
//               own row max, and leaves its own there before the exponentials,
//               so the two warpgroups run half a block apart.  Each keeps the
//               row sum of its own blocks.  One warpgroup for every block made
//               its own latencies (barriers, TMEM round trips, ~2700 clocks a
//               block with masks) the period; with two, measured at 16K (32
//               heads, d 128) local 275 -> 236 us and global 242 -> 223 us, at
//               8K (2 x 16 heads, d 64) local 140 -> 105 us.  What is left is
//               ~1600 clocks a block against ~1350 of the same kernel without
//               any softmax arithmetic.
//   warps 8..11 epilogue: the two row sums combined, O out of TMEM once an
//               item's last P.V is done, normalised and stored while the
//               softmax warps are on the next item.
// The KV blocks of an item are only those some row can see; blocks where
// every row sees every key skip the per-element predicate (App. B's
// three-region traversal; for the local branch the window edge is a second
// masked region), and inside a masked block only the 32-key groups a row
// sees in part are tested key by key.  Global items come from a schedule
// ordered by cost (longest first) that one block of the kernel before builds on
// the device, so nothing here needs the selected count on the host.
#include <cuda_bf16.h>

#include <cstdint>

#include "attn_common.cuh"
#include "host_common.h"
#include "sm100.cuh"

namespace logo {
namespace {

template <int D>
struct FwdCfg {
    static constexpr int kSub = D / 64;             // 64-column (128-byte) sub-tiles per row
    static constexpr int kTileBytes = kBM * D * 2;  // one Q / K / V tile
    // K and V are two rings with a producer each: a K stage is free once S of
    // its block is done, a V stage once P.V is.  (One ring whose stage holds K
    // and V of a block made S of block n + 3 wait for P.V of block n: with two
    // softmax warpgroups that chain, not the tensor pipe, set the local
    // branch's period.)  Three stages each at d = 128.
    // d = 64 has the shared memory for six stages, and for a second Q buffer,
    // so that an item's Q lands while the item before is computed.
    static constexpr int kStages = D == 64 ? 6 : 3;
    static constexpr int kQBufs = D == 64 ? 2 : 1;
    static constexpr int kOffQ = 0;
    static constexpr int kOffK = kOffQ + kQBufs * kTileBytes;
    static constexpr int kOffV = kOffK + kStages * kTileBytes;
    // the dynamic array is declared with the tiles' 1024-byte alignment, so it
    // starts at the kernel's (at most 3 KB of) static shared memory rounded up
    static constexpr int kSmemBytes = kOffV + kStages * kTileBytes;
    // O accumulator (D columns, fp32); d = 64 has room for two, used in turn by
    // the items, so that an item's first P.V never waits for the epilogue
    static constexpr int kOBufs = D == 64 ? 2 : 1;
    static constexpr uint32_t kColO = 0;
    static constexpr uint32_t kColS0 = 128;  // S buffers (128 columns, fp32)
    static constexpr uint32_t kColS1 = 256;
    static constexpr uint32_t kColP0 = 384;  // P buffers (128 keys as bf16 pairs: 64 columns)
    static constexpr uint32_t kColP1 = 448;
    static constexpr uint32_t kTmemCols = 512;
    // 16 warps: softmax of even and of odd blocks (0..3, 4..7), epilogue
    // (8..11), Q/K producer, S issuer, P.V issuer, V producer (12..15).  Launched at 128 registers a thread (512 x 128 =
    // 65,536); the softmax warpgroups take 184 (a row of S lives in
    // registers; spills cost more than anything else here, as they miss the
    // few KB of L1 that the tiles leave), the epilogue 96, the control warps 48:
    // 128 x (184 + 184 + 96 + 48) = 65,536.
    static constexpr int kThreads = 512;
    static constexpr uint32_t kRegsSoftmax = 184;
    static constexpr uint32_t kRegsEpilogue = 96;
    static constexpr uint32_t kRegsControl = 48;
};

// Division of 0 <= n < 2^31 by a fixed d: n / d = (n m) >> (31 + l) with
// l = ceil(log2 d), m = ceil(2^(31+l) / d) < 2^32 (Granlund and Montgomery,
// "Division by invariant integers using multiplication").
struct FastDiv {
    uint32_t m, l;
    int d;
    FastDiv(int div = 1) : d(div)
    {
        l = 0;
        while ((1ll << l) < div) ++l;
        m = static_cast<uint32_t>(((1ull << (31 + l)) + div - 1) / div);
    }
    __device__ __forceinline__ int div(int n) const
    {
        return static_cast<int>(__umulhi(static_cast<uint32_t>(n) << 1, m) >> l);
    }
};

struct FwdParams {
    CUtensorMap tm_q;  // local: Q [B,T,Hq,D]; global: packed Qc [1,cap+128,Hq,D]
    CUtensorMap tm_k;  // [B,T,Hkv,D]
    CUtensorMap tm_v;
    logo_bf16* o;      // local: [B,T,Hq,D]; global: packed [cap,Hq,D]
    float* lse;        // local: [B,Hq,T];   global: [Hq,cap]
    const int32_t* pos;            // global: packed positions
    const GlobalTile* tiles;       // global: schedule
    const int32_t* n_tiles;        // global: schedule length (device)
    int32_t* next_item;            // global: work counter, zeroed by the schedule kernel
    float* o_part;                 // global split entries: unnormalised O [slot * Hq + h][D][128]
    float* m_part;                 // ... their running max (log2 units) [slot * Hq + h][128]
    float* l_part;                 // ... and their row sums
    int B, T, Hq, Hkv, window, cap;
    int q_tiles;                   // local: query tiles per sequence
    FastDiv by_hq, by_group, by_q_tiles;  // Hq, Hq / Hkv, q_tiles: every role decodes every item
    float scale_log2;              // softmax scale * log2(e)
};

template <bool GLOBAL>
__device__ __forceinline__ FwdItem decode_item(const FwdParams& p, int k)
{
    FwdItem it;
    const int tile = p.by_hq.div(k);
    it.h = k - tile * p.Hq;
    it.kvh = p.by_group.div(it.h);
    if (!GLOBAL) {
        it.b = p.by_q_tiles.div(tile);
        const int qt = tile - it.b * p.q_tiles;
        it.row0 = qt * kBM;
        it.nrows = min(kBM, p.T - it.row0);
        it.pos_min = it.row0;
        it.pos_max = it.row0 + it.nrows - 1;
        it.blk_lo = max(0, it.pos_min - p.window + 1) / kBN;
        it.blk_hi = it.pos_max / kBN;
        it.slot = -1;
    } else {
        const GlobalTile g = p.tiles[tile];
        it.b = g.b;
        it.row0 = g.row0;
        it.nrows = g.nrows;
        it.pos_min = g.min_pos;
        it.pos_max = g.max_pos;
        it.blk_lo = g.blk_lo;
        it.blk_hi = g.blk_hi;
        it.slot = g.slot;
    }
    return it;
}

// Visibility inside one 128-key block: the row sees keys c with lo <= c <= hi;
// every other s[c] becomes -inf.  One 32-bit mask per 32 keys, whose bits
// become the predicates of the selects: straight-line code, a select per key
// and nothing per key to compare.  (Sorting the groups of 32 into seen whole,
// unseen and cut, with a loop for each, was fewer instructions and took
// 1100-2300 clocks a masked block against 300-500 of an unmasked one: its
// branches ran from cold instruction cache.)
__device__ __forceinline__ void mask_row_block(float (&s)[kBN], int lo, int hi)
{
#pragma unroll
    for (int g = 0; g < kBN / 32; ++g) {
        const uint32_t m = column_mask(lo - 32 * g, hi - 32 * g);
#pragma unroll
        for (int i = 0; i < 32; ++i) s[32 * g + i] = (m & (1u << i)) ? s[32 * g + i] : -INFINITY;
    }
}

template <int D, bool GLOBAL>
__global__ void __launch_bounds__(512, 1) attn_fwd_kernel(const __grid_constant__ FwdParams p)
{
    using C = FwdCfg<D>;
    static_assert(128 * (2 * C::kRegsSoftmax + C::kRegsEpilogue + C::kRegsControl) <= 512 * 128,
                  "register split exceeds the launch allocation");
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar_q_full[C::kQBufs], bar_q_empty[C::kQBufs], bar_drain, bar_drain_pv;
    __shared__ __align__(8) uint64_t bar_k_full[C::kStages], bar_k_empty[C::kStages];
    __shared__ __align__(8) uint64_t bar_v_full[C::kStages], bar_v_empty[C::kStages];
    __shared__ __align__(8) uint64_t bar_s_full[2], bar_s_empty[2], bar_p_full[2];
    // P.V of block n done, for the softmax: barrier n % 2.  Its waits, for n - 2
    // and then perhaps n - 1, are made at block n: the phases before are known to
    // have ended, the ones after need block n's P.  For the epilogue, P.V of an
    // item's last block done: a barrier per O buffer, whose next phase needs that
    // buffer's bar_o_free.  (It cannot wait on bar_pv_done: with two O buffers
    // the next item's products go on beside it and end later phases.)
    __shared__ __align__(8) uint64_t bar_pv_done[2], bar_o_full[C::kOBufs];
    // running max of every row after the newest block, handed from one softmax
    // warpgroup's thread of the row to the other's (so one copy is enough): a
    // barrier per warp and block parity
    __shared__ __align__(8) uint64_t bar_m[2][4];
    __shared__ float sh_m[kBM];
    // softmax -> epilogue: max and sum of every row of an item over the even
    // and over the odd blocks, and O's columns free again once the epilogue
    // has copied them out
    __shared__ __align__(8) uint64_t bar_l_full, bar_l_empty, bar_o_free[C::kOBufs];
    __shared__ float2 sh_ml[2][kBM];
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_flag;
    // global branch: items are taken dynamically (longest first, whichever CTA
    // is free next); the producer passes each index to the other roles
    // through this 4-slot ring (-1 ends the work)
    __shared__ volatile int item_ring[4];
    __shared__ __align__(8) uint64_t bar_item_full[4], bar_item_empty[4];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sQ = smem_u32(smem + C::kOffQ);
    const uint32_t sK = smem_u32(smem + C::kOffK);
    const uint32_t sV = smem_u32(smem + C::kOffV);

    if (smem_u32(smem) & 1023u) {  // (uniform) the swizzled tiles need the alignment asked for
        record_status(LOGO_ERR_CUDA);
        return;
    }
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < C::kQBufs; ++s) {
            mbar_init(smem_u32(&bar_q_full[s]), 1);
            mbar_init(smem_u32(&bar_q_empty[s]), 1);
        }
        mbar_init(smem_u32(&bar_drain), 1);
        mbar_init(smem_u32(&bar_drain_pv), 1);
        for (int s = 0; s < C::kStages; ++s) {
            mbar_init(smem_u32(&bar_k_full[s]), 1);
            mbar_init(smem_u32(&bar_k_empty[s]), 1);
            mbar_init(smem_u32(&bar_v_full[s]), 1);
            mbar_init(smem_u32(&bar_v_empty[s]), 1);
        }
        for (int s = 0; s < 4; ++s) {
            mbar_init(smem_u32(&bar_item_full[s]), 1);
            // the V producer, the two MMA threads, one lane per softmax / epilogue warp
            mbar_init(smem_u32(&bar_item_empty[s]), 15);
            mbar_init(smem_u32(&bar_m[0][s]), 1);
            mbar_init(smem_u32(&bar_m[1][s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bar_s_full[s]), 1);
            mbar_init(smem_u32(&bar_s_empty[s]), 128);
            mbar_init(smem_u32(&bar_p_full[s]), 128);
            mbar_init(smem_u32(&bar_pv_done[s]), 1);
        }
        mbar_init(smem_u32(&bar_l_full), 256);
        mbar_init(smem_u32(&bar_l_empty), 128);
        for (int s = 0; s < C::kOBufs; ++s) {
            mbar_init(smem_u32(&bar_o_full[s]), 1);
            mbar_init(smem_u32(&bar_o_free[s]), 128);
        }
        fence_mbar_init();
    }
    if (warp == 13) {
        tmem_alloc(smem_u32(&tmem_base_sh), C::kTmemCols);
        tmem_relinquish();
    }
    const int n_items = GLOBAL ? (*p.n_tiles) * p.Hq : p.B * p.q_tiles * p.Hq;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;

    // u-th work item of this CTA for a consumer role, or -1 when done.
    // whole_warp: called by all 32 lanes (the softmax warps), which then
    // arrive once per warp; otherwise by the single MMA-issuing thread.
    auto consume_item = [&](int u, bool* ok, bool whole_warp) -> int {
        if (!GLOBAL) {
            const int k = blockIdx.x + u * gridDim.x;
            return k < n_items ? k : -1;
        }
        const int slot = u & 3;
        const uint32_t full = smem_u32(&bar_item_full[slot]), turn = (u >> 2) & 1;
        *ok = whole_warp ? mbar_wait_warp(full, turn, &abort_flag) : mbar_wait(full, turn, &abort_flag);
        if (!*ok) return -1;
        const int k = item_ring[slot];
        if (whole_warp) {
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_item_empty[slot]));
        } else {
            mbar_arrive(smem_u32(&bar_item_empty[slot]));
        }
        return k;
    };

    if (warp >= 12) {
        // ------------------------------------------------------------ control warps
        setmaxnreg_dec<C::kRegsControl>();
    if (warp == 12) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            tma_prefetch_desc(&p.tm_q);
            tma_prefetch_desc(&p.tm_k);
            tma_prefetch_desc(&p.tm_v);
            const uint64_t pol_q = policy_evict_first();
            const uint64_t pol_kv = policy_evict_last();
            int kv_it = 0, item_i = 0;
            int last_fill[C::kStages];
            for (int s = 0; s < C::kStages; ++s) last_fill[s] = -1;
            int q_fills = 0;
            bool ok = true;
            for (;; ++item_i) {
                int k;
                if (GLOBAL) {
                    const int slot = item_i & 3;
                    if (!(ok = mbar_wait(smem_u32(&bar_item_empty[slot]), ((item_i >> 2) & 1) ^ 1, &abort_flag))) break;
                    k = atomicAdd(p.next_item, 1);
                    if (k >= n_items) k = -1;
                    item_ring[slot] = k;
                    mbar_arrive(smem_u32(&bar_item_full[slot]));
                } else {
                    k = blockIdx.x + item_i * gridDim.x;
                    if (k >= n_items) k = -1;
                }
                if (k < 0) break;
                const FwdItem it = decode_item<GLOBAL>(p, k);
                const int qs = item_i % C::kQBufs, qf = item_i / C::kQBufs;
                if (!(ok = mbar_wait(smem_u32(&bar_q_empty[qs]), (qf & 1) ^ 1, &abort_flag))) break;
                const uint32_t qb = smem_u32(&bar_q_full[qs]);
                mbar_arrive_expect_tx(qb, C::kTileBytes);
                for (int s = 0; s < C::kSub; ++s)
                    tma_load_4d(sQ + qs * C::kTileBytes + s * 16384, &p.tm_q, qb, 64 * s, it.h, it.row0, GLOBAL ? 0 : it.b, pol_q);
                ++q_fills;
                if (!GLOBAL && C::kQBufs == 1 && k + gridDim.x < n_items) {
                    // one Q buffer: the next item's Q can only be copied once S of
                    // this item's last block is done, so bring it as far as L2 now
                    const FwdItem nx = decode_item<GLOBAL>(p, k + gridDim.x);
                    for (int s = 0; s < C::kSub; ++s) tma_prefetch_4d(&p.tm_q, 64 * s, nx.h, nx.row0, nx.b);
                }
                for (int n = it.blk_lo; n <= it.blk_hi; ++n, ++kv_it) {
                    const int st = kv_it % C::kStages, f = kv_it / C::kStages;
                    if (!(ok = mbar_wait(smem_u32(&bar_k_empty[st]), (f & 1) ^ 1, &abort_flag))) break;
                    const uint32_t kb = smem_u32(&bar_k_full[st]);
                    mbar_arrive_expect_tx(kb, C::kTileBytes);
                    for (int s = 0; s < C::kSub; ++s)
                        tma_load_4d(sK + st * C::kTileBytes + s * 16384, &p.tm_k, kb, 64 * s, it.kvh, n * kBN, it.b,
                                    pol_kv);
                    last_fill[st] = f;
                }
                if (!ok) break;
            }
            if (!ok) {  // let copies already issued land before the CTA exits
                for (int i = max(0, q_fills - C::kQBufs); i < q_fills; ++i)
                    mbar_wait_drain(smem_u32(&bar_q_full[i % C::kQBufs]), (i / C::kQBufs) & 1);
                for (int s = 0; s < C::kStages; ++s)
                    if (last_fill[s] >= 0) mbar_wait_drain(smem_u32(&bar_k_full[s]), last_fill[s] & 1);
            }
        }
    } else if (warp == 13) {
        // ------------------------------------------------------------ S issuer
        // S = Q K^T of every block; the P.V products come from warp 14, so that
        // neither stream's waits leave the tensor pipe without queued work
        // (the issue queue is short: an issuing thread runs only a few
        // instructions ahead of execution)
        if (lane == 0) {
            constexpr uint32_t idS = idesc_bf16_f32(kBM, kBN, false, false);
            int kv_it = 0, s_it = 0, item_i = 0;
            bool ok = true;
            for (;; ++item_i) {
                const int k = consume_item(item_i, &ok, false);
                if (k < 0) break;
                const FwdItem it = decode_item<GLOBAL>(p, k);
                const int nblk = it.blk_hi - it.blk_lo + 1;
                const int qs = item_i % C::kQBufs;
                const uint32_t qbase = sQ + qs * C::kTileBytes;
                if (!(ok = mbar_wait(smem_u32(&bar_q_full[qs]), (item_i / C::kQBufs) & 1, &abort_flag))) break;
                for (int j = 0; j < nblk && ok; ++j) {
                    const int itg = s_it + j;
                    const int st = (kv_it + j) % C::kStages, f = (kv_it + j) / C::kStages;
                    const int buf = itg & 1, use = itg >> 1;
                    if (!(ok = mbar_wait(smem_u32(&bar_k_full[st]), f & 1, &abort_flag))) break;
                    if (!(ok = mbar_wait(smem_u32(&bar_s_empty[buf]), (use & 1) ^ 1, &abort_flag))) break;
                    tc_fence_after();
                    const uint32_t kbase = sK + st * C::kTileBytes;
                    const uint32_t dcol = tmem + (buf ? C::kColS1 : C::kColS0);
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        const uint32_t off = (ks >> 2) * 16384 + (ks & 3) * 32;
                        umma_bf16_ss(dcol, sdesc_sw128(qbase + off, 16, 1024), sdesc_sw128(kbase + off, 16, 1024), idS,
                                     ks > 0 ? 1u : 0u);
                    }
                    umma_commit(smem_u32(&bar_s_full[buf]));
                    umma_commit(smem_u32(&bar_k_empty[st]));  // K of this block is read
                }
                if (!ok) break;
                umma_commit(smem_u32(&bar_q_empty[qs]));
                kv_it += nblk;
                s_it += nblk;
            }
            if (!ok) {  // wait for MMAs in flight before TMEM is released
                umma_commit(smem_u32(&bar_drain));
                mbar_wait_drain(smem_u32(&bar_drain), 0);
            }
        }
    } else if (warp == 14) {
        // ------------------------------------------------------------ P.V issuer
        if (lane == 0) {
            constexpr uint32_t idPV = idesc_bf16_f32(kBM, D, false, true);
            int kv_it = 0, s_it = 0, item_i = 0;
            bool ok = true;
            for (;; ++item_i) {
                const int k = consume_item(item_i, &ok, false);
                if (k < 0) break;
                const FwdItem it = decode_item<GLOBAL>(p, k);
                const int nblk = it.blk_hi - it.blk_lo + 1;
                const int ob = item_i % C::kOBufs;
                const uint32_t ocol = tmem + C::kColO + ob * D;
                for (int j = 0; j < nblk && ok; ++j) {
                    const int itg = s_it + j;
                    const int st = (kv_it + j) % C::kStages, f = (kv_it + j) / C::kStages;
                    if (!(ok = mbar_wait(smem_u32(&bar_p_full[itg & 1]), (itg >> 1) & 1, &abort_flag))) break;
                    if (!(ok = mbar_wait(smem_u32(&bar_v_full[st]), f & 1, &abort_flag))) break;
                    // the item's first P.V overwrites O: the epilogue warps have
                    // copied the previous item's O out of TMEM
                    if (j == 0 && !(ok = mbar_wait(smem_u32(&bar_o_free[ob]), ((item_i / C::kOBufs) & 1) ^ 1, &abort_flag)))
                        break;
                    tc_fence_after();
                    const uint32_t vbase = sV + st * C::kTileBytes;
                    const uint32_t pcol = tmem + ((itg & 1) ? C::kColP1 : C::kColP0);
#pragma unroll
                    for (int ks = 0; ks < kBN / 16; ++ks) {
                        const uint64_t bdesc = sdesc_sw128(vbase + ks * 2048, 16384, 1024);
                        umma_bf16_ts(ocol, pcol + ks * 8, bdesc, idPV, (j > 0 || ks > 0) ? 1u : 0u);
                    }
                    umma_commit(smem_u32(&bar_pv_done[itg & 1]));
                    umma_commit(smem_u32(&bar_v_empty[st]));  // V of this block is read
                }
                if (!ok) break;
                umma_commit(smem_u32(&bar_o_full[ob]));
                kv_it += nblk;
                s_it += nblk;
            }
            if (!ok) {
                umma_commit(smem_u32(&bar_drain_pv));
                mbar_wait_drain(smem_u32(&bar_drain_pv), 0);
            }
        }
    } else {
        // ------------------------------------------------------------ V producer
        // V blocks through their own ring (a stage is freed by the P.V that
        // read it), so a V load never holds up the next K load
        if (lane == 0) {
            const uint64_t pol_kv = policy_evict_last();
            int kv_it = 0;
            int last_fill[C::kStages];
            for (int s = 0; s < C::kStages; ++s) last_fill[s] = -1;
            bool ok = true;
            for (int item_i = 0;; ++item_i) {
                const int k = consume_item(item_i, &ok, false);
                if (k < 0) break;
                const FwdItem it = decode_item<GLOBAL>(p, k);
                for (int n = it.blk_lo; n <= it.blk_hi; ++n, ++kv_it) {
                    const int st = kv_it % C::kStages, f = kv_it / C::kStages;
                    if (!(ok = mbar_wait(smem_u32(&bar_v_empty[st]), (f & 1) ^ 1, &abort_flag))) break;
                    const uint32_t vb = smem_u32(&bar_v_full[st]);
                    mbar_arrive_expect_tx(vb, C::kTileBytes);
                    for (int s = 0; s < C::kSub; ++s)
                        tma_load_4d(sV + st * C::kTileBytes + s * 16384, &p.tm_v, vb, 64 * s, it.kvh, n * kBN, it.b,
                                    pol_kv);
                    last_fill[st] = f;
                }
                if (!ok) break;
            }
            if (!ok) {  // let copies already issued land before the CTA exits
                for (int s = 0; s < C::kStages; ++s)
                    if (last_fill[s] >= 0) mbar_wait_drain(smem_u32(&bar_v_full[s]), last_fill[s] & 1);
            }
        }
    }
    } else if (warp < 8) {
        // ------------------------------------------------------------ softmax
        setmaxnreg_inc<C::kRegsSoftmax>();
        const int par = warp >> 2;  // this warpgroup takes the blocks with itg % 2 == par
        const int quad = warp & 3;  // TMEM lane quadrant this warp may access
        const int r = quad * 32 + lane;
        const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
        const uint32_t scol = tmem + lane_off + (par ? C::kColS1 : C::kColS0);
        const uint32_t pcol = tmem + lane_off + (par ? C::kColP1 : C::kColP0);
        const uint32_t bar_m_mine = smem_u32(&bar_m[par][quad]), bar_m_other = smem_u32(&bar_m[par ^ 1][quad]);
        int itg0 = 0;  // KV blocks of the items before this one
        bool ok = true;
        for (int item_i = 0;; ++item_i) {
            const int k = consume_item(item_i, &ok, true);
            if (k < 0) break;
            // all that the loop below keeps of the item: its blocks, the ones that
            // every row sees whole (open_lo .. open_hi), and this row's position
            int nblk, blk_lo, open_lo, open_hi, mypos;
            {
                const FwdItem it = decode_item<GLOBAL>(p, k);
                blk_lo = it.blk_lo;
                nblk = it.blk_hi - it.blk_lo + 1;
                open_hi = (it.pos_min + 1) / kBN - 1;
                open_lo = GLOBAL || it.pos_max < p.window ? 0 : (it.pos_max - p.window) / kBN + 1;
                const bool row_valid = r < it.nrows;
                if (GLOBAL) mypos = row_valid ? p.pos[it.row0 + r] : it.pos_max;
                else mypos = row_valid ? it.row0 + r : it.pos_max;
            }
            // The barriers a block waits on are nearly always complete by then; each
            // is tested (non-blocking) well before, so that the test's latency
            // overlaps other work, and only a warp that found one open waits.
            bool s_seen = false;  // S of the next block
            float m_own = -INFINITY;  // running max (log2 domain) this warpgroup's row sum is relative to
            float l = 0.f;
#pragma unroll 1
            for (int j = (itg0 ^ par) & 1; j < nblk; j += 2) {
                const int itg = itg0 + j, n = blk_lo + j;
                if (!__all_sync(0xffffffffu, s_seen)) {
                    // (the __syncwarp here and at the waits below: without any, the
                    // allocator spills 40 bytes of the row of S)
                    ok = mbar_wait_warp(smem_u32(&bar_s_full[par]), (itg >> 1) & 1, &abort_flag);
                    __syncwarp();
                    if (!ok) break;
                }
                tc_fence_after();
                float s[kBN];
                {
                    uint32_t v[kBN / 32][32];
#pragma unroll
                    for (int c = 0; c < kBN / 32; ++c) tmem_ld32(scol + c * 32, v[c]);
                    tmem_wait_ld();  // one wait for all four loads
#pragma unroll
                    for (int c = 0; c < kBN / 32; ++c)
#pragma unroll
                        for (int i = 0; i < 32; ++i) s[c * 32 + i] = __uint_as_float(v[c][i]);
                }
                tc_fence_before();
                mbar_arrive(smem_u32(&bar_s_empty[par]));
                const bool m_seen = itg == 0 || mbar_test(bar_m_other, ((itg - 1) >> 1) & 1);
                float m_ref = sh_m[r];  // (of no use unless m_seen)
                if (n < open_lo || n > open_hi)
                    mask_row_block(s, GLOBAL ? -1 : mypos - p.window + 1 - n * kBN, mypos - n * kBN);
                // 4 independent 3-input max chains and 4 packed-pair sums keep
                // dependency chains short; exp arguments are formed two at a
                // time with f32x2 FMAs
                float mx4[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
                for (int c = 4; c < kBN; c += 8) {
                    mx4[0] = max3f(mx4[0], s[c], s[c + 1]);
                    mx4[1] = max3f(mx4[1], s[c + 2], s[c + 3]);
                    if (c + 4 < kBN) {
                        mx4[2] = max3f(mx4[2], s[c + 4], s[c + 5]);
                        mx4[3] = max3f(mx4[3], s[c + 6], s[c + 7]);
                    }
                }
                const float mx = max3f(mx4[0], mx4[1], fmaxf(mx4[2], mx4[3]));
                // the running max after the block before.  Waited for across an
                // item's edge too (its value does not count there), so that the
                // two warpgroups' phases on these barriers never drift apart
                if (!__all_sync(0xffffffffu, m_seen)) {
                    ok = mbar_wait_warp(bar_m_other, ((itg - 1) >> 1) & 1, &abort_flag);
                    __syncwarp();
                    if (!ok) break;
                    m_ref = sh_m[r];
                }
                if (j == 0) m_ref = -INFINITY;
                const float m_new = fmaxf(m_ref, mx * p.scale_log2);
                float alpha = 1.f;
                bool rescale = false;
                if (m_new > m_ref + 8.0f) {  // also taken when m_ref is still -inf
                    // a row that has seen no key yet has P = 0 behind it: its O
                    // needs no scaling (the window's last rows at an item's second
                    // block, where the wait for P.V would stop their warp each time)
                    rescale = m_ref != -INFINITY;
                    if (rescale) alpha = ex2_approx(m_ref - m_new);
                    m_ref = m_new;
                }
                sh_m[r] = m_ref;
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_m_mine);
                // (global branch only: the local one has no register left for it)
                const bool pv_seen =
                    itg < 2 || (GLOBAL && mbar_test(smem_u32(&bar_pv_done[(itg - 2) & 1]), ((itg - 2) >> 1) & 1));
                const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;
                const uint64_t scale2 = f2_pack(p.scale_log2, p.scale_log2);
                const uint64_t negm2 = f2_pack(-m_use, -m_use);
                uint64_t acc2[4] = {0ull, 0ull, 0ull, 0ull};
                uint32_t pk[2][32];  // P as bf16 pairs
#pragma unroll
                for (int c = 0; c < kBN; c += 2) {
                    float x0, x1;
                    f2_unpack(f2_fma(f2_pack(s[c], s[c + 1]), scale2, negm2), x0, x1);
                    x0 = ex2_approx(x0);
                    x1 = ex2_approx(x1);
                    acc2[(c >> 1) & 3] = f2_add(acc2[(c >> 1) & 3], f2_pack(x0, x1));
                    pk[c >> 6][(c >> 1) & 31] = cvt_bf16x2(x0, x1);
                }
                float rs;
                {
                    float a0, a1, b0, b1, c0, c1, d0, d1;
                    f2_unpack(acc2[0], a0, a1);
                    f2_unpack(acc2[1], b0, b1);
                    f2_unpack(acc2[2], c0, c1);
                    f2_unpack(acc2[3], d0, d1);
                    rs = ((a0 + a1) + (b0 + b1)) + ((c0 + c1) + (d0 + d1));
                }
                if (m_ref > m_own) {  // by this block or by one of the other warpgroup's
                    l *= ex2_approx(m_own - m_ref);
                    m_own = m_ref;
                }
                l += rs;
                // the P buffer is free once the P.V two blocks back is done
                if (!__all_sync(0xffffffffu, pv_seen)) {
                    ok = mbar_wait_warp(smem_u32(&bar_pv_done[(itg - 2) & 1]), ((itg - 2) >> 1) & 1, &abort_flag);
                    __syncwarp();
                    if (!ok) break;
                }
                tc_fence_after();
#pragma unroll
                for (int h = 0; h < 2; ++h) tmem_st32(pcol + 32 * h, pk[h]);
                // O may only be rescaled once the P.V of the previous block is done.
                // Done here, where the row of S no longer takes registers
                if (__any_sync(0xffffffffu, rescale)) {
                    ok = mbar_wait_warp(smem_u32(&bar_pv_done[(itg - 1) & 1]), ((itg - 1) >> 1) & 1, &abort_flag);
                    __syncwarp();
                    if (!ok) break;
                    tc_fence_after();
                    // tcgen05.ld/st are warp-collective: rows that keep their max
                    // multiply by alpha = 1
                    const uint32_t ocol = tmem + lane_off + C::kColO + (item_i % C::kOBufs) * D;
#pragma unroll 1
                    for (int c = 0; c < D / 32; ++c) {
                        uint32_t v[32];
                        tmem_ld32(ocol + c * 32, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * alpha);
                        tmem_st32(ocol + c * 32, v);
                    }
                }
                s_seen = j + 2 < nblk && mbar_test(smem_u32(&bar_s_full[par]), ((itg + 2) >> 1) & 1);
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(smem_u32(&bar_p_full[par]));
            }
            if (!ok) break;
            itg0 += nblk;
            // ---- end of the item: this warpgroup's max and row sum to the epilogue warps
            ok = mbar_wait_warp(smem_u32(&bar_l_empty), (item_i & 1) ^ 1, &abort_flag);
            if (!ok) break;
            sh_ml[par][r] = make_float2(m_own, l);
            mbar_arrive(smem_u32(&bar_l_full));
        }
    } else {
        // ------------------------------------------------------------ epilogue
        // warps 8..11: the row's max and sum from the two softmax warpgroups;
        // once an item's last P.V is done, O out of TMEM (then the next item's
        // first P.V may overwrite it), and O / l and lse = (m + log2 l) ln 2 to
        // memory (or, for one share of a split KV range, the unnormalised O, the
        // max and the row sum)
        setmaxnreg_dec<C::kRegsEpilogue>();
        const int quad = warp & 3;
        const int r = quad * 32 + lane;
        const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
        bool ok = true;
        for (int item_i = 0;; ++item_i) {
            const int k = consume_item(item_i, &ok, true);
            if (k < 0) break;
            const FwdItem it = decode_item<GLOBAL>(p, k);
            const bool row_valid = r < it.nrows;
            ok = mbar_wait_warp(smem_u32(&bar_l_full), item_i & 1, &abort_flag);
            if (!ok) break;
            const float2 ml0 = sh_ml[0][r], ml1 = sh_ml[1][r];
            mbar_arrive(smem_u32(&bar_l_empty));
            const float m = fmaxf(ml0.x, ml1.x);
            const float l = (ml0.x == -INFINITY ? 0.f : ml0.y * ex2_approx(ml0.x - m)) +
                            (ml1.x == -INFINITY ? 0.f : ml1.y * ex2_approx(ml1.x - m));
            const bool whole = !GLOBAL || it.slot < 0;
            const int64_t unit = static_cast<int64_t>(it.slot) * p.Hq + it.h;  // split entries only
            if (row_valid) {
                if (whole) {
                    const float lse = (m + log2f(l)) * kLn2;
                    if (GLOBAL) p.lse[static_cast<int64_t>(it.h) * p.cap + it.row0 + r] = lse;
                    else p.lse[(static_cast<int64_t>(it.b) * p.Hq + it.h) * p.T + it.row0 + r] = lse;
                } else {
                    p.m_part[unit * kBM + r] = m;
                    p.l_part[unit * kBM + r] = l;
                }
            }
            const float inv_l = 1.0f / l;
            float inv[2][2];
#pragma unroll
            for (int i = 0; i < 4; ++i) inv[i >> 1][i & 1] = __shfl_sync(0xffffffffu, inv_l, i * 8 + (lane >> 2));
            // the item's last P.V is done
            const int ob = item_i % C::kOBufs;
            ok = mbar_wait_warp(smem_u32(&bar_o_full[ob]), (item_i / C::kOBufs) & 1, &abort_flag);
            if (!ok) break;
            tc_fence_after();
            const uint32_t ocol = tmem + lane_off + C::kColO + ob * D;
            // this lane's 16-byte column slice of the warp's first row
            logo_bf16* o0 = p.o + ((GLOBAL ? 0 : static_cast<int64_t>(it.b) * p.T) + it.row0 + quad * 32) * p.Hq * D +
                            it.h * D + (lane & 3) * 8;
            if (!whole) {
                // one share of a split KV range: unnormalised O, stored transposed
                // ([d][row]) so that the warp's 32 rows of a column are one line
                float* pcol = p.o_part + unit * kBM * D + r;
#pragma unroll 1
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t v[32];
                    tmem_ld32(ocol + c * 32, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i) pcol[(c * 32 + i) * kBM] = __uint_as_float(v[i]);
                }
                tc_fence_before();
                mbar_arrive(smem_u32(&bar_o_free[ob]));
                continue;
            }
            // O in 16 x 256-bit pieces (lane t: rows t / 4 and t / 4 + 8, two columns
            // of every 8), as bf16 pairs; four lanes then trade pairs so that each
            // has 8 adjacent columns, and a warp store is 8 rows of 64 contiguous
            // bytes.  With a row per lane (32 rows, 32 lines a store) the item's
            // stores held the load/store pipe for ~2000 clocks, and with it the
            // softmax warps' barriers and TMEM stores.  O's columns are given back
            // as soon as the last of them is read: the first 32 go out at once,
            // the others wait as pairs until then.
            constexpr int kEarly = 1;
            uint32_t w[D / 32][2][2][4];  // [32 columns][rows 0..15 or 16..31][row t / 4 or t / 4 + 8][pairs]
            auto load32 = [&](int c) {
                uint32_t v[2][16];
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) tmem_ld_16x256b_x4(ocol + (static_cast<uint32_t>(hf * 16) << 16) + c * 32, v[hf]);
                tmem_wait_ld();
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const float ia = inv[hf][0], ib = inv[hf][1];
#pragma unroll
                    for (int k4 = 0; k4 < 4; ++k4) {
                        const uint32_t* x = v[hf] + 4 * k4;
                        w[c][hf][0][k4] = cvt_bf16x2(__uint_as_float(x[0]) * ia, __uint_as_float(x[1]) * ia);
                        w[c][hf][1][k4] = cvt_bf16x2(__uint_as_float(x[2]) * ib, __uint_as_float(x[3]) * ib);
                    }
                }
            };
            auto store32 = [&](int c) {
#pragma unroll
                for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                    for (int ab = 0; ab < 2; ++ab) {
                        const uint4 o = quad_gather8(w[c][hf][ab], lane);
                        const int row = hf * 16 + ab * 8 + (lane >> 2);
                        if (quad * 32 + row < it.nrows)
                            *reinterpret_cast<uint4*>(o0 + static_cast<int64_t>(row) * p.Hq * D + c * 32) = o;
                    }
            };
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
                load32(c);
                if (c == D / 32 - 1) {
                    tc_fence_before();
                    mbar_arrive(smem_u32(&bar_o_free[ob]));
                }
                if (c < kEarly) store32(c);
            }
#pragma unroll
            for (int c = kEarly; c < D / 32; ++c) store32(c);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 13) {
        tc_fence_after();
        tmem_dealloc(tmem, C::kTmemCols);
    }
}

// ---------------------------------------------------------------- global prep
// Split-K of the global forward.  When the selected rows make too few work
// items to fill the GPU (query tiles x heads < 2 x SMs: small sequences, high
// sparsity), long tiles are cut into shares of their KV range, each share a
// work item of its own that leaves its unnormalised O, row max and row sum in
// a slot; merge_splits_kernel then combines the shares of each row exactly
// (rescaling each share by 2^(m_s - M) to the common max M).  At most
// kMaxPartialUnits (slot, head) pairs of partial results exist.
constexpr int kMaxPartialUnits = 1024;
constexpr int kMinSplitBlocks = 8;
constexpr int kMaxShares = 64;  // shares of one tile
// Splitting pays only when it shortens the longest item by more than the merge
// and the extra items cost (measured: about a dozen blocks' time); below this
// many blocks of gain the tiles stay whole.
constexpr int kSplitMinGainBlocks = 24;

// One block: split every sequence's packed rows into tiles of 128, split long
// tiles' KV ranges if the tiles are too few, and order the entries by their
// KV-block count, longest first.
__device__ __forceinline__ int sched_block_scan(int v, int* total, int* sh)
{
    // exclusive scan over the 1024 threads, in thread order
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const int w0 = sh[lane];
        int w = w0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        sh[lane] = w - w0;
        if (lane == 31) sh[32] = w;
    }
    __syncthreads();
    const int r = sh[warp] + x - v;
    *total = sh[32];
    __syncthreads();
    return r;
}

__device__ __forceinline__ void global_schedule(const int32_t* __restrict__ pos, const int32_t* __restrict__ cu_q, int B,
                                                int Hq, int n_sm, int32_t* __restrict__ tile_off,
                                                GlobalTile* __restrict__ unsorted, GlobalTile* __restrict__ sorted,
                                                int32_t* __restrict__ n_tiles, int32_t* __restrict__ next_item,
                                                SplitTile* __restrict__ splits, int32_t* __restrict__ n_splits)
{
    __shared__ int sh_nt, sh_chunk, sh_worth;
    __shared__ int sh_scan[33];
    __shared__ unsigned long long sh_total;
    __shared__ int sh_longest;
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int b = 0; b < B; ++b) {
            tile_off[b] = acc;
            acc += (cu_q[b + 1] - cu_q[b] + kBM - 1) / kBM;
        }
        tile_off[B] = acc;
        sh_nt = acc;
        sh_total = 0;
        sh_longest = 0;
        *next_item = 0;
    }
    __syncthreads();
    const int nt = sh_nt;
    // few tiles to fill the GPU with: split the long ones (then nt < 2 x SMs <= 1024)
    const bool split = static_cast<int64_t>(nt) * Hq < 2ll * n_sm && Hq <= kMaxPartialUnits && nt <= 1024;
    auto make_tile = [&](int t) {
        int lo = 0, hi = B - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (tile_off[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        const int b = lo, i = t - tile_off[b];
        GlobalTile g;
        g.row0 = cu_q[b] + i * kBM;
        g.nrows = min(kBM, cu_q[b + 1] - g.row0);
        g.b = b;
        g.min_pos = pos[g.row0];
        g.max_pos = pos[g.row0 + g.nrows - 1];
        g.blk_lo = 0;
        g.blk_hi = g.max_pos / kBN;
        g.slot = -1;
        g.cost = g.blk_hi + 1;
        g.pad0 = g.pad1 = g.pad2 = 0;
        return g;
    };
    int ne = nt;
    if (!split) {
        for (int t = threadIdx.x; t < nt; t += blockDim.x) unsorted[t] = make_tile(t);
        if (threadIdx.x == 0) *n_splits = 0;
    } else {
        // thread t < nt holds tile t
        GlobalTile g{};
        if (threadIdx.x < nt) {
            g = make_tile(threadIdx.x);
            atomicAdd(&sh_total, static_cast<unsigned long long>(g.cost));
            atomicMax(&sh_longest, g.cost);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            // cut only what is longer than an even share of the work per SM (the
            // longest item bounds the launch; every extra item costs a pipeline
            // restart and a partial write), in shares of at least kMinSplitBlocks
            // blocks and at most kMaxShares per tile
            const long long even = (static_cast<long long>(sh_total) * Hq + n_sm - 1) / n_sm;
            int chunk = static_cast<int>(even > kMinSplitBlocks ? even : kMinSplitBlocks);
            chunk = max(chunk, (sh_longest + kMaxShares - 1) / kMaxShares);
            sh_chunk = chunk;
            sh_worth = sh_longest - chunk >= kSplitMinGainBlocks;
        }
        __syncthreads();
    }
    if (split && !sh_worth) {  // too little to gain: the whole tiles after all
        for (int t = threadIdx.x; t < nt; t += blockDim.x) unsorted[t] = make_tile(t);
        if (threadIdx.x == 0) *n_splits = 0;
    } else if (split) {
        GlobalTile g{};
        if (threadIdx.x < nt) g = make_tile(threadIdx.x);
        // grow the shares until the split tiles fit in the partial-result slots
        const int max_slots = kMaxPartialUnits / Hq;
        int sp = 1, slots = 0;
        for (;;) {
            const int chunk = sh_chunk;
            sp = threadIdx.x < nt ? (g.cost + chunk - 1) / chunk : 0;
            sched_block_scan(sp > 1 ? sp : 0, &slots, sh_scan);
            if (slots <= max_slots) break;
            if (threadIdx.x == 0) sh_chunk = chunk * 2;
            __syncthreads();
        }
        int n_entries, n_split_tiles;
        const int e0 = sched_block_scan(threadIdx.x < nt ? sp : 0, &n_entries, sh_scan);
        const int s0 = sched_block_scan(sp > 1 ? sp : 0, &slots, sh_scan);
        const int t0 = sched_block_scan(sp > 1 ? 1 : 0, &n_split_tiles, sh_scan);
        if (threadIdx.x < nt) {
            if (sp == 1) {
                unsorted[e0] = g;
            } else {
                splits[t0] = SplitTile{g.row0, g.nrows, s0, sp};
                for (int s = 0; s < sp; ++s) {
                    GlobalTile e = g;
                    e.blk_lo = static_cast<int>(static_cast<int64_t>(g.cost) * s / sp);
                    e.blk_hi = static_cast<int>(static_cast<int64_t>(g.cost) * (s + 1) / sp) - 1;
                    e.slot = s0 + s;
                    e.cost = e.blk_hi - e.blk_lo + 1;
                    unsorted[e0 + s] = e;
                }
            }
        }
        if (threadIdx.x == 0) *n_splits = n_split_tiles;
        ne = n_entries;
    }
    if (threadIdx.x == 0) *n_tiles = ne;
    __syncthreads();  // entries written
    for (int t = threadIdx.x; t < ne; t += blockDim.x) {
        const int c = unsorted[t].cost;
        int rank = 0;
        for (int u = 0; u < ne; ++u) {
            const int cu = unsorted[u].cost;
            rank += (cu > c) || (cu == c && u < t);
        }
        sorted[rank] = unsorted[t];
    }
}

struct GlobalFwdWs {
    logo_bf16* qc;
    GlobalTile* unsorted;
    GlobalTile* sorted;
    int32_t* tile_off;
    int32_t* n_tiles;
    int32_t* next_item;
    int32_t* n_splits;
    SplitTile* splits;
    float* o_part;
    float* m_part;
    float* l_part;
};

// Both preparations of a global call in one launch: block 0 makes the schedule,
// the others gather the selected rows of the dense Q into the packed layout
// (App. B), 256 threads a row, and zero the 128 rows after the last one, so that
// a partial final tile reads finite values.  Each is a chain of a few dependent
// loads in a launch of its own otherwise, one after the other (5-7.5 and 5-6 us
// on the device at 2 x 4K to 16K tokens; together 6-8).
__global__ void __launch_bounds__(1024) global_prep_kernel(const logo_bf16* __restrict__ q, const int32_t* __restrict__ pos,
                                                           const int32_t* __restrict__ cu_q,
                                                           const int32_t* __restrict__ n_sel, int B, int T, int Hq,
                                                           int row_elems, int n_sm, GlobalFwdWs ws)
{
    if (blockIdx.x == 0) {
        global_schedule(pos, cu_q, B, Hq, n_sm, ws.tile_off, ws.unsorted, ws.sorted, ws.n_tiles, ws.next_item, ws.splits,
                        ws.n_splits);
        return;
    }
    const int n = *n_sel;
    const int vecs = row_elems / 8;
    for (int row = (blockIdx.x - 1) * 4 + (threadIdx.x >> 8); row < n + kBM; row += (gridDim.x - 1) * 4) {
        uint4* dst = reinterpret_cast<uint4*>(ws.qc + static_cast<int64_t>(row) * row_elems);
        if (row < n) {
            const int b = seq_of_row(cu_q, B, row);
            const uint4* src = reinterpret_cast<const uint4*>(q + (static_cast<int64_t>(b) * T + pos[row]) * row_elems);
            for (int v = threadIdx.x & 255; v < vecs; v += 256) dst[v] = src[v];
        } else {
            for (int v = threadIdx.x & 255; v < vecs; v += 256) dst[v] = make_uint4(0, 0, 0, 0);
        }
    }
}

// Combine the shares of every split tile: per (row, head), M = max_s m_s,
// L = sum_s 2^(m_s - M) l_s, O = sum_s 2^(m_s - M) O_s / L, lse = (M + log2 L)
// ln 2.  A share whose keys the row cannot see has m_s = -inf and weighs 0.
// Work unit = (split tile, head, group of 8 columns); a block of 128 threads
// (thread = row) takes units in a grid stride, so every unit's 8 x shares
// loads per row are spread over the whole GPU; the transposed partials make
// each of a warp's loads one 128-byte line.
template <int D>
__global__ void __launch_bounds__(128) merge_splits_kernel(const SplitTile* __restrict__ splits,
                                                           const int32_t* __restrict__ n_splits, int Hq, int cap,
                                                           const float* __restrict__ o_part,
                                                           const float* __restrict__ m_part,
                                                           const float* __restrict__ l_part,
                                                           logo_bf16* __restrict__ o, float* __restrict__ lse)
{
    constexpr int kGroups = D / 8;
    const int n_units = *n_splits * Hq * kGroups;
    const int r = threadIdx.x;
    for (int un = blockIdx.x; un < n_units; un += gridDim.x) {
        const int g = un % kGroups, pr = un / kGroups;
        const SplitTile st = splits[pr / Hq];
        const int h = pr % Hq;
        if (r >= st.nrows) continue;
        const int64_t unit0 = static_cast<int64_t>(st.slot0) * Hq + h;  // share s: unit0 + s * Hq
        float M = -INFINITY;
        for (int s = 0; s < st.nsplit; ++s) M = fmaxf(M, m_part[(unit0 + static_cast<int64_t>(s) * Hq) * kBM + r]);
        float L = 0.f;
        float acc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = 0.f;
        for (int s = 0; s < st.nsplit; ++s) {
            const int64_t unit = unit0 + static_cast<int64_t>(s) * Hq;
            const float m = m_part[unit * kBM + r];
            const float w = m == -INFINITY ? 0.f : ex2_approx(m - M);
            L += w * l_part[unit * kBM + r];
            const float* src = o_part + unit * kBM * D + (g * 8) * kBM + r;
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = src[e * kBM];
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] += w * v[e];
        }
        const float inv = 1.0f / L;
        uint4 w4;
        w4.x = pack_bf16x2(acc[0] * inv, acc[1] * inv);
        w4.y = pack_bf16x2(acc[2] * inv, acc[3] * inv);
        w4.z = pack_bf16x2(acc[4] * inv, acc[5] * inv);
        w4.w = pack_bf16x2(acc[6] * inv, acc[7] * inv);
        *reinterpret_cast<uint4*>(o + (static_cast<int64_t>(st.row0 + r) * Hq + h) * D + g * 8) = w4;
        if (g == 0) lse[static_cast<int64_t>(h) * cap + st.row0 + r] = (M + log2f(L)) * kLn2;
    }
}

size_t global_fwd_ws_layout(const logo_dims& d, char* base, GlobalFwdWs* ws)
{
    const size_t cap = static_cast<size_t>(d.B) * d.T;
    const size_t max_tiles = cap / kBM + d.B + 1;
    const size_t max_entries = max_tiles + kMaxPartialUnits;  // each split adds at most one entry per slot
    size_t off = 0;
    const size_t o_qc = off;
    off = round_up(off + (cap + kBM) * d.Hq * d.D * 2, 256);
    const size_t o_un = off;
    off = round_up(off + max_entries * sizeof(GlobalTile), 256);
    const size_t o_so = off;
    off = round_up(off + max_entries * sizeof(GlobalTile), 256);
    const size_t o_to = off;
    off = round_up(off + (d.B + 1) * sizeof(int32_t), 256);
    const size_t o_nt = off;
    off = round_up(off + 4 * sizeof(int32_t), 256);
    const size_t o_sp = off;
    off = round_up(off + max_tiles * sizeof(SplitTile), 256);
    const size_t o_op = off;
    off = round_up(off + static_cast<size_t>(kMaxPartialUnits) * kBM * d.D * sizeof(float), 256);
    const size_t o_mp = off;
    off = round_up(off + static_cast<size_t>(kMaxPartialUnits) * kBM * sizeof(float), 256);
    const size_t o_lp = off;
    off = round_up(off + static_cast<size_t>(kMaxPartialUnits) * kBM * sizeof(float), 256);
    if (ws) {
        ws->qc = reinterpret_cast<logo_bf16*>(base + o_qc);
        ws->unsorted = reinterpret_cast<GlobalTile*>(base + o_un);
        ws->sorted = reinterpret_cast<GlobalTile*>(base + o_so);
        ws->tile_off = reinterpret_cast<int32_t*>(base + o_to);
        ws->n_tiles = reinterpret_cast<int32_t*>(base + o_nt);
        ws->next_item = ws->n_tiles + 1;
        ws->n_splits = ws->n_tiles + 2;
        ws->splits = reinterpret_cast<SplitTile*>(base + o_sp);
        ws->o_part = reinterpret_cast<float*>(base + o_op);
        ws->m_part = reinterpret_cast<float*>(base + o_mp);
        ws->l_part = reinterpret_cast<float*>(base + o_lp);
    }
    return off;
}

template <int D, bool GLOBAL>
int launch_fwd(const FwdParams& prm, int n_items_upper, cudaStream_t st)
{
    using C = FwdCfg<D>;
    static bool attr_done = false;  // benign race: setting the attribute twice is harmless
    if (!attr_done) {
        if (set_smem_limit(attn_fwd_kernel<D, GLOBAL>, C::kSmemBytes) != cudaSuccess) return LOGO_ERR_CUDA;
        attr_done = true;
    }
    const int grid = max(1, min(n_items_upper, device_sm_count()));
    attn_fwd_kernel<D, GLOBAL><<<grid, C::kThreads, C::kSmemBytes, st>>>(prm);
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}

int check_attn_ptrs(const void* q, const void* k, const void* v)
{
    if (!q || !k || !v) return LOGO_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v)) return LOGO_ERR_UNSUPPORTED;
    return LOGO_OK;
}

}  // namespace

int attn_fwd_tu_status(int clear) { return read_tu_status(clear); }

}  // namespace logo

using namespace logo;

extern "C" int logo_local_attn_fwd(const logo_bf16* q, const logo_bf16* k, const logo_bf16* v, logo_bf16* o,
                                   float* lse, logo_dims dims, int window, float scale, void* stream)
{
    int rc = check_dims(dims);
    if (rc != LOGO_OK) return rc;
    if ((rc = check_attn_ptrs(q, k, v)) != LOGO_OK) return rc;
    if (!o || !lse || window < 1) return LOGO_ERR_INVALID_ARG;
    if (!aligned16(o)) return LOGO_ERR_UNSUPPORTED;
    if (!(scale >= 0.0f)) return LOGO_ERR_INVALID_ARG;
    if (scale == 0.0f) scale = 1.0f / sqrtf(static_cast<float>(dims.D));
    FwdParams prm{};
    const int w = window > dims.T ? dims.T : window;
    if (!encode_bf16_4d(&prm.tm_q, q, dims.D, dims.Hq, dims.T, dims.B, 64, kBM) ||
        !encode_bf16_4d(&prm.tm_k, k, dims.D, dims.Hkv, dims.T, dims.B, 64, kBN) ||
        !encode_bf16_4d(&prm.tm_v, v, dims.D, dims.Hkv, dims.T, dims.B, 64, kBN))
        return LOGO_ERR_CUDA;
    prm.o = o;
    prm.lse = lse;
    prm.B = dims.B;
    prm.T = dims.T;
    prm.Hq = dims.Hq;
    prm.Hkv = dims.Hkv;
    prm.window = w;
    prm.cap = dims.B * dims.T;
    prm.q_tiles = (dims.T + kBM - 1) / kBM;
    prm.by_hq = FastDiv(dims.Hq);
    prm.by_group = FastDiv(dims.Hq / dims.Hkv);
    prm.by_q_tiles = FastDiv(prm.q_tiles);
    prm.scale_log2 = scale * kLog2e;
    const int n_items = dims.B * prm.q_tiles * dims.Hq;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return dims.D == 128 ? launch_fwd<128, false>(prm, n_items, st) : launch_fwd<64, false>(prm, n_items, st);
}

extern "C" size_t logo_global_attn_fwd_workspace_size(logo_dims dims)
{
    if (check_dims(dims) != LOGO_OK) return 0;
    return global_fwd_ws_layout(dims, nullptr, nullptr);
}

extern "C" int logo_global_sparse_attn_fwd(const logo_bf16* q, const logo_bf16* k, const logo_bf16* v,
                                           const int32_t* pos, const int32_t* cu_q, const int32_t* n_sel_total,
                                           logo_bf16* o_c, float* lse_c, logo_dims dims, float scale,
                                           void* workspace, size_t workspace_bytes, void* stream)
{
    int rc = check_dims(dims);
    if (rc != LOGO_OK) return rc;
    if ((rc = check_attn_ptrs(q, k, v)) != LOGO_OK) return rc;
    if (!pos || !cu_q || !n_sel_total || !o_c || !lse_c) return LOGO_ERR_INVALID_ARG;
    if (!aligned16(o_c)) return LOGO_ERR_UNSUPPORTED;
    if (!(scale >= 0.0f)) return LOGO_ERR_INVALID_ARG;
    if (scale == 0.0f) scale = 1.0f / sqrtf(static_cast<float>(dims.D));
    const size_t need = global_fwd_ws_layout(dims, nullptr, nullptr);
    if (!workspace || workspace_bytes < need || !aligned16(workspace)) return LOGO_ERR_WORKSPACE;
    GlobalFwdWs ws;
    global_fwd_ws_layout(dims, static_cast<char*>(workspace), &ws);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int cap = dims.B * dims.T;
    const int row_elems = dims.Hq * dims.D;
    const int n_sm = device_sm_count();
    const int grid = 1 + min((cap + kBM + 3) / 4, n_sm * 2 - 1);
    global_prep_kernel<<<grid, 1024, 0, st>>>(q, pos, cu_q, n_sel_total, dims.B, dims.T, dims.Hq, row_elems, n_sm, ws);
    if (cudaGetLastError() != cudaSuccess) return LOGO_ERR_CUDA;
    FwdParams prm{};
    if (!encode_bf16_4d(&prm.tm_q, ws.qc, dims.D, dims.Hq, static_cast<uint64_t>(cap) + kBM, 1, 64, kBM) ||
        !encode_bf16_4d(&prm.tm_k, k, dims.D, dims.Hkv, dims.T, dims.B, 64, kBN) ||
        !encode_bf16_4d(&prm.tm_v, v, dims.D, dims.Hkv, dims.T, dims.B, 64, kBN))
        return LOGO_ERR_CUDA;
    prm.o = o_c;
    prm.lse = lse_c;
    prm.pos = pos;
    prm.tiles = ws.sorted;
    prm.n_tiles = ws.n_tiles;
    prm.next_item = ws.next_item;
    prm.o_part = ws.o_part;
    prm.m_part = ws.m_part;
    prm.l_part = ws.l_part;
    prm.B = dims.B;
    prm.T = dims.T;
    prm.Hq = dims.Hq;
    prm.Hkv = dims.Hkv;
    prm.window = kNoWindow;
    prm.cap = cap;
    prm.q_tiles = 0;
    prm.by_hq = FastDiv(dims.Hq);
    prm.by_group = FastDiv(dims.Hq / dims.Hkv);
    prm.scale_log2 = scale * kLog2e;
    const int n_items_upper =
        static_cast<int>((static_cast<int64_t>(cap) / kBM + dims.B) * dims.Hq + kMaxPartialUnits);
    rc = dims.D == 128 ? launch_fwd<128, true>(prm, n_items_upper, st) : launch_fwd<64, true>(prm, n_items_upper, st);
    if (rc != LOGO_OK) return rc;
    // Splitting a tile takes kSplitMinGainBlocks of gain over shares of at least
    // kMinSplitBlocks: with fewer blocks in a sequence nothing is ever split.
    // Otherwise the merge is always launched (a fixed launch sequence, capturable
    // in a graph); it exits at once without splits.  (Its launch was 3 of the 25 us
    // of device time, and as much of the host's, in a 512-token layer.)
    if ((dims.T + kBN - 1) / kBN < kMinSplitBlocks + kSplitMinGainBlocks)
        return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
    const int merge_grid = n_sm * 4;
    if (dims.D == 128)
        merge_splits_kernel<128><<<merge_grid, 128, 0, st>>>(ws.splits, ws.n_splits, dims.Hq, cap, ws.o_part,
                                                             ws.m_part, ws.l_part, o_c, lse_c);
    else
        merge_splits_kernel<64><<<merge_grid, 128, 0, st>>>(ws.splits, ws.n_splits, dims.Hq, cap, ws.o_part,
                                                            ws.m_part, ws.l_part, o_c, lse_c);
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}
