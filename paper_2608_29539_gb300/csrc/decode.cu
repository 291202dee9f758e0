// decode.cu -- one decoding step of both attention branches, compacting the
// global branch to the selected sequences (Sec. 3.3 Autoregressive Decoding:
// the gate is known before the global call, so unselected tokens skip it; the
// paper's serving path launches a dense call and masks, and leaves a kernel
// that compacts active decode rows as the missing piece).
//
//   logo_decode_local_attn          every sequence's new token attends the last
//                                   W positions, read from a ring cache (Eq. 6)
//   logo_decode_global_sparse_attn  only the packed selected rows attend their
//                                   sequence's whole dense cache (Eq. 8)
//
// Both run one persistent kernel per call.  The work is the sub-tiles (64
// cache rows) of every (sequence, KV head) pair of the call, in order, and
// each CTA takes an equal run of them, wherever pairs begin and end: sequences
// differ in length and pairs seldom divide by the CTAs (chunks of 1024 rows
// handed out one by one: 4 of 32 sequences of 8K to 16K rows selected 58 us,
// now 49; all 32 selected 360 us, now 252, 6.5 TB/s).  Where that saves little
// (many short pairs of equal length, as the rings are) a CTA takes whole pairs.
// A CTA (4 warps) walks its run through a 3-stage TMA ring (128-byte
// swizzle), a stage refilled once all four warps have released it, and
// serves every query head of the KV head's group from each: S = q.K^T and
// O = P.V as warp-level bf16 products (mma.sync m16n8k16: the group's heads
// are the 16 rows, so a group of up to 16 heads fills one tile).  Each warp
// takes 16 rows of every sub-tile and keeps its own online softmax (running
// max and sum per head, in log2 units) across the piece's sub-tiles, P going
// from the S fragments straight into the A fragments of the P.V product, so
// nothing inside the sub-tile loop waits for another warp; the four warps'
// results are combined exactly at the end of the piece.
// A pair that lies whole inside one CTA's run gets its output written by that
// CTA.  The pieces of the others (at most two a CTA: one at either end of its
// run) leave their unnormalised O, max and sum, and the last piece of a pair to
// finish (a counter per pair, cleared by the call) combines them exactly.
// Decoding is bound by HBM: every cache byte serves only the group's heads.
// In the global call unselected sequences have no sub-tiles, so they cost no
// cache traffic and no host synchronisation is needed.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "attn_common.cuh"
#include "host_common.h"
#include "logo_status.cuh"
#include "sm100.cuh"

namespace logo {
namespace {

constexpr int kDecThreads = 128;  // 4 warps
constexpr int kDecRows = 64;      // cache rows per sub-tile, 16 per warp
constexpr int kDecRowsPerWarp = kDecRows / 4;
constexpr int kDecMaxGroup = 16;  // query heads per KV head (the mma tile's 16 rows)
constexpr int kDecMinSub = 2;     // sub-tiles of a CTA's run at least
constexpr int kDecSplitCost = 8;  // what cutting pairs into pieces has to save, in sub-tiles
constexpr int kDecMaxWholeDense = 24, kDecMaxWholeRing = 32;  // sub-tiles of a pair left whole at most
constexpr int kDecStages = 3;     // TMA ring depth

struct DecParams {
    CUtensorMap tm_k;  // cache [B, R, Hkv, D], box {64, 1, 128, 1}
    CUtensorMap tm_v;
    const logo_bf16* q;       // [B, Hq, D]
    const int32_t* seq_len;   // [B] tokens in the cache, the new one included
    const int32_t* cu_q;      // global: [B+1] packed rows of the (B, 1) selection
    const int32_t* n_sel;     // global: [1]
    float* part;              // [2 CTAs, group, D]: unnormalised o of a CTA's pieces of shared pairs
    float2* part_ml;          // [2 CTAs, group]: their running max (log2 units) and sum
    int32_t* done;            // [B, Hkv] pieces finished (cleared by the call); NULL: whole pairs only
    logo_bf16* out;           // [B, Hq, D] (global: packed rows)
    int B, R, Hq, Hkv, window, min_sub;
    float scale_log2;
};

template <int D>
struct DecCfg {
    static constexpr int kHalfBytes = kDecRows * 128;         // 64 head-dim columns of the sub-tile's rows
    static constexpr int kTileBytes = (D / 64) * kHalfBytes;  // K or V sub-tile
    static constexpr int kStageBytes = 2 * kTileBytes;        // K then V
    static constexpr int kOffW = kDecStages * kStageBytes;    // merge weights [group][pieces] fp32
    static constexpr int kOffM = kOffW + 16 * 64 * 4;         // the warps' partial results, sized per group:
    // [warp][group][D + 2] fp32: unnormalised o, then m, l
    static constexpr int merge_bytes(int group) { return 4 * group * (D + 2) * 4; }
    static constexpr int smem_bytes(int group) { return kOffM + merge_bytes(group) + 1024; }
};
constexpr int kDecMaxPieces = 64;  // pieces of a pair at most (the merge's weights: group x pieces <= 16 x 64)

// Which rows of a cache the new token sees.  Dense cache: rows below its
// length.  Ring of R slots: position s sits in slot s mod R, so slot j holds
// the position `age` before the newest (slot `newest`), and is seen while age
// is below the window; slots past the ring's end (a last sub-tile may reach
// there) hold nothing.
template <bool RING>
struct DecVisible {
    int used, newest, R, window;

    __device__ __forceinline__ DecVisible(int len, int R_, int window_)
        : used(max(0, min(len, R_))), newest(RING ? (len - 1) % R_ : 0), R(R_), window(window_)
    {
    }
    __device__ __forceinline__ bool row(int j) const
    {
        return j < used && (!RING || newest - j + (j > newest ? R : 0) < window);
    }
    __device__ __forceinline__ bool all16(int j) const  // rows j .. j + 15
    {
        return j + 16 <= used && (!RING || window >= used);
    }
};

// Sub-tiles of sequence b's cache that the call reads (per KV head): its rows
// in use; none for a sequence the global call does not have (n_rows: its packed
// rows, read once).
template <bool RING>
__device__ __forceinline__ int dec_subs(const DecParams& p, int n_rows, int b, int* len)
{
    int n = p.seq_len[b];
    if (!RING) {
        n = min(n, p.R);  // a dense cache holds at most R tokens
        const int row = p.cu_q[b];
        if (p.cu_q[b + 1] == row || row >= n_rows) n = 0;
    }
    *len = n;
    return (max(0, min(n, p.R)) + kDecRows - 1) / kDecRows;
}

// A piece of a CTA's run: sub-tiles s .. s1 - 1 (s = s1: none, the run is
// over) of pair (b, kvh), which has `subs` of them, the first at index pair0 of
// the call's sequence; `left`: the run's sub-tiles after the piece.
struct DecPiece {
    int b, kvh, s, s1, subs, len, left, pair;
    long long pair0;
};

// The next piece: of the next pair in order, or (whole pairs) of the pair a
// grid further on: of all that the call could have while each gets a CTA of its
// own or all are selected, else among those of the packed rows.  (Dealt out over
// all the sequences, a few CTAs had two of the pairs of 14 selected of 49 x 192
// rows, 8 KV heads of 128, and most had none: 10.4 us, now 7.0.  Finding a row's
// sequence costs 0.5 us.)
template <bool RING>
__device__ __forceinline__ void dec_next_piece(const DecParams& p, int n_rows, DecPiece& c)
{
    c.pair0 += c.subs;
    c.s = c.s1 = 0;
    if (!p.done) {
        c.subs = 0;
        while (c.subs == 0) {
            c.pair += gridDim.x;
            const bool direct = RING || p.B * p.Hkv <= static_cast<int>(gridDim.x) || n_rows == p.B;
            if (c.pair >= (direct ? p.B : min(n_rows, p.cu_q[p.B])) * p.Hkv) return;
            const int r = c.pair / p.Hkv;
            c.b = direct ? r : seq_of_row(p.cu_q, p.B, r);
            c.kvh = c.pair - r * p.Hkv;
            c.subs = dec_subs<RING>(p, n_rows, c.b, &c.len);
        }
        c.s1 = c.subs;
        return;
    }
    if (c.left == 0) return;
    if (++c.kvh == p.Hkv) {
        c.kvh = 0;
        c.subs = 0;
        while (c.subs == 0 && ++c.b < p.B) c.subs = dec_subs<RING>(p, n_rows, c.b, &c.len);
    }
    c.s1 = min(c.subs, c.left);
    c.left -= c.s1;
}

template <int D, bool RING>
__global__ void __launch_bounds__(kDecThreads, 2) decode_attn_kernel(const __grid_constant__ DecParams p)
{
    using C = DecCfg<D>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // bar_full: a stage's K/V sub-tile landed; bar_empty: the four warps are done with it
    __shared__ __align__(8) uint64_t bar_full[kDecStages], bar_empty[kDecStages];
    __shared__ volatile int abort_flag;
    __shared__ int sh_last;
    __shared__ float sh_wm[4][kDecMaxGroup];  // per head: weight of each warp's partial, 1 / L
    __shared__ float sh_M[kDecMaxGroup], sh_L[kDecMaxGroup];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int gid = lane >> 2, tig = lane & 3;  // mma fragment coordinates
    const int mi = lane >> 3, rr = lane & 7;    // ldmatrix: matrix index, row in the matrix
    const int group = p.Hq / p.Hkv;
    float* sW = reinterpret_cast<float*>(smem + C::kOffW);
    float* sM = reinterpret_cast<float*>(smem + C::kOffM);
    const uint32_t sRing = smem_u32(smem);
    __shared__ long long sh_scan[4];
    __shared__ DecPiece sh_start;
    if (tid == 0) {
        abort_flag = 0;
        for (int s = 0; s < kDecStages; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 4);
        }
        fence_mbar_init();
        tma_prefetch_desc(&p.tm_k);
        tma_prefetch_desc(&p.tm_v);
    }
    const int n_rows = RING ? 0 : *p.n_sel;
    DecPiece cur{};
    long long S = 0, G = 0;
    // a b / c; in 32 bits (a tenth of the instructions) for up to 1M sub-tiles: G < 2^11
    auto muldiv = [&](long long a, long long b, long long c) -> long long {
        if (S < (1 << 20)) return static_cast<uint32_t>(a * b) / static_cast<uint32_t>(c);
        return a * b / c;
    };
    if (!p.done) {  // whole pairs, a grid apart
        __syncthreads();
        cur.pair = static_cast<int>(blockIdx.x) - static_cast<int>(gridDim.x);
        dec_next_piece<RING>(p, n_rows, cur);
    } else {
        // this CTA's run [lo, hi) of the call's S sub-tiles: the total first,
        // then the pair that holds sub-tile lo
        int len0 = 0;
        const int subs0 = tid < p.B ? dec_subs<RING>(p, n_rows, tid, &len0) : 0;  // of sequence tid, for both passes
        long long mine = subs0;
        int len;
        for (int b = tid + kDecThreads; b < p.B; b += kDecThreads) mine += dec_subs<RING>(p, n_rows, b, &len);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
        if (lane == 0) sh_scan[warp] = mine;
        __syncthreads();
        S = (sh_scan[0] + sh_scan[1] + sh_scan[2] + sh_scan[3]) * p.Hkv;
        __syncthreads();
        G = max(1ll, min(static_cast<long long>(gridDim.x), S / p.min_sub));
        if (blockIdx.x >= G || S == 0) return;
        const long long lo = muldiv(S, blockIdx.x, G), hi = muldiv(S, blockIdx.x + 1, G);
        long long carry = 0;
        for (int b0 = 0; b0 < p.B; b0 += kDecThreads) {  // (one round for up to 128 sequences)
            const int b = b0 + tid;
            int n = len0;
            const int subs = b0 == 0 ? subs0 : (b < p.B ? dec_subs<RING>(p, n_rows, b, &n) : 0);
            long long x = static_cast<long long>(subs) * p.Hkv;
            const long long v = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) sh_scan[warp] = x;
            __syncthreads();
            long long base = carry;
            for (int w = 0; w < warp; ++w) base += sh_scan[w];
            const long long first = base + x - v;  // b's first sub-tile
            if (subs > 0 && lo >= first && lo < first + v) {
                DecPiece c{};
                c.b = b;
                c.subs = subs;
                c.len = n;
                c.kvh = static_cast<int>(lo - first) / subs;
                c.pair0 = first + static_cast<long long>(c.kvh) * subs;
                c.s = static_cast<int>(lo - c.pair0);
                c.s1 = static_cast<int>(min(static_cast<long long>(subs), c.s + hi - lo));
                c.left = static_cast<int>(hi - lo) - (c.s1 - c.s);
                sh_start = c;
            }
            carry += sh_scan[0] + sh_scan[1] + sh_scan[2] + sh_scan[3];
            __syncthreads();
            if (carry > lo) break;
        }
        cur = sh_start;
    }
    // the CTA whose run holds sub-tile x
    auto cta_of = [&](long long x) { return static_cast<int>(muldiv((x + 1) * G - 1, 1, S)); };

    // ---- the producer (thread 0) walks the same run as the consumers, up to
    //      kDecStages ahead; a stage is refilled once every warp has released it
    DecPiece pit = cur;
    int issued = 0;
    bool ok = true;
    auto issue = [&]() {
        if (tid != 0 || !ok || pit.s == pit.s1) return;
        const int st = issued % kDecStages;
        if (!(ok = mbar_wait(smem_u32(&bar_empty[st]), ((issued / kDecStages) & 1) ^ 1, &abort_flag))) return;
        const uint32_t bar = smem_u32(&bar_full[st]);
        const uint32_t base = sRing + st * C::kStageBytes;
        const uint64_t pol = policy_evict_first();
        mbar_arrive_expect_tx(bar, C::kStageBytes);
        for (int h = 0; h < D / 64; ++h) {
            tma_load_4d(base + h * C::kHalfBytes, &p.tm_k, bar, 64 * h, pit.kvh, pit.s * kDecRows, pit.b, pol);
            tma_load_4d(base + C::kTileBytes + h * C::kHalfBytes, &p.tm_v, bar, 64 * h, pit.kvh, pit.s * kDecRows,
                        pit.b, pol);
        }
        ++issued;
        if (++pit.s == pit.s1) dec_next_piece<RING>(p, n_rows, pit);
    };
    for (int i = 0; i < kDecStages - 1; ++i) issue();

    // Each warp takes 16 rows of every sub-tile (rows 16w..16w+15) and keeps an
    // online softmax of its own across the piece's sub-tiles, so no instruction
    // inside the sub-tile loop waits for another warp: S = q.K^T lands in mma
    // fragments, P = 2^(S - m) goes from those straight into the A fragments
    // of O += P.V (a pair of 8-column S tiles is one 16-deep A fragment), and
    // the four warps' results are combined once per piece.
    constexpr int NT = D / 8;
    int consumed = 0;
    for (; cur.s < cur.s1 && ok; dec_next_piece<RING>(p, n_rows, cur)) {
        const DecPiece it = cur;
        const int h0 = it.kvh * group;
        const int out_row = RING ? it.b : p.cu_q[it.b];
        const DecVisible<RING> sees(it.len, p.R, p.window);
        // the group's queries as mma A fragments (rows = heads, zero past the group)
        uint32_t qa[D / 16][4];
        {
            const logo_bf16* q0 = p.q + (static_cast<int64_t>(it.b) * p.Hq + h0) * D;
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int hh = gid + (i & 1) * 8;
                    const int d = ks * 16 + (i >> 1) * 8 + 2 * tig;
                    qa[ks][i] = hh < group ? *reinterpret_cast<const uint32_t*>(q0 + hh * D + d) : 0u;
                }
            }
        }
        // this lane's two heads (fragment rows gid and gid + 8): running max
        // (log2 units), what the running sum and O are relative to (below), the
        // sum, and O
        float m_run[2] = {-INFINITY, -INFINITY}, m_ref[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
        float oc[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) oc[nt][i] = 0.f;

        for (int s = it.s; s < it.s1; ++s, ++consumed) {
            issue();
            const int st = consumed % kDecStages;
            const uint32_t sK = sRing + st * C::kStageBytes, sV = sK + C::kTileBytes;
            // the warp leaves together, lane 0's failed issue included (mma.sync needs all lanes)
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_full[st]), (consumed / kDecStages) & 1, &abort_flag) && ok);
            if (!ok) break;
            const int j0 = s * kDecRows + warp * kDecRowsPerWarp;  // this warp's first cache row
            const bool open = sees.all16(j0);
            if (!open) {
                if (lane < kDecRowsPerWarp && !sees.row(j0 + lane)) {
                    // a cache row the token does not see may hold anything, NaN included:
                    // zero its V so that P = 0 keeps it out of the product
                    const int row = warp * kDecRowsPerWarp + lane;
#pragma unroll
                    for (int half = 0; half < D / 64; ++half)
#pragma unroll
                        for (int ch = 0; ch < 8; ++ch)
                            st_shared_v4(sV + half * C::kHalfBytes + sw128_offset(row, ch), 0u, 0u, 0u, 0u);
                }
                __syncwarp();
            }
            // ---- S = q.K^T over the warp's 16 rows (two 8-row tiles)
            float sc[2][4];
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) sc[nt][i] = 0.f;
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
                const int half = ks / 4, ch0 = (ks % 4) * 2;
                const int row = warp * kDecRowsPerWarp + (mi >> 1) * 8 + rr;
                uint32_t b0, b1, b2, b3;
                ldsm_x4(sK + half * C::kHalfBytes + sw128_offset(row, ch0 + (mi & 1)), b0, b1, b2, b3);
                mma_bf16_16816(sc[0], qa[ks], b0, b1);
                mma_bf16_16816(sc[1], qa[ks], b2, b3);
            }
            // ---- online softmax per head: c0, c1 -> head gid, c2, c3 -> head
            //      gid + 8; the 16 rows of a head sit in one lane quad
            float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    sc[nt][i] *= p.scale_log2;
                    if (!open && !sees.row(j0 + nt * 8 + 2 * tig + (i & 1))) sc[nt][i] = -INFINITY;
                    mx[i >> 1] = fmaxf(mx[i >> 1], sc[nt][i]);
                }
            }
            // P is rounded to bf16 against the running max, but a whole number of
            // powers of two above or below this sub-tile's own max, within half of
            // one of the running max: the largest P of the 16 rows is then a power
            // of two, which the rounding leaves as it is, in every sub-tile and
            // wherever the run was cut.  (Against the running max itself that holds
            // only where the max is set, so the error grew with the run: relative L2
            // against 64 bits over nine sizes from 1 x 868 to 32 x 16K tokens,
            // local 0.00204 and global 0.00202, now 0.00197 and 0.00193.)  A sub-tile
            // whose max lies 64 octaves below has nothing to keep exact, and with
            // scores of 2^24 and more below the sum would be off by octaves: the
            // reference stays.
            float alpha[2], m_use[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
                mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
                m_run[r] = fmaxf(m_run[r], mx[r]);
                const float old = m_ref[r];
                if (mx[r] - m_run[r] > -64.f) m_ref[r] = mx[r] + rintf(m_run[r] - mx[r]);
                m_use[r] = m_ref[r] == -INFINITY ? 0.f : m_ref[r];
                alpha[r] = ex2_approx(old - m_use[r]);  // 0 while nothing was seen
            }
            float ls[2] = {0.f, 0.f};
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    sc[nt][i] = ex2_approx(sc[nt][i] - m_use[i >> 1]);
                    ls[i >> 1] += sc[nt][i];
                }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                ls[r] += __shfl_xor_sync(0xffffffffu, ls[r], 1);
                ls[r] += __shfl_xor_sync(0xffffffffu, ls[r], 2);
                l_run[r] = l_run[r] * alpha[r] + ls[r];
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                oc[nt][0] *= alpha[0];
                oc[nt][1] *= alpha[0];
                oc[nt][2] *= alpha[1];
                oc[nt][3] *= alpha[1];
            }
            // P as the A fragment of rows = heads, k = the warp's 16 cache rows
            uint32_t pa[4];
            pa[0] = pack_bf16x2(sc[0][0], sc[0][1]);
            pa[1] = pack_bf16x2(sc[0][2], sc[0][3]);
            pa[2] = pack_bf16x2(sc[1][0], sc[1][1]);
            pa[3] = pack_bf16x2(sc[1][2], sc[1][3]);
            // ---- O += P.V over the warp's 16 cache rows, all D columns
#pragma unroll
            for (int np = 0; np < NT / 2; ++np) {  // pairs of 8-column tiles of V
                // matrices: (rows k0..+7, cols n), (rows k0+8..+15, cols n), then n + 8
                const int row = warp * kDecRowsPerWarp + (mi & 1) * 8 + rr;
                const int col = np * 16 + (mi >> 1) * 8;  // first head-dim column of the 16-byte chunk
                uint32_t b0, b1, b2, b3;
                ldsm_x4_trans(sV + (col / 64) * C::kHalfBytes + sw128_offset(row, (col % 64) / 8), b0, b1, b2, b3);
                mma_bf16_16816(oc[2 * np], pa, b0, b1);
                mma_bf16_16816(oc[2 * np + 1], pa, b2, b3);
            }
            // the warp is done with the stage (its V-row writes ordered before
            // the stage's next TMA write)
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_empty[st]));
        }
        // every thread of the CTA reaches this barrier, and all stop together if
        // any wait gave up
        if (!__syncthreads_and(ok)) break;
        // ---- the four warps' partials: [warp][head][D + 2] in shared memory
        {
            float* mw = sM + warp * group * (D + 2);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int hh = gid + (i >> 1) * 8;
                    const int d = nt * 8 + 2 * tig + (i & 1);
                    if (hh < group) mw[hh * (D + 2) + d] = oc[nt][i];
                }
            }
            if (tig == 0) {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int hh = gid + 8 * r;
                    if (hh < group) {
                        mw[hh * (D + 2) + D] = m_ref[r];
                        mw[hh * (D + 2) + D + 1] = l_run[r];
                    }
                }
            }
        }
        __syncthreads();
        if (tid < group) {  // per head: M = max_w m_w, L = sum_w 2^(m_w - M) l_w
            float M = -INFINITY;
#pragma unroll
            for (int wv = 0; wv < 4; ++wv) M = fmaxf(M, sM[(wv * group + tid) * (D + 2) + D]);
            float L = 0.f;
#pragma unroll
            for (int wv = 0; wv < 4; ++wv) {
                const float mv = sM[(wv * group + tid) * (D + 2) + D];
                const float wgt = (M == -INFINITY || mv == -INFINITY) ? 0.f : ex2_approx(mv - M);
                sh_wm[wv][tid] = wgt;
                L += wgt * sM[(wv * group + tid) * (D + 2) + D + 1];
            }
            sh_M[tid] = M;
            sh_L[tid] = L;
        }
        __syncthreads();
        if (it.s == 0 && it.s1 == it.subs) {  // the whole pair: normalise and write the output
            for (int i = tid; i < group * D; i += kDecThreads) {
                const int hh = i / D, d = i % D;
                float acc = 0.f;
#pragma unroll
                for (int wv = 0; wv < 4; ++wv) acc += sh_wm[wv][hh] * sM[(wv * group + hh) * (D + 2) + d];
                const float L = sh_L[hh];
                const __nv_bfloat16 bv = __float2bfloat16_rn(L > 0.f ? acc / L : 0.f);
                p.out[(static_cast<int64_t>(out_row) * p.Hq + h0 + hh) * D + d] = *reinterpret_cast<const logo_bf16*>(&bv);
            }
            __syncthreads();  // the merge buffer is reused by the next piece
            continue;
        }
        // ---- a piece of a pair that other CTAs have pieces of: partial result in
        //      slot 1 of the pair's first CTA and slot 0 of the others, then the
        //      last piece merges
        const int c_first = cta_of(it.pair0), npieces = cta_of(it.pair0 + it.subs - 1) - c_first + 1;
        {
            const int64_t slot = static_cast<int64_t>(2 * blockIdx.x + (static_cast<int>(blockIdx.x) == c_first ? 1 : 0)) * group;
            for (int i = tid; i < group * D; i += kDecThreads) {
                const int hh = i / D, d = i % D;
                float acc = 0.f;
#pragma unroll
                for (int wv = 0; wv < 4; ++wv) acc += sh_wm[wv][hh] * sM[(wv * group + hh) * (D + 2) + d];
                p.part[slot * D + i] = acc;
            }
            if (tid < group) p.part_ml[slot + tid] = make_float2(sh_M[tid], sh_L[tid]);
        }
        __syncthreads();  // every partial of this piece is written
        if (tid == 0) {
            __threadfence();
            const int prev = atomicAdd(p.done + static_cast<int64_t>(it.b) * p.Hkv + it.kvh, 1);
            sh_last = prev == npieces - 1;
            if (sh_last) __threadfence();
        }
        __syncthreads();
        if (sh_last) {
            // M = max_c m_c, L = sum_c 2^(m_c - M) l_c, o = sum_c 2^(m_c - M) o_c / L.
            // A warp per head for the weights (a lane per piece, two at most: every
            // max and sum arrives in one round of loads), then four columns a
            // thread, eight pieces' loads in flight
            auto slot_of = [&](int c) { return static_cast<int64_t>(2 * (c_first + c) + (c == 0 ? 1 : 0)) * group; };
            for (int hh = warp; hh < group; hh += 4) {
                float2 ml[2];
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    ml[k] = lane + 32 * k < npieces ? __ldcg(p.part_ml + slot_of(lane + 32 * k) + hh)
                                                    : make_float2(-INFINITY, 0.f);
                float M = fmaxf(ml[0].x, ml[1].x);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
                float w[2], L = 0.f;
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    w[k] = ml[k].x == -INFINITY ? 0.f : ex2_approx(ml[k].x - M);
                    L += w[k] * ml[k].y;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
                const float inv = L > 0.f ? 1.0f / L : 0.f;
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    if (lane + 32 * k < npieces) sW[hh * npieces + lane + 32 * k] = w[k] * inv;
            }
            __syncthreads();
            for (int i = tid; i < group * (D / 4); i += kDecThreads) {
                const int hh = i / (D / 4);
                const float* wts = sW + hh * npieces;
                float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
                for (int c = 0; c < npieces; ++c) {
                    const float4 v = __ldcg(reinterpret_cast<const float4*>(p.part + slot_of(c) * D) + i);
                    const float w = wts[c];
                    o.x += w * v.x;
                    o.y += w * v.y;
                    o.z += w * v.z;
                    o.w += w * v.w;
                }
                *reinterpret_cast<uint2*>(p.out + (static_cast<int64_t>(out_row) * p.Hq + h0) * D + 4 * i) =
                    make_uint2(pack_bf16x2(o.x, o.y), pack_bf16x2(o.z, o.w));
            }
        }
        __syncthreads();  // sW and the merge buffer are reused by the next piece
    }
    if (!ok && tid == 0) {  // let copies already issued land before the CTA exits
        for (int k = consumed; k < issued; ++k) mbar_wait_drain(smem_u32(&bar_full[k % kDecStages]), (k / kDecStages) & 1);
    }
}

constexpr int kDecCtasPerSm = 2;  // resident at most: what the registers of 128 threads allow

// How a call's sub-tiles are cut into runs: at least min_sub each (short enough
// to fill the GPU, at least kDecMinSub, and long enough for kDecMaxPieces pieces
// of a pair), by at most `ctas` CTAs.
struct DecCut {
    int min_sub;
    long long ctas;
};

DecCut dec_cut(const logo_dims& d, long long resident)
{
    const long long n_sub = (d.T + kDecRows - 1) / kDecRows, subs = static_cast<long long>(d.B) * d.Hkv * n_sub;
    const long long min_sub = std::max<long long>(kDecMinSub, (n_sub + kDecMaxPieces - 3) / (kDecMaxPieces - 2));
    return DecCut{static_cast<int>(min_sub), std::max(1ll, std::min(subs / min_sub, resident))};
}

// part: [2 x CTAs, group, D] fp32, part_ml: [2 x CTAs, group] fp32 pairs, done: [B, Hkv] int32
size_t decode_ws_layout(const logo_dims& d, char* base, DecParams* p)
{
    const long long ctas = dec_cut(d, static_cast<long long>(kDecCtasPerSm) * device_sm_count()).ctas;
    const size_t rows = 2 * static_cast<size_t>(ctas) * (d.Hq / d.Hkv);
    size_t off = round_up(rows * d.D * sizeof(float), 256);
    const size_t o_ml = off;
    off = round_up(off + rows * sizeof(float2), 256);
    const size_t o_done = off;
    off = round_up(off + static_cast<size_t>(d.B) * d.Hkv * sizeof(int32_t), 256);
    if (p) {
        p->part = reinterpret_cast<float*>(base);
        p->part_ml = reinterpret_cast<float2*>(base + o_ml);
        p->done = reinterpret_cast<int32_t*>(base + o_done);
    }
    return off;
}

int check_decode(const logo_dims& d)
{
    int rc = check_dims(d);
    if (rc != LOGO_OK) return rc;
    if (d.Hq / d.Hkv > kDecMaxGroup) return LOGO_ERR_UNSUPPORTED;
    return LOGO_OK;
}

template <int D, bool RING>
int launch_decode(DecParams& prm, const logo_dims& dims, cudaStream_t st)
{
    static bool attr_done = false;  // benign race: setting the attribute twice is harmless
    if (!attr_done) {
        if (set_smem_limit(decode_attn_kernel<D, RING>, DecCfg<D>::smem_bytes(kDecMaxGroup)) != cudaSuccess)
            return LOGO_ERR_CUDA;
        attr_done = true;
    }
    // as many resident CTAs as fit (each keeps up to three sub-tiles' K/V loads in
    // flight); the merge buffer, and so the fit, depends on the group size
    const int group = prm.Hq / prm.Hkv;
    const int smem = DecCfg<D>::smem_bytes(group);
    static int per_sm_of[kDecMaxGroup + 1] = {};
    int per_sm = per_sm_of[group];
    if (per_sm == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, decode_attn_kernel<D, RING>, kDecThreads, smem) !=
                cudaSuccess ||
            per_sm < 1)
            per_sm = 1;
        per_sm_of[group] = per_sm;
    }
    const long long n_sub = (prm.R + kDecRows - 1) / kDecRows, pairs = static_cast<long long>(prm.B) * prm.Hkv;
    const long long ctas = static_cast<long long>(std::min(per_sm, kDecCtasPerSm)) * device_sm_count();
    // Whole pairs when cutting them saves less than kDecSplitCost sub-tiles of
    // the longest run (with full caches), else equal runs: finding the runs, the
    // counters' clearing and the merge cost about that many.  A call in runs of two
    // sub-tiles takes 12 to 16 us (28 x 448 rows, one head of 64), whole pairs of
    // seven 7.5; 90 x 768 rows, 8 heads of 128, whole and cut 50.4 and 53.6 with
    // all selected, 15.2 and 21.3 with 23.  What is selected and how long the
    // sequences are is not known here, so a pair of more than kMaxWhole sub-tiles
    // is always cut: one CTA takes 0.7 us for a sub-tile and may be the only one
    // with work.  38 sequences of 16K rows and 8 KV heads (a pair a CTA) whole and
    // cut: 4 selected 192 and 50 us, all 375 and 378; of 2K rows: 2 selected 30
    // and 12, all 51 and 55; a ring of 4K slots, one sequence long 60 and 17, all
    // 94 and 99.
    constexpr int kMaxWhole = RING ? kDecMaxWholeRing : kDecMaxWholeDense;
    const long long whole_run = (pairs + ctas - 1) / ctas * n_sub;
    const long long cut_run = std::max<long long>(kDecMinSub, (pairs * n_sub + ctas - 1) / ctas);
    long long grid;
    if (n_sub <= kMaxWhole && whole_run <= cut_run + kDecSplitCost) {
        prm.done = nullptr;
        grid = std::min(pairs, ctas);
    } else {
        const DecCut cut = dec_cut(dims, ctas);
        prm.min_sub = cut.min_sub;
        grid = cut.ctas;
        if (cudaMemsetAsync(prm.done, 0, static_cast<size_t>(pairs) * sizeof(int32_t), st) != cudaSuccess)
            return LOGO_ERR_CUDA;
    }
    decode_attn_kernel<D, RING><<<static_cast<unsigned>(grid), kDecThreads, smem, st>>>(prm);
    return cudaGetLastError() == cudaSuccess ? LOGO_OK : LOGO_ERR_CUDA;
}

int run_decode(bool ring, const logo_bf16* q, const logo_bf16* k, const logo_bf16* v, const int32_t* seq_len,
               const int32_t* cu_q, const int32_t* n_sel, logo_bf16* out, const logo_dims& dims, int window,
               float scale, void* workspace, size_t workspace_bytes, void* stream)
{
    int rc = check_decode(dims);
    if (rc != LOGO_OK) return rc;
    if (!q || !k || !v || !seq_len || !out) return LOGO_ERR_INVALID_ARG;
    if (!ring && (!cu_q || !n_sel)) return LOGO_ERR_INVALID_ARG;
    if (ring && window < 1) return LOGO_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out)) return LOGO_ERR_UNSUPPORTED;
    if (!(scale >= 0.0f)) return LOGO_ERR_INVALID_ARG;
    if (scale == 0.0f) scale = 1.0f / sqrtf(static_cast<float>(dims.D));
    const size_t need = decode_ws_layout(dims, nullptr, nullptr);
    if (!workspace || workspace_bytes < need || !aligned16(workspace)) return LOGO_ERR_WORKSPACE;
    DecParams prm{};
    if (!encode_bf16_4d(&prm.tm_k, k, dims.D, dims.Hkv, dims.T, dims.B, 64, kDecRows) ||
        !encode_bf16_4d(&prm.tm_v, v, dims.D, dims.Hkv, dims.T, dims.B, 64, kDecRows))
        return LOGO_ERR_CUDA;
    prm.q = q;
    prm.seq_len = seq_len;
    prm.cu_q = cu_q;
    prm.n_sel = n_sel;
    decode_ws_layout(dims, static_cast<char*>(workspace), &prm);
    prm.out = out;
    prm.B = dims.B;
    prm.R = dims.T;
    prm.Hq = dims.Hq;
    prm.Hkv = dims.Hkv;
    prm.window = window;
    prm.scale_log2 = scale * kLog2e;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (dims.D == 128) return ring ? launch_decode<128, true>(prm, dims, st) : launch_decode<128, false>(prm, dims, st);
    return ring ? launch_decode<64, true>(prm, dims, st) : launch_decode<64, false>(prm, dims, st);
}

}  // namespace

int decode_tu_status(int clear) { return read_tu_status(clear); }

}  // namespace logo

using namespace logo;

extern "C" size_t logo_decode_workspace_size(logo_dims dims)
{
    if (check_decode(dims) != LOGO_OK) return 0;
    return decode_ws_layout(dims, nullptr, nullptr);
}

extern "C" int logo_decode_local_attn(const logo_bf16* q, const logo_bf16* k_ring, const logo_bf16* v_ring,
                                      const int32_t* seq_len, logo_bf16* o, logo_dims dims, int window, float scale,
                                      void* workspace, size_t workspace_bytes, void* stream)
{
    return run_decode(true, q, k_ring, v_ring, seq_len, nullptr, nullptr, o, dims, window, scale, workspace,
                      workspace_bytes, stream);
}

extern "C" int logo_decode_global_sparse_attn(const logo_bf16* q, const logo_bf16* k_cache, const logo_bf16* v_cache,
                                              const int32_t* seq_len, const int32_t* cu_q,
                                              const int32_t* n_sel_total, logo_bf16* o_c, logo_dims dims,
                                              float scale, void* workspace, size_t workspace_bytes, void* stream)
{
    return run_decode(false, q, k_cache, v_cache, seq_len, cu_q, n_sel_total, o_c, dims, kNoWindow, scale, workspace,
                      workspace_bytes, stream);
}
