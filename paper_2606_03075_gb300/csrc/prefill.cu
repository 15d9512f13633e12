// Causal prefill attention on the 5th-generation tensor cores (tcgen05) that
// also keeps what the eviction step needs from the rows at its query
// positions, so that the step's own pass over the row statistics goes away.
//
// Every token i of every (layer l, query head h) attends to the keys j <= i of
// its KV head g = h / G (Eq. 2 over all N rows):
//
//     o_i = sum_{j <= i} softmax_j(scale <q_i, k_j>) v_j
//
// A work item is two neighbouring 128-row tiles of one (layer, query head):
// two independent streams over the head's K and V tiles 0..t, which come through
// one TMA ring K_0, V_0, K_1, V_1, ... (stream 0, the lower tile, ends one tile
// earlier).  Per stream and key tile j:
//
//   S_j = Q K_j^T            TMEM, 128 columns
//   softmax warpgroup (thread = row): P_j = 2^(x sl2 - m) rounded to bf16 over
//            S_j's columns, running normaliser l and vision mass; O is rescaled
//            only when a row's maximum rises more than 2^8 above the reference m
//            it uses (m then moves up to the new maximum)
//   O += P_j V_j             TMEM, D columns; P is the A operand in TMEM, V the
//            MN-major operand in shared memory
//
// What bounds it: the chain S_j -> P_j -> PV_j, QK_{j+1} of a stream has no slack
// in itself (512 TMEM columns hold two S and two O, no second S per stream), and
// one stream alone would leave the tensor pipe idle during its softmax.  With two
// streams the chain takes about 2700 clocks per key tile -- softmax 1040, P's
// store and the issuer's wake 350, 16 MMAs 1040, the last ones' drain 300 -- of
// which 2 x 1024 are tensor time.  So:
//   * a warp of its own issues each stream's MMAs, and the two take turns block by
//     block (turn): in one queue order the streams stay half a period apart, where
//     interleaved MMAs finish together and both softmaxes then run while the tensor
//     pipe idles (4240 clocks); a single issuer for both streams pays each block's
//     waits in turn (3450);
//   * an issuer runs warp-uniformly and elects a lane at the MMAs, so that their
//     operands stay in uniform registers (one divergent lane: 110 clocks per MMA
//     instead of 64), and waits for all of a block's barriers at once, a lane each;
//   * the exponentials are taken against the reference the row has before the
//     tile's maximum is known: a sum of at most 2^8 shows that no term is above
//     2^8, so the reference stays; the maximum is looked for only otherwise;
//   * the row's 128 terms are one branch-free block without spills (192 registers
//     by setmaxnreg), the same for all four warps of a tile, and what is rare is
//     rolled: straight-line code that is cold costs about 20 clocks per instruction;
//   * items end for the softmax with the row sums; a further warpgroup divides O by
//     them and stores it while the streams run the next item.
// Measured (one launch, 28 layers of 28/4 heads, d = 128, N = 4352): 3.60 ms with
// one tile per CTA, P in shared memory and the maximum taken for every tile, 2.46 ms
// now (1550 TFLOP/s); 32 layers of 32 heads, N = 3008: 3.05 -> 1.68 ms, also because
// heads are worked on in batches whose K and V stay in L2.
//
// Solo form, for launches with few row tiles (see launch_prefill): one tile per
// item and both S buffers for it, so that a tile's softmax overlaps the MMAs of
// the tile before; one issuer, one softmax warpgroup.
//
// At the rows whose position is one of the eviction step's query positions
// (text_pos) the softmax writes (m, Z, V): the row's reference maximum in
// base-2 units (logit x log2 e), Z = sum_j 2^(x_ij sl2 - m) and the same sum
// over the vision keys (Eq. 6's slice); the output warps copy the rows' queries
// to q_text.  The eviction's score passes read them instead of computing them
// (Eq. 2, 5, 6): the prefill already streams every key of those rows.
//
// Items are claimed from a counter in the workspace, in batches of heads, longest
// causal range first within a batch.
//
// Every wait is bounded (about 1 s of SM cycles); a timeout sets
// TGVKV_STATUS_TIMEOUT and the CTA unwinds after its copies and MMAs have
// finished.
#include <cuda_bf16.h>

#include <math.h>

#include "common.cuh"
#include "launch.h"
#include "tc05.cuh"

namespace tgvkv {
namespace {

constexpr int PM = 128;                 // query rows per tile = TMEM lanes
constexpr int PN = 128;                 // keys per K / V tile
constexpr int PST = 4;                  // ring stages
constexpr int PIQ = 4;                  // items fetched ahead
// warps 0-3 / 4-7: the softmax of stream 0 / 1; 8-11: the output rows; then one
// warp per role
constexpr int P_THREADS = 512;
constexpr int OUT_WARP = 8, LOAD_WARP = 12, MMA_WARP = 13 /* and 14 */;
// warps that read an item: both softmaxes, the output, both issuers (in the solo
// form one softmax and one issuer)
constexpr int P_READERS = 8 + 4 + 2, P_READERS_SOLO = 4 + 4 + 1;
// Registers per thread after launch: 128 at launch (65536 / 512); the
// warpgroups' shares add up to 4 x 128, so that no increase waits for more
// than the block holds.
constexpr int P_REGS = 128, SOFT_REGS = 192, OUT_REGS = 40, ROLE_REGS = 88;
static_assert(2 * SOFT_REGS + OUT_REGS + ROLE_REGS <= 4 * P_REGS, "register split");
// solo form: the first softmax warpgroup has no stream
constexpr int IDLE_REGS = 24, SOLO_SOFT_REGS = 208, SOLO_OUT_REGS = 104;
static_assert(IDLE_REGS + SOLO_SOFT_REGS + SOLO_OUT_REGS + ROLE_REGS <= 4 * P_REGS,
              "register split, solo form");
// TMEM columns: S_w at 128 w (P_w over its first 64), O_w from 256
constexpr int P_TMEM_COLS = 512;
constexpr uint32_t O_COL = 256;
constexpr float kRescaleLog2 = 8.f;     // a stale reference maximum may trail by 2^8
constexpr float kTermLimit = 256.f;      // 2^kRescaleLog2
// K and V of the heads worked on together, so that they stay in L2: 12 to 64 MB take the
// same time within 1.5%; one group at a time 179 us for 32 layers of 32 heads of 675
// tokens (167 so), 96 MB 1789 us for 3008 tokens (1727), all heads 1976, and 28 layers of
// 28/4 heads of 8704 tokens 9.66 ms (9.26).
constexpr size_t kBatchBytes = 48u << 20;

template <int D>
struct FSmem {
    uint64_t full[PST], empty[PST];
    uint64_t q_full[2], q_empty[2];
    uint64_t it_full[PIQ], it_empty[PIQ];
    // per stream; in the solo form s_full and p_full per S buffer (two tiles of the
    // stream are in flight, and a warp may be a tile ahead of another)
    uint64_t s_full[2], p_full[2], o_full[2], o_empty[2], turn[2], mma_done[2];
    uint64_t l_full[2][4];              // [stream][its item % 4]
    int item_hi[PIQ], item_lhq[PIQ];
    uint32_t tmem_base;
    int abort_flag, never;
    float lsum[2][4][PM];               // [stream][its item % 4][row]: the rows' normalisers
    uint16_t wtile[kMaxN / PM + 1];     // first query row at or after position 128 t
    // bits of each position (with query rows only): a vision key, a query row
    alignas(16) uint32_t vis[kMaxN / 32], rows[kMaxN / 32];
    alignas(1024) uint16_t q[2][D / 64][PM * 64];     // per stream and 64 dims, 128-byte swizzled rows
    uint16_t kv[PST][D / 64][PN * 64];  // the ring
};

// A work item: row tiles hi - 1 (stream 0; absent when hi = 0) and hi (stream 1),
// or row tile hi alone (solo form), of query head lhq = l H_q + h, whose KV head
// is lhq / G.  hi < 0: none.
struct PItem {
    int hi, lhq;
};

// Items: batches of `batch` query heads, within a batch the row tiles (pairs of
// them, `each` = 2) from the last one down (longest first), then the heads.
__device__ __forceinline__ PItem prefill_item(const Problem& p, int n_qt, int each, int batch, int i) {
    const int per_head = (n_qt + each - 1) / each;
    const int per = batch * per_head;
    const int b = i / per, within = i - b * per;
    const int left = p.L * p.H_q - b * batch;
    const int size = left < batch ? left : batch;
    const int s = within / size;
    PItem it;
    it.hi = n_qt - 1 - each * s;
    it.lhq = b * batch + (within - s * size);
    return it;
}

__device__ __forceinline__ bool warp_wait_all(uint64_t* bar, uint32_t parity, volatile int* abort) {
    const bool got = tc::mbar_wait(bar, parity, abort);
    return __all_sync(~0u, got);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&b);
}

// O (+)= P V for one key tile: K = 128 keys in steps of 16.  A step of P is 8
// TMEM columns (bf16 pairs); V (MN-major) advances 16 key rows = 2048 bytes.
template <int D>
__device__ __forceinline__ void pv_block(uint32_t d_tmem, uint32_t p_tmem, uint64_t vdesc,
                                         bool accumulate) {
    constexpr uint32_t IDESC_PV = tc::idesc_bf16_bmn(PM, D);
#pragma unroll
    for (int kk = 0; kk < PN / 16; ++kk)
        tc::mma_bf16_ts(d_tmem, p_tmem + (uint32_t)(8 * kk), vdesc + (uint64_t)(kk * (16 * 128 / 16)),
                        IDESC_PV, (accumulate || kk > 0) ? 1u : 0u);
}

// Q K^T for one key tile: D / 16 MMAs of 128 x 128, K = D.
template <int D>
__device__ __forceinline__ void qk_block(uint32_t d_tmem, uint64_t qdesc, uint64_t kdesc) {
    constexpr uint32_t IDESC_QK = tc::idesc_bf16(PM, PN);
    constexpr uint32_t HALF = PM * 64 * 2 / 16;   // next 64 dims, 16-byte units
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
        const uint64_t a = qdesc + (uint64_t)((kk >> 2) * HALF + (kk & 3) * 2);
        const uint64_t b = kdesc + (uint64_t)((kk >> 2) * HALF + (kk & 3) * 2);
        if (kk == 0)
            tc::mma_bf16_c<0>(d_tmem, a, b, IDESC_QK);
        else
            tc::mma_bf16_c<1>(d_tmem, a, b, IDESC_QK);
    }
}

// Keys c > lim of a 32-key word become -inf (a masked key then adds 2^-inf = 0).
__device__ __forceinline__ void mask_word(float (&x)[32], int lim) {
#pragma unroll
    for (int c = 0; c < 32; ++c)
        if (c > lim) x[c] = -INFINITY;
}

// A row's 128 logits of a score tile (TMEM columns from ts); those of keys past lim
// (>= 127: none) become -inf.
__device__ __forceinline__ void load_row(uint32_t ts, int lim, float (&x)[4][32]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) tc::tmem_ld32(ts + (uint32_t)(32 * c), x[c]);
    tc::tmem_wait_ld();
    if (!__all_sync(~0u, lim >= 127)) {
#pragma unroll
        for (int c = 0; c < 4; ++c) mask_word(x[c], lim - 32 * c);
    }
}

// A row's 128 logits of a score tile as 2^(x sl2 - m), packed in pk in bf16 pairs; z: their fp32 sum, v: the part of it at the vision
// keys (bits in vw, the same for every lane of the warp): whole 32-key words, or
// MIXED, for tiles with a word of both kinds, key by key.  One branch-free block: the words' latencies overlap, and
// rows with and without a query run the same code.  (The mixed words' logits
// read and exponentiated once more instead, before P is handed on: 10.77 ms for 28
// layers of N = 8704 whose query rows stand between 32 frames, 9.75 so.)
template <bool MIXED>
__device__ __forceinline__ void exp_row(const float (&x)[4][32], float sl2, float m,
                                        const uint32_t (&vw)[4], uint32_t (&pk)[64], float& z,
                                        float& v) {
    const float2 s2 = make_float2(sl2, sl2), n2 = make_float2(-m, -m);
    z = 0.f;
    v = 0.f;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        float2 za = make_float2(0.f, 0.f), zb = za, va = za, vb = za;
#pragma unroll
        for (int c = 0; c < 32; c += 4) {
            const float2 t0 = fma2(make_float2(x[w][c], x[w][c + 1]), s2, n2);
            const float2 t1 = fma2(make_float2(x[w][c + 2], x[w][c + 3]), s2, n2);
            const float2 e0 = make_float2(fast_exp2(t0.x), fast_exp2(t0.y));
            const float2 e1 = make_float2(fast_exp2(t1.x), fast_exp2(t1.y));
            pk[16 * w + c / 2] = pack_bf16(e0.x, e0.y);
            pk[16 * w + c / 2 + 1] = pack_bf16(e1.x, e1.y);
            za = add2(za, e0);
            zb = add2(zb, e1);
            if (MIXED) {
                if ((vw[w] >> c) & 1u) va.x += e0.x;
                if ((vw[w] >> c) & 2u) va.y += e0.y;
                if ((vw[w] >> c) & 4u) vb.x += e1.x;
                if ((vw[w] >> c) & 8u) vb.y += e1.y;
            }
        }
        const float zw = (za.x + za.y) + (zb.x + zb.y);
        z += zw;
        if (MIXED)
            v += (va.x + va.y) + (vb.x + vb.y);
        else
            v += vw[w] != 0u ? zw : 0.f;
    }
}

// Maximum of a row's 128 logits.
__device__ __forceinline__ float max_row(const float (&x)[4][32]) {
    return fmaxf(fmax3(max32(x[0]), max32(x[1]), max32(x[2])), max32(x[3]));
}

template <int D, bool SOLO>
__global__ void __launch_bounds__(P_THREADS, 1)
    prefill_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                   const __grid_constant__ CUtensorMap tmap_v, Problem p, int n_qt, int batch, int n_items,
                   const uint16_t* __restrict__ q, const uint8_t* __restrict__ modality,
                   const int32_t* __restrict__ text_pos, uint16_t* __restrict__ o,
                   uint16_t* __restrict__ q_text, float* __restrict__ row_stats,
                   uint32_t* __restrict__ work_counter, uint32_t* __restrict__ status) {
    // the tiles' swizzle needs 1024-byte alignment, which the declaration asks for
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    FSmem<D>& s = *reinterpret_cast<FSmem<D>*>(smem_raw);
    if (smem_u32(smem_raw) & 1023u) {
        raise_status(status, TGVKV_STATUS_TIMEOUT);
        return;
    }
    constexpr uint32_t TILE_BYTES = (D / 64) * PN * 128;
    constexpr uint32_t BOX_UNITS = PM * 64 * 2 / 16;          // one 64-wide box, 16-byte units
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint32_t* done_counter = work_counter + 1;

    if (tid == 0) {
        s.abort_flag = 0;
        s.never = 0;
        for (int i = 0; i < PST; ++i) {
            tc::mbar_init(&s.full[i], 1);
            tc::mbar_init(&s.empty[i], SOLO ? 1 : 2);        // the streams
        }
        for (int i = 0; i < PIQ; ++i) {
            tc::mbar_init(&s.it_full[i], 1);
            tc::mbar_init(&s.it_empty[i], SOLO ? P_READERS_SOLO : P_READERS);
        }
        for (int w = 0; w < 2; ++w) {
            tc::mbar_init(&s.q_full[w], 1);
            tc::mbar_init(&s.q_empty[w], 1);
            tc::mbar_init(&s.s_full[w], 1);
            tc::mbar_init(&s.p_full[w], 4);       // a softmax warp each
            for (int i = 0; i < 4; ++i) tc::mbar_init(&s.l_full[w][i], 4);
            tc::mbar_init(&s.o_full[w], 1);
            tc::mbar_init(&s.o_empty[w], 4);      // an output warp each
            tc::mbar_init(&s.turn[w], 1);
            tc::mbar_init(&s.mma_done[w], 1);
        }
        tc::fence_mbar_init();
    }
    if (warp == MMA_WARP) {
        tc::tmem_alloc(&s.tmem_base, P_TMEM_COLS);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = s.tmem_base;
    volatile int* abort_flag = &s.abort_flag;

    // the n-th item of this CTA, as the producer claimed it (hi = -1: none, -2: a
    // failed wait); every lane of the calling warp takes part
    auto warp_item = [&](int n) {
        const int slot = n % PIQ;
        PItem it;
        if (warp_wait_all(&s.it_full[slot], (n / PIQ) & 1, abort_flag)) {
            it.hi = s.item_hi[slot];
            it.lhq = s.item_lhq[slot];
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&s.it_empty[slot]);
        } else {
            s.abort_flag = 1;
            raise_status(status, TGVKV_STATUS_TIMEOUT);
            it.hi = -2;
            it.lhq = 0;
        }
        return it;
    };

    // the softmax warps wait for the output warps' tables
    constexpr int TABLE_READERS = SOLO ? 8 * 32 : 12 * 32;
    if (SOLO && warp < 4) {
        tc::regs_dec<IDLE_REGS>();
    } else if (warp < OUT_WARP) {
        // -------------------------------------------------------- softmax
        tc::regs_inc<SOLO ? SOLO_SOFT_REGS : SOFT_REGS>();
        tc::named_bar_sync(2, TABLE_READERS);
        // Stream and row tile come from lane 0, so that the branches on them are seen to be
        // the warp's (64-dim heads, 8 of 2511 keys 22.8 -> 22.0 us, 96 of 2286 82.2 -> 78.8).
        const int w = __shfl_sync(~0u, warp >> 2, 0), quarter = warp & 3;   // stream, lane quarter
        const int r = quarter * 32 + lane;                   // this thread's row = TMEM lane
        const uint32_t tl = tmem + ((uint32_t)(quarter * 32) << 16);
        const uint32_t to = tl + O_COL + (uint32_t)(w * D);
        const float sl2 = p.scale_log2;
        int st = 0, items = 0;        // tiles and items of this stream so far
        bool ok = true;
        for (int n = 0; ok; ++n) {
            const PItem itm = warp_item(n);
            if (itm.hi < 0) break;
            const int t = __shfl_sync(~0u, itm.hi, 0) - 1 + w;
            if (t < 0) continue;
            const int pos = t * PM + r;
            const bool valid = pos < p.N;
            // query row of the eviction step at this position: the tile's first one,
            // plus those at the tile's positions before (rows out of order, which the
            // status reports, may count past the end)
            int wi = -1;
            bool want_v = false;
            if (p.n_win > 0) {
                const uint4 u = *reinterpret_cast<const uint4*>(&s.rows[4 * t]);
                // for the whole tile, so that its four warps run the same code: with only the
                // warps that hold a query row in the mixed form the two forms took turns in the
                // instruction cache (32 layers of 32 heads of 100 tokens 30.1 -> 25.7 us, of 171
                // tokens 47.5 -> 45.3)
                want_v = (u.x | u.y | u.z | u.w) != 0u;
                const uint32_t own = quarter == 0 ? u.x : quarter == 1 ? u.y : quarter == 2 ? u.z : u.w;
                if ((own >> lane) & 1u) {
                    wi = s.wtile[t] + __popc(own & ((1u << lane) - 1u)) + (quarter > 0 ? __popc(u.x) : 0) +
                         (quarter > 1 ? __popc(u.y) : 0) + (quarter > 2 ? __popc(u.z) : 0);
                    if (!valid || wi >= p.n_win) wi = -1;
                }
            }
            float m = -INFINITY, lsum = 0.f, vsum = 0.f;
            for (int j = 0; j <= t; ++j) {
                uint32_t vw[4] = {0u, 0u, 0u, 0u};
                if (want_v) {
                    const uint4 u = *reinterpret_cast<const uint4*>(&s.vis[4 * j]);
                    vw[0] = u.x;
                    vw[1] = u.y;
                    vw[2] = u.z;
                    vw[3] = u.w;
                }
                const bool mixed = vw[0] + 1u > 1u || vw[1] + 1u > 1u || vw[2] + 1u > 1u || vw[3] + 1u > 1u;
                // the logits of tile st of this stream: its own S, or S 0 and 1 in turn
                const int sb = SOLO ? st & 1 : w;
                const uint32_t ts = tl + (uint32_t)(sb * PN);
                if (!warp_wait_all(&s.s_full[sb], (SOLO ? st >> 1 : st) & 1, abort_flag)) {
                    ok = false;
                    s.abort_flag = 1;
                    break;
                }
                ++st;
                tc::fence_after_sync();
                // keys c <= r are visible in the diagonal tile, all of them below it
                const int lim = j == t ? r : 127;
                uint32_t pk[64];
                float z, v;
                // With the reference the row has: a sum of at most 2^8 shows that no
                // term is above 2^8, so that m stays.  Only otherwise (and for the
                // first tile) is the tile's maximum looked for, in the logits that the
                // exponentials then take.  (Read for each of the two: 3700 clocks per first
                // tile instead of 2700; 32 layers of 32 heads of 171 tokens 56 -> 48 us, of
                // 675 tokens 189 -> 185.)
                bool again = j == 0;
                for (;;) {
                    float x[4][32];
                    load_row(ts, lim, x);
                    if (again) {
                        const float m_tile = max_row(x) * sl2;
                        const bool up = m_tile > m + kRescaleLog2;   // also the first tile
                        float alpha = 1.f;
                        if (up) {
                            alpha = fast_exp2(m - m_tile);
                            m = m_tile;
                            lsum *= alpha;
                            vsum *= alpha;
                        }
                        // PV_{j-1} has finished: S_j came after it.  (Solo: S_j came after
                        // PV_{j-2}; what comes after PV_{j-1} is the S of the tile after this
                        // one, whose barrier this warp awaits for every tile, so that its phase
                        // is known: it cannot be past that S before this warp's P.)
                        if (SOLO && j > 0 && !warp_wait_all(&s.s_full[sb ^ 1], (st >> 1) & 1, abort_flag)) {
                            ok = false;
                            s.abort_flag = 1;
                            break;
                        }
                        if (SOLO) tc::fence_after_sync();
                        if (j > 0 && __any_sync(~0u, up)) {
#pragma unroll 1
                            for (int c = 0; c < D / 16; ++c) {
                                float y[16];
                                tc::tmem_ld16(to + (uint32_t)(16 * c), y);
                                tc::tmem_wait_ld();
#pragma unroll
                                for (int e = 0; e < 16; ++e) y[e] *= alpha;
                                tc::tmem_st16(to + (uint32_t)(16 * c), y);
                            }
                            tc::tmem_wait_st();
                        }
                    }
                    if (mixed)
                        exp_row<true>(x, sl2, m, vw, pk, z, v);
                    else
                        exp_row<false>(x, sl2, m, vw, pk, z, v);
                    if (again || __all_sync(~0u, z <= kTermLimit)) break;
                    again = true;
                }
                if (!ok) break;
                lsum += z;
                // (lanes without a query row sum a vision mass that is never written)
                vsum += v;
                tc::tmem_st32u(ts, *reinterpret_cast<const uint32_t(*)[32]>(pk));
                tc::tmem_st32u(ts + 32u, *reinterpret_cast<const uint32_t(*)[32]>(pk + 32));
                tc::tmem_wait_st();
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&s.p_full[sb]);
            }
            if (!ok) break;
            // the row's normaliser for the output warps, and the eviction rows'
            // statistics.  (Four buffers and barriers: an item's scores come after a PV of
            // at most two items before it, that one after every warp's P of its item and
            // after the output of the item before it was read.)
            s.lsum[w][items & 3][r] = lsum;
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&s.l_full[w][items & 3]);
            ++items;
            if (wi >= 0) {
                const size_t qr = (size_t)itm.lhq * p.n_win + wi;
                row_stats[3 * qr] = m;
                row_stats[3 * qr + 1] = lsum;
                row_stats[3 * qr + 2] = vsum;
            }
        }
        if (!ok) raise_status(status, TGVKV_STATUS_TIMEOUT);
    } else if (warp < LOAD_WARP) {
        // -------------------------------------------------------- output rows
        tc::regs_dec<SOLO ? SOLO_OUT_REGS : OUT_REGS>();
        // The tables: the query rows of each row tile t, indices wtile[t] ..
        // wtile[t + 1] of text_pos (positions ascend), as the first row at or after
        // position 128 t; their positions as bits; and the modality as bits, whole
        // tiles (keys past the end: text).  Done here, while the first loads and MMAs
        // are on their way.
        constexpr int WARPS = LOAD_WARP - OUT_WARP;
        const int ot = tid - 32 * OUT_WARP, ow = warp - OUT_WARP;
        for (int t = ot; t <= n_qt; t += 32 * WARPS) s.wtile[t] = (uint16_t)p.n_win;
        for (int t = ot; t < 4 * n_qt; t += 32 * WARPS) s.rows[t] = 0u;
        tc::named_bar_sync(1, 32 * WARPS);
        for (int i = ot; i < p.n_win; i += 32 * WARPS) {
            const int pi = __ldg(text_pos + i);
            const int before = i > 0 ? __ldg(text_pos + i - 1) : -1;
            if (blockIdx.x == 0 && (pi < 0 || pi >= p.N || before >= pi))
                raise_status(status, TGVKV_STATUS_TEXT_POS);
            if (pi >= 0 && pi < p.N) atomicOr(&s.rows[pi >> 5], 1u << (pi & 31));
            if (pi >= 0 && pi < p.N && before < pi)
                for (int t = before < 0 ? 0 : before / PM + 1; t <= pi / PM; ++t) s.wtile[t] = (uint16_t)i;
        }
        for (int w0 = ow; p.n_win > 0 && w0 < 4 * n_qt; w0 += 8 * WARPS) {
            uint8_t b[8];     // eight loads of a warp in flight
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int key = 32 * (w0 + i * WARPS) + lane;
                b[i] = key < p.N ? __ldg(modality + key) : (uint8_t)0;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t bits = __ballot_sync(~0u, b[i] != 0);
                if (lane == 0 && w0 + i * WARPS < 4 * n_qt) s.vis[w0 + i * WARPS] = bits;
            }
        }
        tc::named_bar_sync(2, TABLE_READERS);
        const int quarter = warp & 3;
        const int r = quarter * 32 + lane;
        const uint32_t tl = tmem + ((uint32_t)(quarter * 32) << 16);
        constexpr int LPR = D / 8, RPI = 32 / LPR;   // lanes per copied row, rows at a time
        uint32_t done0 = 0, done1 = 0;      // items of stream 0 / 1 finished
        bool ok = true;
        for (int n = 0; ok; ++n) {
            const PItem itm = warp_item(n);
            if (itm.hi < 0) break;
            // q_text[l][h][r] = q[l][h][text_pos[r]] for the query rows of the item's
            // tiles, 16 bytes a lane, while the softmax works on them (after the output, the
            // last item's copy ended the launch: 0.4 us; by a warp of its own, its code took
            // turns with the softmax's in the instruction cache, 32 layers of 32 heads of 384
            // tokens 82 -> 90 us)
            const int ws = s.wtile[itm.hi > 0 && !SOLO ? itm.hi - 1 : itm.hi], we = s.wtile[itm.hi + 1];
            const uint16_t* qh = q + (size_t)itm.lhq * p.N * D;
            uint16_t* qt = q_text + (size_t)itm.lhq * p.n_win * D;
#pragma unroll 4
            for (int e = ws + ow * RPI + lane / LPR; e < we; e += WARPS * RPI) {
                const int pos = __ldg(text_pos + e);
                if (pos < 0 || pos >= p.N) continue;
                reinterpret_cast<uint4*>(qt + (size_t)e * D)[lane % LPR] =
                    __ldg(reinterpret_cast<const uint4*>(qh + (size_t)pos * D) + lane % LPR);
            }
            for (int w = SOLO ? 1 : 0; ok && w < 2; ++w) {
                const int t = itm.hi - 1 + w;
                if (t < 0) continue;
                const uint32_t c = w ? done1++ : done0++;
                if (!warp_wait_all(&s.l_full[w][c & 3u], (c >> 2) & 1u, abort_flag) ||
                    !warp_wait_all(&s.o_full[w], c & 1u, abort_flag)) {
                    ok = false;
                    s.abort_flag = 1;
                    break;
                }
                tc::fence_after_sync();
                const int pos = t * PM + r;
                const bool valid = pos < p.N;
                const float lsum = s.lsum[w][c & 3u][r];
                const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
                uint16_t* orow = o + ((size_t)itm.lhq * p.N + (valid ? pos : 0)) * D;
                const uint32_t to = tl + O_COL + (uint32_t)(w * D);
#pragma unroll 1
                for (int e = 0; e < D / 16; ++e) {
                    float y[16];
                    tc::tmem_ld16(to + (uint32_t)(16 * e), y);
                    tc::tmem_wait_ld();
                    if (e == D / 16 - 1) {      // O is read: the stream may overwrite it
                        tc::fence_before_sync();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(&s.o_empty[w]);
                    }
                    if (valid) {
#pragma unroll
                        for (int v4 = 0; v4 < 2; ++v4) {
                            uint4 u;
                            u.x = pack_bf16(y[8 * v4] * inv, y[8 * v4 + 1] * inv);
                            u.y = pack_bf16(y[8 * v4 + 2] * inv, y[8 * v4 + 3] * inv);
                            u.z = pack_bf16(y[8 * v4 + 4] * inv, y[8 * v4 + 5] * inv);
                            u.w = pack_bf16(y[8 * v4 + 6] * inv, y[8 * v4 + 7] * inv);
                            *reinterpret_cast<uint4*>(orow + 16 * e + 8 * v4) = u;
                        }
                    }
                }
            }
        }
        if (!ok) raise_status(status, TGVKV_STATUS_TIMEOUT);
    } else {
        tc::regs_dec<ROLE_REGS>();
        if (warp == LOAD_WARP && lane == 0) {
            // ---------------------------------------------------- producer
            tc::tma_prefetch_desc(&tmap_q);
            tc::tma_prefetch_desc(&tmap_k);
            tc::tma_prefetch_desc(&tmap_v);
            int it = 0, q0 = 0, q1 = 0;   // ring stages used, loads of each Q slot
            int g = 0, v_tile[2] = {0, 0}, v_row[2] = {0, 0};   // solo: tiles so far, the V to load
            bool ok = true;
            // the first item of CTA c is item c (grid <= items); later ones are claimed,
            // an item ahead, so that the claim's latency hides behind the item's loads
            uint32_t id = blockIdx.x;
            for (int n = 0; ok; ++n) {
                const int islot = n % PIQ;
                if (!tc::mbar_wait(&s.it_empty[islot], ((n / PIQ) & 1) ^ 1, abort_flag)) {
                    ok = false;
                    break;
                }
                auto load = [&](const CUtensorMap* map, int j, int kv_row) {
                    const int stg = it % PST;
                    if (!tc::mbar_wait(&s.empty[stg], ((it / PST) & 1) ^ 1, abort_flag)) {
                        ok = false;
                        return;
                    }
                    tc::mbar_arrive_expect_tx(&s.full[stg], TILE_BYTES);
#pragma unroll
                    for (int hd = 0; hd < D / 64; ++hd)
                        tc::tma_load_2d(&s.kv[stg][hd][0], map, hd * 64, kv_row + j * PN, &s.full[stg]);
                    ++it;
                };
                PItem itm;
                itm.hi = -1;
                itm.lhq = 0;
                const bool more = id < (uint32_t)n_items;
                if (more) itm = prefill_item(p, n_qt, SOLO ? 1 : 2, batch, (int)id);
                s.item_hi[islot] = itm.hi;
                s.item_lhq[islot] = itm.lhq;
                tc::mbar_arrive(&s.it_full[islot]);
                if (!more) {
                    if (SOLO && g > 1) load(&tmap_v, v_tile[0], v_row[0]);
                    if (SOLO && ok && g > 0) load(&tmap_v, v_tile[1], v_row[1]);
                    break;
                }
                const uint32_t next = claim_item(work_counter, gridDim.x, n_items, status);
                const int q_row = itm.lhq * p.N, kv_row = (itm.lhq / p.G) * p.N;
                auto load_q = [&](int slot, int t) {
                    int& uses = slot == 0 ? q0 : q1;
                    if (!tc::mbar_wait(&s.q_empty[slot], (uses & 1) ^ 1, abort_flag)) {
                        ok = false;
                        return;
                    }
                    if (t >= 0) {
                        tc::mbar_arrive_expect_tx(&s.q_full[slot], TILE_BYTES);
#pragma unroll
                        for (int hd = 0; hd < D / 64; ++hd)
                            tc::tma_load_2d(&s.q[slot][hd][0], &tmap_q, hd * 64, q_row + t * PM,
                                            &s.q_full[slot]);
                    } else {
                        tc::mbar_arrive(&s.q_full[slot]);   // an absent tile
                    }
                    ++uses;
                };
                if (SOLO) {
                    // in the issuer's order: every K goes two tiles ahead of its V
                    load_q(n & 1, itm.hi);
                    for (int j = 0; ok && j <= itm.hi; ++j, ++g) {
                        if (g >= 2) load(&tmap_v, v_tile[0], v_row[0]);
                        if (ok) load(&tmap_k, j, kv_row);
                        v_tile[0] = v_tile[1];
                        v_row[0] = v_row[1];
                        v_tile[1] = j;
                        v_row[1] = kv_row;
                    }
                } else {
                    load_q(0, itm.hi - 1);
                    if (ok) load(&tmap_k, 0, kv_row);
                    if (ok) load_q(1, itm.hi);
                    if (ok) load(&tmap_v, 0, kv_row);
                    for (int j = 1; ok && j <= itm.hi; ++j) {
                        load(&tmap_k, j, kv_row);
                        if (ok) load(&tmap_v, j, kv_row);
                    }
                }
                id = next;
            }
            if (!ok) {
                s.abort_flag = 1;
                raise_status(status, TGVKV_STATUS_TIMEOUT);
            }
            // the last CTA to run out of work (or to give up) re-arms the counters for the
            // next launch
            if (atomicAdd(done_counter, 1u) == gridDim.x - 1) {
                atomicExch(work_counter, 0u);
                atomicExch(done_counter, 0u);
                __threadfence();
            }
            // every copy this CTA issued has landed before it may exit
            if (q0 > 0) tc::mbar_wait(&s.q_full[0], (q0 - 1) & 1, &s.never);
            if (q1 > 0) tc::mbar_wait(&s.q_full[1], (q1 - 1) & 1, &s.never);
            for (int i = it - PST > 0 ? it - PST : 0; i < it; ++i)
                tc::mbar_wait(&s.full[i % PST], (i / PST) & 1, &s.never);
        } else if (SOLO && warp == MMA_WARP + 1) {
            // ---------------------------------------------------- MMA issuer, solo form
            // One row tile at a time, its S in two buffers: over the tiles g of all items
            // the order is QK_0, QK_1, then PV_g, QK_{g+2} once P_g is there, so that a
            // tile's softmax overlaps the MMAs of the tile before.  Ring: K(0), K(1), then
            // V(g), K(g+2) for each g.
            const uint64_t qd0 = tc::sdesc_k_sw128(smem_u32(&s.q[0][0][0]));
            const uint64_t kd0 = tc::sdesc_k_sw128(smem_u32(&s.kv[0][0][0]));
            const uint64_t vd0 = tc::sdesc_mn_sw128(smem_u32(&s.kv[0][0][0]), PN * 64 * 2);
            constexpr uint32_t SLOT = (D / 64) * BOX_UNITS;
            const uint32_t tm = __shfl_sync(~0u, tmem, 0);
            const uint32_t to = tm + O_COL + (uint32_t)D;
            bool ok = true;
            // lane b polls barrier b: the V stage, the K stage, P, O read, Q
            auto wait_all = [&](bool v, int vi, bool k, int ki, bool pp, int g, bool o, uint32_t o_par,
                                bool q, int n) {
                if (!ok) return;
                const uint64_t* bar = lane == 0   ? &s.full[vi % PST]
                                      : lane == 1 ? &s.full[ki % PST]
                                      : lane == 2 ? &s.p_full[g & 1]
                                      : lane == 3 ? &s.o_empty[1]
                                                  : &s.q_full[n & 1];
                const uint32_t parity = lane == 0   ? (uint32_t)(vi / PST) & 1u
                                        : lane == 1 ? (uint32_t)(ki / PST) & 1u
                                        : lane == 2 ? (uint32_t)(g >> 1) & 1u
                                        : lane == 3 ? o_par
                                                    : (uint32_t)(n >> 1) & 1u;
                const bool mine = lane == 0 ? v : lane == 1 ? k : lane == 2 ? pp : lane == 3 ? o
                                                                        : lane == 4 && q;
                const uint32_t addr = smem_u32(bar);
                bool got = !mine || tc::mbar_try_wait_addr(addr, parity);
                if (!__all_sync(~0u, got)) {
                    const long long c0 = clock64();
                    for (uint32_t i = 1;; ++i) {
                        if (!got) got = tc::mbar_try_wait_addr(addr, parity);
                        if (__all_sync(~0u, got)) break;
                        if ((i & 63u) == 0 &&
                            __any_sync(~0u, *abort_flag != 0 || clock64() - c0 > tc::kWaitLimitCycles)) {
                            ok = false;
                            break;
                        }
                    }
                }
                __syncwarp();   // (the vote orders no memory: see the pairs' wait_all)
                tc::fence_after_sync();
            };
            // the next tile to take QK of: tile j of item n (hi < 0: no more)
            int n = 0, j = 0, hi = __shfl_sync(~0u, warp_item(0).hi, 0);
            auto advance = [&]() {
                if (j < hi) {
                    ++j;
                } else {
                    ++n;
                    j = 0;
                    hi = __shfl_sync(~0u, warp_item(n).hi, 0);
                    if (hi == -2) ok = false;
                }
            };
            auto qk = [&](int g, int i) {     // S of tile g from ring stage i and item n's Q
                qk_block<D>(tm + (uint32_t)((g & 1) * PN), qd0 + (uint64_t)((n & 1) * SLOT),
                            kd0 + (uint64_t)((i % PST) * SLOT));
                tc::mma_commit(&s.s_full[g & 1]);
                tc::mma_commit(&s.empty[i % PST]);
                if (j == hi) tc::mma_commit(&s.q_empty[n & 1]);
            };
            if (hi == -2) ok = false;
            // the tiles whose PV is due (bit 0: an item's first, bit 1: its last tile; -1: none)
            int due[2] = {-1, -1}, it = 0;
            for (int g = 0; g < 2; ++g) {
                if (!ok || hi < 0) break;
                wait_all(false, 0, true, it, false, 0, false, 0, j == 0, n);
                if (ok && tc::elect_one()) qk(g, it);
                __syncwarp();
                ++it;
                due[g] = (j == 0 ? 1 : 0) | (j == hi ? 2 : 0);
                advance();
            }
            uint32_t done = 0;                // items begun
            for (int g = 0; ok && due[0] >= 0; ++g) {
                const bool first = due[0] & 1, last = due[0] & 2, more = hi >= 0;
                wait_all(true, it, more, it + 1, true, g, first, (done & 1u) ^ 1u, more && j == 0, n);
                if (ok && tc::elect_one()) {
                    pv_block<D>(to, tm + (uint32_t)((g & 1) * PN), vd0 + (uint64_t)((it % PST) * SLOT),
                                !first);
                    if (last) tc::mma_commit(&s.o_full[1]);
                    tc::mma_commit(&s.empty[it % PST]);
                    if (more)
                        qk(g, it + 1);
                    else    // no further tile: the softmax may still wait for PV_g here
                        tc::mma_commit(&s.s_full[g & 1]);
                }
                __syncwarp();
                if (first) ++done;
                it += more ? 2 : 1;
                due[0] = due[1];
                due[1] = -1;
                if (more) {
                    due[1] = (j == 0 ? 1 : 0) | (j == hi ? 2 : 0);
                    advance();
                }
            }
            if (!ok) {
                s.abort_flag = 1;
                raise_status(status, TGVKV_STATUS_TIMEOUT);
            }
            __syncwarp();
            if (tc::elect_one()) {
                tc::mma_commit(&s.mma_done[1]);
                tc::mbar_wait(&s.mma_done[1], 0, &s.never);
            }
            __syncwarp();
        } else if (!SOLO && (warp == MMA_WARP || warp == MMA_WARP + 1)) {
            // ---------------------------------------------------- MMA issuers
            // One warp per stream w, each running the loop as a whole with one lane
            // elected to issue.  They take turns (turn[w]): slot j of an item is PV_j,
            // QK_{j+1} of stream 0, then of stream 1; where a stream has no further
            // tile, its QK is the next item's first.  One queue order keeps the streams
            // half a period apart (MMAs of both interleaved would finish together, and
            // the two softmaxes then run side by side while the tensor pipe idles), and
            // a warp's waits run while the other one issues.
            const int w = __shfl_sync(~0u, warp, 0) - MMA_WARP;
            const uint64_t qd = tc::sdesc_k_sw128(smem_u32(&s.q[w][0][0]));
            const uint64_t kd0 = tc::sdesc_k_sw128(smem_u32(&s.kv[0][0][0]));
            const uint64_t vd0 = tc::sdesc_mn_sw128(smem_u32(&s.kv[0][0][0]), PN * 64 * 2);
            constexpr uint32_t SLOT = (D / 64) * BOX_UNITS;
            const uint32_t tm = __shfl_sync(~0u, tmem, 0);
            const uint32_t ts = tm + (uint32_t)(w * PN), to = tm + O_COL + (uint32_t)(w * D);
            // lane b polls barrier b of a slot: the V stage, the K stage, P, O read, Q, the turn
            const uint64_t* my_bar = lane == 2   ? &s.p_full[w]
                                     : lane == 3 ? &s.o_empty[w]
                                     : lane == 4 ? &s.q_full[w]
                                     : lane == 5 ? &s.turn[w]
                                                 : &s.full[0];
            const uint32_t my_addr = smem_u32(my_bar);
            uint32_t my_phase = lane == 3 || (lane == 5 && w == 0) ? 1u : 0u;
            constexpr uint32_t NEED_V = 1, NEED_K = 2, NEED_P = 4, NEED_O = 8, NEED_Q = 16, NEED_TURN = 32;
            bool ok = true;
            // wait for the barriers in `need`; K and V at ring stage i
            auto wait_all = [&](uint32_t need, int vi, int ki) {
                if (!ok) return;
                const int i = lane == 0 ? vi : ki;
                const uint32_t addr = my_addr + (lane < 2 ? (uint32_t)(i % PST) * 8u : 0u);
                const uint32_t parity = lane < 2 ? (uint32_t)(i / PST) & 1u : my_phase;
                const bool mine = (need >> lane) & 1u;
                bool got = !mine || tc::mbar_try_wait_addr(addr, parity);
                if (!__all_sync(~0u, got)) {
                    const long long c0 = clock64();
                    for (uint32_t n = 1;; ++n) {
                        if (!got) got = tc::mbar_try_wait_addr(addr, parity);
                        if (__all_sync(~0u, got)) break;
                        if ((n & 63u) == 0 &&
                            __any_sync(~0u, *abort_flag != 0 || clock64() - c0 > tc::kWaitLimitCycles)) {
                            ok = false;
                            break;
                        }
                    }
                }
                if (mine && lane >= 2) my_phase ^= 1u;
                // what each lane's barrier guards, for whichever lane issues the MMAs: the vote
                // orders no memory, this does
                __syncwarp();
                tc::fence_after_sync();
            };
            // S = Q K^T of ring stage i; last: the tile's last use of its Q slot; alone: the
            // other stream does not use the stage
            auto qk = [&](int i, bool last, bool alone) {
                qk_block<D>(ts, qd, kd0 + (uint64_t)((i % PST) * SLOT));
                tc::mma_commit(&s.s_full[w]);
                if (last) tc::mma_commit(&s.q_empty[w]);
                tc::mma_commit(&s.empty[i % PST]);
                if (alone) tc::mma_commit(&s.empty[i % PST]);
            };
            // O (+)= P V of ring stage i
            auto pv = [&](int i, bool first, bool last, bool alone) {
                pv_block<D>(to, ts, vd0 + (uint64_t)((i % PST) * SLOT), !first);
                if (last) tc::mma_commit(&s.o_full[w]);
                tc::mma_commit(&s.empty[i % PST]);
                if (alone) tc::mma_commit(&s.empty[i % PST]);
            };
            int hi = __shfl_sync(~0u, warp_item(0).hi, 0);
            int it = 0;
            if (hi >= 0) {       // the first item's first scores
                wait_all(NEED_Q | NEED_TURN | NEED_K, 0, 0);
                if (ok && tc::elect_one()) {
                    if (w == 1 || hi > 0) qk(0, hi + w == 1, hi == 0);
                    else tc::mbar_arrive(&s.q_empty[0]);
                    tc::mbar_arrive(&s.turn[1 - w]);
                }
                __syncwarp();
            }
            for (int n = 0; ok && hi >= 0; ++n) {
                // ring: K_j at it + 2 j, V_j at it + 2 j + 1; the next item's K_0 after them
                const int nk = hi + w;          // this stream's key tiles
                for (int j = 0; ok && j < hi; ++j) {
                    const int vi = it + 2 * j + 1;
                    const bool more = j + 1 < nk;
                    wait_all(NEED_V | NEED_P | NEED_TURN | (more ? NEED_K : 0u) | (j == 0 ? NEED_O : 0u), vi,
                             vi + 1);
                    if (ok && tc::elect_one()) {
                        pv(vi, j == 0, j + 1 == nk, false);
                        if (more) qk(vi + 1, j + 2 == nk, j + 1 == hi);
                        tc::mbar_arrive(&s.turn[1 - w]);
                    }
                    __syncwarp();
                }
                if (!ok) break;
                // the last slot: stream 1's last tile, and both streams' next item
                const int vi = it + 2 * hi + 1;
                const int next = __shfl_sync(~0u, warp_item(n + 1).hi, 0);
                if (next == -2) {
                    ok = false;
                    break;
                }
                if (w == 1) {
                    wait_all(NEED_V | NEED_P | NEED_TURN | (hi == 0 ? NEED_O : 0u), vi, vi);
                    if (ok && tc::elect_one()) pv(vi, hi == 0, true, true);
                    __syncwarp();
                }
                wait_all((next >= 0 ? NEED_K | NEED_Q : 0u) | (w == 0 ? NEED_TURN : 0u), vi, vi + 1);
                if (ok && tc::elect_one()) {
                    if (next + w > 0) qk(vi + 1, next + w == 1, next == 0);
                    else if (next == 0) tc::mbar_arrive(&s.q_empty[0]);
                    tc::mbar_arrive(&s.turn[1 - w]);
                }
                __syncwarp();
                it += 2 * (hi + 1);
                hi = next;
            }
            if (!ok || hi == -2) {
                s.abort_flag = 1;
                raise_status(status, TGVKV_STATUS_TIMEOUT);
            }
            // every MMA this warp issued has finished before TMEM is released (the
            // elected lane is the same each time: the commit covers them all)
            __syncwarp();
            if (tc::elect_one()) {
                tc::mma_commit(&s.mma_done[w]);
                tc::mbar_wait(&s.mma_done[w], 0, &s.never);
            }
            __syncwarp();
        }
    }

    // ------------------------------------------------------------ teardown
    tc::fence_before_sync();
    __syncthreads();
    if (warp == MMA_WARP) {
        __syncwarp();
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, P_TMEM_COLS);
    }
}

template <int D, bool SOLO>
cudaError_t launch_prefill_d(const Problem& p, const uint16_t* q, const uint16_t* k,
                             const uint16_t* v, const uint8_t* modality, const int32_t* text_pos,
                             uint16_t* o, uint16_t* q_text, float* row_stats, uint32_t* work_counter,
                             uint32_t* status, int sms, cudaStream_t stream) {
    static_assert(sizeof(FSmem<D>) <= 227 * 1024, "shared memory of one CTA");
    alignas(64) CUtensorMap mq, mk, mv;
    if (!make_tile_map(&mq, q, (uint64_t)p.L * p.H_q * p.N, D, PM) ||
        !make_tile_map(&mk, k, (uint64_t)p.L * p.H_kv * p.N, D, PN) ||
        !make_tile_map(&mv, v, (uint64_t)p.L * p.H_kv * p.N, D, PN))
        return cudaErrorInvalidValue;
    const size_t smem = sizeof(FSmem<D>);
    cudaError_t e = cudaFuncSetAttribute(prefill_kernel<D, SOLO>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // the register split adds up only for the register count it was written for
    if (!has_registers<prefill_kernel<D, SOLO>>(P_REGS)) return cudaErrorInvalidConfiguration;
    const int n_qt = (p.N + PM - 1) / PM;
    const int n_items = p.L * p.H_q * (SOLO ? n_qt : (n_qt + 1) / 2);
    // heads worked on together: whole KV groups whose K and V fit kBatchBytes
    const size_t kv_bytes = (size_t)p.N * D * 2 * 2;
    const int groups = (int)(kBatchBytes / kv_bytes > 0 ? kBatchBytes / kv_bytes : 1);
    const int batch = groups < p.L * p.H_kv ? groups * p.G : p.L * p.H_q;
    const int grid = n_items < sms ? n_items : sms;
    prefill_kernel<D, SOLO><<<grid, P_THREADS, smem, stream>>>(mq, mk, mv, p, n_qt, batch, n_items, q,
                                                               modality, text_pos, o, q_text, row_stats,
                                                               work_counter, status);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_prefill(const Problem& p, const uint16_t* q, const uint16_t* k,
                           const uint16_t* v, const uint8_t* modality, const int32_t* text_pos,
                           uint16_t* o, uint16_t* q_text, float* row_stats, char* ws,
                           const WsLayout& lay, cudaStream_t stream) {
    uint32_t* work_counter = reinterpret_cast<uint32_t*>(ws + lay.counters);
    uint32_t* status = reinterpret_cast<uint32_t*>(ws + lay.status);
    const int sms = device_sm_count();
    if (sms <= 0) return cudaErrorInvalidDevice;
    // One tile per item, or two.  Mean time of the one-tile form over that of the pairs,
    // for heads of 100 to 3200 keys, d = 64 and 128, 1 to 100 layers of 8 and 28 heads, by
    // row tiles per SM and (across) row tiles per head:
    //                1     2     3     4     5    >5
    //     up to 1  1.00  0.94  0.90  0.88  0.83  0.80   a pair's tiles wait in one SM
    //         1-2  1.02  1.15  1.03  1.04  0.96  0.94
    //         2-3  0.99  1.00  1.04  0.98  0.93  0.96
    //         3-4  0.97  1.06  0.92  1.10  1.04  0.98
    //     above 4  0.98  0.99  0.97  0.99  1.13  1.11   the pairs share K and V tiles
    // (between, the two round up to whole items per SM at different sizes).  So: one-tile
    // heads, which make no pair, and launches of up to a tile per SM take the one-tile form;
    // two-tile heads pairs; longer ones the one-tile form up to four tiles per SM.
    const int n_qt = (p.N + PM - 1) / PM;
    const long long tiles = (long long)p.L * p.H_q * n_qt;
    const bool solo = n_qt == 1 || tiles <= sms || (n_qt > 2 && tiles <= 4ll * sms);
    const auto launch = p.d == 64 ? (solo ? launch_prefill_d<64, true> : launch_prefill_d<64, false>)
                                  : (solo ? launch_prefill_d<128, true> : launch_prefill_d<128, false>);
    return launch(p, q, k, v, modality, text_pos, o, q_text, row_stats, work_counter, status, sms,
                  stream);
}

}  // namespace tgvkv
