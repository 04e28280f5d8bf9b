// Causal prefill on the 5th-generation tensor cores (tcgen05.mma, accumulators in tensor memory).
//
// One CTA owns two 128-row sub-tiles whose S = Q K^T and O += P V products ping-pong on the tensor
// pipe while the other sub-tile's softmax runs on the CUDA cores. The two sub-tiles are the same 128
// query rows of TWO query heads that share a KV head (query-head groups of even size: both sub-tiles
// then visit the same K/V tiles, their causal spans are equal, and work items are half as coarse), or
// 256 consecutive rows of ONE query head (odd group sizes, multi-head attention included).
//
//   warps 0-3   softmax of sub-tile 0: thread t owns row t (= TMEM lane t): reads S from TMEM,
//               keeps the running max / sum in fp32, writes P (bf16) back into TMEM over S
//   warps 4-7   the same for sub-tile 1
//   warp  8     TMA producer: Q, then K_j, V_j tiles (128 tokens, 128-byte swizzle) through a ring of shared-memory slots, item
//               after item
//   warp  9     MMA issuer (one lane): S_i = Q_i K_j^T from shared memory, O_i += P_i V_j with P read
//               from TMEM and V as an MN-major shared-memory operand; owns the TMEM allocation
//   warps 10-11 what leaves: the block's diagonal K/V tiles into the KV cache (first query head of a KV group only), output rows
//
// A CTA that is through with its block goes on with blocks of the launch that have not started (cluster launch control), until none is
// left: the next item's loads run ahead through the ring under the last tiles of the present one, and its first product follows the
// last of this one. A block of its own for every item paid 5.7 us of launch, set-up, first loads and last stores around its tiles; an item
// that follows another pays 1.3. The claim comes when the item's last loads are on their way, about two tile pairs ahead of its end: later
// than that the loads would start late, earlier the order of the heaviest first would suffer. The MMA issuer's warp has uniform control flow
// (values broadcast, one vote per tile, an elected lane): with branches per lane a tile pair took 3500-3640 cycles instead of 3250-3350,
// which is more than the items gain. Figures (kept up, where the power cap sets the clock; a block per item first): four prompts of 8192 2198 and
// 2129 us, one of 2048 45.1 and 43.5, six of 517 to 1592 with the rotation 139.7 and 128.0, five paged chunks 117.7 and 116.0.
//
// The same kernel serves a chunk of new tokens over a populated cache. The key axis of a sequence is then two runs
// of 128-token tiles: the `past` tokens cached before (tiles of the cache, contiguous or paged, aligned to slot 0;
// every query row sees all of them, the last tile may be partly filled) followed by the new tokens (tiles aligned
// to the chunk's first token, so the causal diagonal sits exactly as in a fresh prompt, which is the case past = 0).
// The new tokens' K/V come from the caller's tensors (and are written to the cache in the same pass) or, when the
// caller has appended them already, from the cache itself at slot past + row.
// A whole sub-tile's output leaves through two slots of the ring and TMA stores.
//
// TMEM columns: S0 [0,128) S1 [128,256) O0 [256,256+D) O1 [256+D,256+2D); P_i aliases the first 64
// columns of S_i. Causal tile skipping: sub-tile i only visits K/V tiles up to its diagonal.
// The tensor pipe executes one thread's MMAs in issue order, which is what makes the S/P aliasing
// safe: QK_{j+1} into S_i is issued after PV_j that reads P_i.
#include "l4l_internal.h"
#include "l4l_ptx.cuh"

namespace l4l {

namespace {

constexpr int kRows = 128;                     // rows per sub-tile == tokens per K/V tile
constexpr int kThreads = 384;                  // 3 warpgroups: softmax 0, softmax 1, {producer, MMA, 2 that move rows to the cache and out}
constexpr uint32_t kHalfBytes = kRows * 128;   // [128 rows][64 bf16], 128-byte swizzled
constexpr int kItemReaders = 11;               // warps that read an item: all but the producer's
constexpr float kRescaleThreshold = 8.f;       // log2 domain: O is rescaled only if the max grew by > 2^8

template <int D>
struct TcCfg {
    static constexpr int kHalves = D / 64;
    static constexpr uint32_t kTileBytes = kHalves * kHalfBytes;        // one Q sub-tile, K tile or V tile
    static constexpr int kSlots = (D == 128) ? 5 : 8;                    // ring of K/V tiles
    static constexpr uint32_t kTmemCols = 512;
    static constexpr uint32_t kColS0 = 0, kColS1 = 128, kColO0 = 256, kColO1 = 256 + D;
    static constexpr int kNumBars = (2 * kSlots + 21 + 1) & ~1;          // even: what follows them is 16-byte aligned
    static constexpr size_t kSmemBytes = 1024 + 2 * kTileBytes + (size_t)kSlots * kTileBytes + kNumBars * 8 + 16 + 2 * 64 + 16;
};

struct TcParams {
    __nv_bfloat16 *o;
    int64_t o_sb, o_st, o_sh;
    __nv_bfloat16 *cache_k, *cache_v;   // destination of the fused cache write (null: nothing is written)
    int64_t c_sb, c_sh, c_st;           // its strides (paged: c_sb is the stride between pages)
    const __nv_bfloat16 *k_new, *v_new; // the new tokens' K/V, for the rows that do not go to the cache from shared memory
    int64_t k_sb, k_st, k_sh, v_sb, v_st, v_sh;
    int cache_slots;                    // token slots per sequence that may be written
    const int32_t *seq_lens;            // [B] new tokens per sequence (prompt or chunk length)
    const int32_t *past_lens;           // [B] tokens cached ahead of them, or null (none)
    const int32_t *block_table;         // paged cache: [B, table_stride] page ids; null: contiguous cache
    int table_stride, page_shift, page_size, num_pages;
    int new_at_past;                    // the new tokens' K/V are read from the cache itself: row r is slot past + r
    int cache_box_t;                    // token rows per TMA box of a cache tile (128, or the page size if smaller)
    float *lse;
    unsigned *status;
    int S_max, B, Hq, Hkv, G, n_qblocks;
    int claims;                         // a CTA goes on with blocks that have not started (every launch that comes here has them)
    int cache_tma;                      // whole tiles are written to the cache by TMA, through the maps of the cache
    int pair_heads;                     // the two sub-tiles are two query heads of one KV group at the same 128 rows
    float scale_log2e;
    TmapCoord cq, ckv, co, ckc;         // ckv: maps of the new tokens' K/V; ckc: maps of the cache (tokens before)
};

__device__ __forceinline__ void order_coords(const TmapCoord &c, int t, int h, int b, int &c1, int &c2, int &c3)
{
    c1 = (c.pos_t == 1) ? t : (c.pos_h == 1) ? h : b;
    c2 = (c.pos_t == 2) ? t : (c.pos_h == 2) ? h : b;
    c3 = (c.pos_t == 3) ? t : (c.pos_h == 3) ? h : b;
}

// Shared-memory matrix descriptor, 128-byte swizzle, 8-row groups 1024 bytes apart.
// K-major operands ignore the leading byte offset; MN-major ones use it as the stride between
// 64-element chunks along M/N.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t smem_addr, uint32_t lbo_bytes)
{
    constexpr uint32_t hi = (1024u >> 4) |      // stride between 8-row groups
                            1u << 14 |          // descriptor version for sm_100
                            2u << 29;           // SWIZZLE_128B
    return pack_u32x2((smem_addr >> 4) | ((lbo_bytes >> 4) << 16), hi);
}

// Instruction descriptor: bf16 x bf16 -> fp32, M = 128.
__host__ __device__ constexpr uint32_t make_idesc(int n, bool b_mn_major)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(kRows >> 4) << 24);
}

// Which row block the block group `g` (the blocks of all heads of one row block) works on when up to 32 sequences have different
// pasts: row blocks are ranked by their work, i.e. the key tiles they visit, heaviest first. Row block qb of a sequence has
// past + (qb + 1) << shift tiles, so the ranking needs no sort: the largest w with more than g row blocks of weight >= w is the
// weight of rank g, found by bisection with a count over the sequences; equal weights go by sequence. A whole warp calls this,
// lane l with the lengths of sequence l (0 past the last). Returns false past the last row block that holds rows.
__device__ __forceinline__ bool row_block_by_work(int len, int past_len, int S_max, int row_shift, int shift, int g, int &b, int &qb)
{
    const int past = (max(past_len, 0) + kRows - 1) / kRows;
    const int blocks = (min(max(len, 0), S_max) + (1 << row_shift) - 1) >> row_shift;
    if (g >= (int)__reduce_add_sync(0xffffffffu, (unsigned)blocks)) return false;
    auto at_least = [&](int w) {
        return (int)__reduce_add_sync(0xffffffffu, (unsigned)max(0, blocks - max(0, ((w - past + (1 << shift) - 1) >> shift) - 1)));
    };
    const unsigned top = blocks > 0 ? (unsigned)(past + (blocks << shift)) : 0u;
    int lo = 1, hi = (int)__reduce_max_sync(0xffffffffu, top) + 1;                     // at_least(lo) > g >= at_least(hi)
    int above = 0;                                                                     // at_least(hi)
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1, n = at_least(mid);
        if (n > g) lo = mid; else hi = mid, above = n;
    }
    // the row block of this very weight with g - above of them ahead (a sequence has one at most)
    const int off = lo - past;
    unsigned who = __ballot_sync(0xffffffffu, off > 0 && (off >> shift) << shift == off && off >> shift <= blocks);
    for (int skip = g - above; skip > 0; --skip) who &= who - 1;
    b = __ffs(who) - 1;
    qb = (__shfl_sync(0xffffffffu, off, b) >> shift) - 1;
    return true;
}

// One work item: 128 rows of two query heads of a KV group, or 256 rows of one head.
struct Item {
    int b, qb, h, kvh;           // sequence, row block, (first) query head and its KV head
    int L, past;                 // new tokens of the sequence, tokens cached ahead of them
    int n_cache;                 // key tiles of the past
    int n_sub0, n_sub1, n_kv;    // key tiles that each sub-tile visits, and the longer of the two
    int g;                       // ring entries used before it
    int share, n_shares;         // which part of its diagonal tiles' rows goes to the cache from here, of how many (0: nothing is written)
    int valid;                   // 0: nothing to do (past the end of its sequence, or no item left)
};

// kRanked: row blocks in the order of their work, not of their place in the sequence (an instantiation of its own: fresh
// prompts do not pay for it)
template <int D, bool kRanked>
__global__ void __launch_bounds__(kThreads, 1)
prefill_tc_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                  const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_o,
                  const __grid_constant__ CUtensorMap tmap_kc, const __grid_constant__ CUtensorMap tmap_vc,
                  const TcParams p)
{
    using C = TcCfg<D>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    uint8_t *q_smem = smem;                                       // 2 sub-tiles
    uint8_t *ring = smem + 2 * C::kTileBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(ring + (size_t)C::kSlots * C::kTileBytes);
    uint64_t *kv_full = bars;
    uint64_t *kv_empty = kv_full + C::kSlots;     // two arrivals: the MMAs, and whoever else reads the slot (or the producer for them)
    uint64_t *q_full = kv_empty + C::kSlots;
    uint64_t *q_empty = q_full + 1;               // the last Q K^T of the item is done
    uint64_t *claim_bar = q_empty + 1;
    uint64_t *s_full = claim_bar + 1;             // [2]
    uint64_t *o_full = s_full + 2;                // [2]
    // One for even, one for odd items: a role may be a whole item behind another, and never two (the place of an item in shared
    // memory is filled again only when all its readers have left it), so that a phase is never passed by unseen.
    uint64_t *item_full = o_full + 2;             // [2] the item is known
    uint64_t *loads_issued = item_full + 2;       // [2] all its tiles have been asked for
    uint64_t *o_granted = loads_issued + 2;       // [2] the slots for its output rows are free
    uint64_t *item_empty = o_granted + 2;         // [2] its readers have left it
    uint64_t *p_full = item_empty + 2;            // [2]
    uint64_t *o_staged = p_full + 2;              // [2][2] a sub-tile's output rows are in shared memory (or written directly)
    uint4 *claim = reinterpret_cast<uint4 *>(bars + C::kNumBars);         // answer to the request for a block
    Item *items = reinterpret_cast<Item *>(claim + 1);                    // [2]
    uint32_t *tmem_base_smem = reinterpret_cast<uint32_t *>(items + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_base_smem + 1);

    // Set-up that depends on nothing the kernel before writes, and overlaps its tail. The producer's warp sets the barriers up itself,
    // a lane each, so that its first loads need not wait for the other warps at the block-wide barrier below.
    if (warp == 8) {
        for (int i = lane; i < (int)(o_staged + 4 - bars); i += 32) {
            uint64_t *bar = bars + i;
            mbar_init(bar, bar >= p_full ? kRows : bar >= item_empty ? kItemReaders : bar >= kv_empty && bar < q_full ? 2 : 1);
        }
        if (lane == 0) {
            *abort_flag = 0;
            tma_prefetch_desc(&tmap_q);
            tma_prefetch_desc(&tmap_k);
            tma_prefetch_desc(&tmap_v);
            tma_prefetch_desc(&tmap_kc);
            tma_prefetch_desc(&tmap_vc);
        }
        fence_barrier_init();
        fence_proxy_async_smem();
        __syncwarp();
    }
    if (D == 128 && warp == 9) {
        tmem_alloc(tmem_base_smem, C::kTmemCols);
        tmem_relinquish_alloc_permit();
    }
    grid_dependency_wait();                       // the lengths may have been written by the previous kernel
    // With 128-wide heads no other block fits beside this one, and tensor memory is there for the taking; with 64-wide heads one
    // might, and if the kernel waited for lets its dependents start before it has taken its own, each would wait for the other.
    if (D != 128 && warp == 9) {
        tmem_alloc(tmem_base_smem, C::kTmemCols);
        tmem_relinquish_alloc_permit();
    }

    // pair mode: sub-tile i is query head h + i at rows q0 ..; else: head h at rows q0 + 128 i ..
    const bool pair = p.pair_heads != 0;
    const int heads = pair ? p.Hq / 2 : p.Hq;
    const int sub_rows = pair ? 0 : kRows;                // rows between the two sub-tiles
    const int sub_heads = pair ? 1 : 0;                   // heads between them
    const int tiles_per_block = pair ? 1 : 2;             // new tiles from one row block to the next

    // Up to 32 sequences: lane l of the producer's warp keeps the lengths of sequence l.
    int len_of = 0, past_of = 0;
    if (warp == 8 && lane < p.B && p.B > 1 && p.B <= 32) {
        len_of = __ldg(p.seq_lens + lane);
        past_of = p.past_lens ? __ldg(p.past_lens + lane) : 0;
    }
    // Block `index` of the launch: heaviest (longest causal span) blocks first, heads of a KV group adjacent. The whole warp calls this.
    auto item_of = [&](int index) {
        Item it = {};
        const int per_block = heads * p.B;
        it.qb = p.n_qblocks - 1 - index / per_block;      // block of 128 (pair mode) or 256 rows
        const int hb = index % per_block;
        it.h = pair ? 2 * (hb % heads) : hb % heads;
        it.b = hb / heads;
        it.kvh = it.h / p.G;
        it.share = pair ? (it.h - it.kvh * p.G) >> 1 : it.h - it.kvh * p.G;
        it.n_shares = p.cache_k == nullptr ? 0 : pair ? p.G >> 1 : p.G;
        it.valid = 1;
        int L_raw, past_raw;
        if (kRanked) {
            L_raw = __shfl_sync(0xffffffffu, len_of, it.b);
            past_raw = __shfl_sync(0xffffffffu, past_of, it.b);
            // With equal pasts (every fresh prompt) the order of places is the order of work, and this vote is all that is paid for.
            if (__builtin_expect(!__all_sync(0xffffffffu, lane >= p.B || past_of == past_raw), 0)) {
                it.valid = row_block_by_work(len_of, past_of, p.S_max, pair ? 7 : 8, pair ? 0 : 1, index / heads, it.b, it.qb);
                it.b = it.valid ? it.b : 0;
                L_raw = __shfl_sync(0xffffffffu, len_of, it.b);
                past_raw = __shfl_sync(0xffffffffu, past_of, it.b);
            }
        } else if (p.B > 1 && p.B <= 32) {
            // By place, the row blocks past the ends of their sequences left out (they would be passed over one by one, a request each): the
            // place is the largest that has more than `left` row blocks at it or above, found by bisection.
            const int blocks = (min(max(len_of, 0), p.S_max) + tiles_per_block * kRows - 1) / (tiles_per_block * kRows);
            const int left = index / heads;
            auto from = [&](int qb) { return (int)__reduce_add_sync(0xffffffffu, (unsigned)max(0, blocks - qb)); };
            int lo = -1, hi = (int)__reduce_max_sync(0xffffffffu, (unsigned)blocks), above = 0;        // from(hi) = above <= left
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1, n = from(mid);
                if (n > left) lo = mid; else hi = mid, above = n;
            }
            it.qb = lo;
            it.valid = lo >= 0;
            unsigned who = __ballot_sync(0xffffffffu, blocks > lo);
            for (int skip = it.valid ? left - above : 0; skip > 0; --skip) who &= who - 1;
            it.b = it.valid ? __ffs(who) - 1 : 0;
            L_raw = __shfl_sync(0xffffffffu, len_of, it.b);
            past_raw = __shfl_sync(0xffffffffu, past_of, it.b);
        } else {
            L_raw = __ldg(p.seq_lens + it.b);
            past_raw = p.past_lens ? __ldg(p.past_lens + it.b) : 0;
        }
        const int q0 = it.qb * tiles_per_block * kRows;
        it.L = L_raw < 0 ? 0 : (L_raw > p.S_max ? p.S_max : L_raw);
        // a block past the end of its sequence has nothing to do (and no rows, for a role that still reads an item whose place it takes after
        // a dead wait)
        if (q0 >= it.L || q0 < 0) it.valid = it.qb = it.L = 0;
        // Tokens already in the cache ahead of these (0 for a fresh prompt): n_cache tiles, seen by every row.
        it.past = past_raw < 0 ? 0 : past_raw;
        it.n_cache = (it.past + kRows - 1) / kRows;
        // sub-tile i (rows q0 + 128 i ..) visits the tiles of the past and the new tokens' tiles up to its diagonal
        it.n_sub0 = it.n_cache + min(q0 + kRows - 1, it.L - 1) / kRows + 1;
        it.n_sub1 = (q0 + sub_rows < it.L) ? it.n_cache + min(q0 + sub_rows + kRows - 1, it.L - 1) / kRows + 1 : 0;
        it.n_kv = max(it.n_sub0, it.n_sub1);
        return it;
    };

    // Whether key tile j goes to the cache from a slot of the ring, by TMA: a whole diagonal tile, contiguous cache. (What does not is
    // copied from the caller's tensors, so that no slot waits for a copy row by row.)
    auto whole_by_tma = [&](const Item &x, int j) {
        const int r_base = (j - x.n_cache) * kRows;
        return x.n_shares > 0 && p.cache_tma && j >= x.n_cache + tiles_per_block * x.qb && min(x.L, p.cache_slots - x.past) - r_base >= kRows;
    };
    auto leaves_ring = [&](const Item &x, int j) { return x.share == 0 && whole_by_tma(x, j); };
    // ---- what the producer asks for (one lane: copies asked for by several lanes of a warp are issued one by one, at many times the
    // cost). Ring entries of an item: K_0, V_0, K_1, V_1, ... then one for each sub-tile's output rows on their way out. `g` counts entries
    // over all items of this block.
    auto request_q = [&](const Item &x, int i) {
        int c1, c2, c3;
        order_coords(p.cq, x.qb * tiles_per_block * kRows + i * sub_rows, x.h + i * sub_heads, x.b, c1, c2, c3);
#pragma unroll
        for (int hf = 0; hf < C::kHalves; ++hf)
            tma_load_4d(q_smem + i * C::kTileBytes + hf * kHalfBytes, &tmap_q, q_full, hf * 64, c1, c2, c3);
    };
    auto request_tile = [&](const Item &x, int g, int idx) {
        const uint32_t s = g % C::kSlots;
        const int j = idx >> 1;
        uint8_t *dst = ring + (size_t)s * C::kTileBytes;
        int c1, c2, c3;
        if (!leaves_ring(x, j)) mbar_arrive(&kv_empty[s]);        // no second reader
        mbar_arrive_expect_tx(&kv_full[s], C::kTileBytes);
        if (j >= x.n_cache) {
            // a tile of the new tokens
            order_coords(p.ckv, (p.new_at_past ? x.past : 0) + (j - x.n_cache) * kRows, x.kvh, x.b, c1, c2, c3);
            const CUtensorMap *tm = (idx & 1) ? &tmap_v : &tmap_k;
#pragma unroll
            for (int hf = 0; hf < C::kHalves; ++hf) tma_load_4d(dst + hf * kHalfBytes, tm, &kv_full[s], hf * 64, c1, c2, c3);
        } else if (p.block_table == nullptr) {
            // a tile of the tokens cached before, contiguous cache
            order_coords(p.ckc, j * kRows, x.kvh, x.b, c1, c2, c3);
            const CUtensorMap *tm = (idx & 1) ? &tmap_vc : &tmap_kc;
#pragma unroll
            for (int hf = 0; hf < C::kHalves; ++hf) tma_load_4d(dst + hf * kHalfBytes, tm, &kv_full[s], hf * 64, c1, c2, c3);
        } else {
            // ... paged cache: one box per page that the tile touches (a page never straddles tiles or boxes), four look-ups at a
            // time. A table entry outside the pool becomes an out-of-range coordinate, which reads zeros.
            const CUtensorMap *tm = (idx & 1) ? &tmap_vc : &tmap_kc;
            const int32_t *row = p.block_table + (size_t)x.b * p.table_stride;
            for (int at = 0; at < kRows; at += 4 * p.cache_box_t) {
                int page[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int r0 = at + u * p.cache_box_t, entry = (j * kRows + r0) >> p.page_shift;
                    page[u] = r0 < kRows && entry < p.table_stride ? __ldg(row + entry) : -1;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int r0 = at + u * p.cache_box_t;
                    if (r0 >= kRows) break;
                    order_coords(p.ckc, (j * kRows + r0) & (p.page_size - 1), x.kvh, page[u] < 0 || page[u] >= p.num_pages ? p.num_pages : page[u], c1, c2, c3);
#pragma unroll
                    for (int hf = 0; hf < C::kHalves; ++hf)
                        tma_load_4d(dst + hf * kHalfBytes + r0 * 128, tm, &kv_full[s], hf * 64, c1, c2, c3);
                }
            }
        }
    };
    // What the first products need is requested before the block-wide barrier, the rest behind it
    Item next = {};
    if (warp == 8) {
        next = item_of(blockIdx.x);
        if (lane == 0 && next.valid) {
            mbar_arrive_expect_tx(q_full, 2 * C::kTileBytes);
            request_q(next, 0);
            request_tile(next, 0, 0);                      // K_0 right behind Q_0: the first product needs both
            request_q(next, 1);
            next.g = 0;
            items[0] = next;
            mbar_arrive(&item_full[0]);
        }
    }
    tcgen05_fence_before_sync();
    __syncthreads();
    tcgen05_fence_after_sync();
    const uint32_t tmem_base = *tmem_base_smem;

    // Every role but the producer takes its items like this, and reads them where the producer leaves them (a copy in registers
    // would cost the softmax warps spills). An item is given back when the next one is asked for.
    int n_read = 0;
    auto all_wait = [&](uint64_t *bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)); };
    auto next_item = [&]() {
        if (n_read > 0) {
            __syncwarp();
            if (lane == 0) mbar_arrive(&item_empty[(n_read - 1) & 1]);
        }
        if (!all_wait(&item_full[n_read & 1], (n_read >> 1) & 1u)) return false;
        ++n_read;
        return items[(n_read - 1) & 1].valid != 0;
    };
    auto item = [&]() { return items + ((n_read - 1) & 1); };

    // Register reallocation: the data-movement warpgroup gives registers to the softmax warpgroups,
    // whose threads hold a whole 128-column score row.
    if (warp >= 8) {
    setmaxnreg_dec<72>();
    if (warp == 8) {
        // ============================================================ TMA producer; takes over blocks that have not started
        int g = next.valid ? 1 : 0, idx = g, n_items = 0;
        unsigned n_asked = 0;
        bool ok = true;
        auto wait_slot = [&]() { return mbar_wait(&kv_empty[g % C::kSlots], ((g / C::kSlots) & 1u) ^ 1u, abort_flag); };
        while (true) {
            // the others learn of the item first (of there being none only where nothing follows)
            if (lane == 0 && idx == 0 && (next.valid || !p.claims || n_asked > 0)) {
                next.g = g;
                if (n_items >= 2) ok = mbar_wait(&item_empty[n_items & 1], ((n_items >> 1) - 1) & 1u, abort_flag);
                items[n_items & 1] = next;
                mbar_arrive(&item_full[n_items & 1]);
            }
            if (!next.valid && (!p.claims || n_asked > 0)) break;
            if (next.valid) {
                if (lane == 0) {
                    if (ok && idx == 0) {
                        ok = n_items == 0 || mbar_wait(q_empty, (n_items - 1) & 1u, abort_flag);
                        if (ok) {
                            mbar_arrive_expect_tx(q_full, 2 * C::kTileBytes);
                            request_q(next, 0);
                        }
                    }
                    for (; ok && idx < 2 * next.n_kv; ++idx, ++g) {
                        ok = wait_slot();
                        if (!ok) break;
                        request_tile(next, g, idx);
                        if (idx == 0) request_q(next, 1);
                    }
                    if (ok) mbar_arrive(&loads_issued[n_items & 1]);
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
            }
            // the next item: a block of the launch that no SM has started (those past the end of their sequence are passed over)
            const bool had_item = next.valid;
            next.valid = 0;
            while (p.claims && !next.valid) {
                int index = -1;
                if (lane == 0) {
                    mbar_arrive_expect_tx(claim_bar, 16);
                    clc_try_cancel(claim, claim_bar);
                    if (mbar_wait(claim_bar, n_asked & 1u, abort_flag)) index = clc_answer(claim);
                    fence_proxy_async_smem();              // the answer has been read before the next one is written
                }
                ++n_asked;
                index = __shfl_sync(0xffffffffu, index, 0);
                if (index < 0) break;
                next = item_of(index);
            }
            if (had_item) {
                // the slots that the outputs of the two sub-tiles leave through: theirs from here on
                if (lane == 0) {
                    for (int i = 0; ok && i < 2; ++i, ++g) {
                        ok = wait_slot();
                        if (ok) {
                            mbar_arrive(&kv_empty[g % C::kSlots]);
                            mbar_arrive(&kv_full[g % C::kSlots]);          // its phase, which nobody waits for
                        }
                    }
                    if (ok) mbar_arrive(&o_granted[n_items & 1]);
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                ++n_items;
                idx = 0;
            }
        }
        // Programmatic dependent launch: the next kernel of the stream may set itself up from here on, while the last items end. (As soon
        // as every block had started, its blocks settled on the SMs that fell idle first, in no order: 5 chunks of 202, 647, 129, 326 and
        // 185 tokens over 563 to 3057, launches back to back 59.3 us, in this place 56.0, with a block per item 55.7.)
        grid_launch_dependents();
        if (lane == 0 && !ok) {                            // a dead wait: the block leaves when what it asked for has landed
            volatile int keep_waiting = 0;
            for (int e = max(0, g - C::kSlots); e < g; ++e)
                mbar_wait_budget(&kv_full[e % C::kSlots], (e / C::kSlots) & 1u, &keep_waiting, kWaitCycleBudget >> 6);
            if (n_asked > 0) mbar_wait_budget(claim_bar, (n_asked - 1) & 1u, &keep_waiting, kWaitCycleBudget >> 6);
        }
    } else if (warp == 10 || warp == 11) {
        // ============================================================ what leaves through shared memory
        // Warp 10: the diagonal K tiles into the cache, output rows of sub-tile 0; warp 11: V and sub-tile 1. An item's diagonal
        // tiles (one or two tiles of the new tokens, from its own rows on) go to the cache at slot past + row, each row once: a
        // tile that leaves by TMA from the first query head of a KV group, the rows of the others in equal shares from all items of the
        // group. Rows >= L and slots the cache does not have are not written.
        // First: if an earlier CTA of this launch already reported a dead wait, do not repeat its time-out in every remaining CTA.
        const int part = warp - 10;
        if (part == 0 && lane == 0 && *reinterpret_cast<volatile unsigned *>(p.status + kStatusErrWord) != 0u)
            *abort_flag = 1;
        bool ok = true;
        while (next_item()) {
            const int g = item()->g;
            const int ev = (n_read - 1) & 1;                  // even or odd item, and its phase
            const uint32_t item_ph = ((n_read - 1) >> 1) & 1u;
            if (item()->n_shares > 0) {
                const int kvh = item()->kvh, past = item()->past, b = item()->b;
                for (int j = item()->n_cache + tiles_per_block * item()->qb; j < item()->n_kv; ++j) {
                    const int r_base = (j - item()->n_cache) * kRows;       // first row of the tile among the new tokens
                    if (whole_by_tma(*item(), j)) {
                        if (item()->share != 0) continue;
                        // (before this the slot may be in an earlier phase, whose parity may be that of the one waited for)
                        const int e = g + 2 * j + part;
                        if (!all_wait(&loads_issued[ev], item_ph) || !all_wait(&kv_full[e % C::kSlots], (e / C::kSlots) & 1u)) { ok = false; break; }
                        if (lane == 0) {
                            const uint8_t *src = ring + (size_t)(e % C::kSlots) * C::kTileBytes;
                            int c1, c2, c3;
                            order_coords(p.ckc, past + r_base, kvh, b, c1, c2, c3);
#pragma unroll
                            for (int hf = 0; hf < C::kHalves; ++hf)
                                tma_store_4d(part ? &tmap_vc : &tmap_kc, src + hf * kHalfBytes, hf * 64, c1, c2, c3);
                            tma_store_commit();
                            tma_store_wait_read_all();
                            mbar_arrive(&kv_empty[e % C::kSlots]);
                        }
                        __syncwarp();
                        continue;
                    }
                    // A lane keeps its 16-byte column and goes down the rows, four at a time; a new page is looked up where one begins. A tile
                    // copied by one warp (sixteen round trips of 1 us for 128 rows) outlasted the products of short items; the rows
                    // are shared out among the items of the KV group instead: 3 chunks of 300..600 over 64..300 in 64-token pages, 40/8 x 128
                    // 60.2 -> 41.7 us, 32/8 35.8 -> 28.8, 64/8 53.6 -> 42.7. (More rows at a time: these warps then spill.)
                    constexpr int kChunks = D / 8, kStep = 32 / kChunks, kBatch = 4;
                    const int all = max(0, min(min(kRows, item()->L - r_base), p.cache_slots - past - r_base));
                    const int rows = all * (item()->share + 1) / item()->n_shares;
                    const int ch = lane % kChunks;
                    const __nv_bfloat16 *const src = (part ? p.v_new : p.k_new) + b * (part ? p.v_sb : p.k_sb) + kvh * (part ? p.v_sh : p.k_sh) +
                                                     (int64_t)r_base * (part ? p.v_st : p.k_st) + ch * 8;
                    const int64_t src_st = part ? p.v_st : p.k_st;
                    __nv_bfloat16 *const base = (part ? p.cache_v : p.cache_k) + kvh * p.c_sh + ch * 8;
                    __nv_bfloat16 *page_at = p.block_table ? nullptr : base + b * p.c_sb;
                    int page_of = -1;
                    for (int r0 = all * item()->share / item()->n_shares + lane / kChunks; r0 < rows; r0 += kStep * kBatch) {
                        uint4 val[kBatch];
#pragma unroll
                        for (int u = 0; u < kBatch; ++u) {
                            const int r = r0 + u * kStep;
                            if (r < rows) val[u] = *reinterpret_cast<const uint4 *>(src + r * src_st);
                        }
#pragma unroll
                        for (int u = 0; u < kBatch; ++u) {
                            const int r = r0 + u * kStep;
                            if (r >= rows) break;
                            int slot = past + r_base + r;
                            if (p.block_table) {
                                const int entry = slot >> p.page_shift;
                                if (entry != page_of) {
                                    page_of = entry;
                                    const int pg = __ldg(p.block_table + (size_t)b * p.table_stride + entry);
                                    page_at = pg < 0 || pg >= p.num_pages ? nullptr : base + (int64_t)pg * p.c_sb;   // null: no page behind this slot
                                }
                                slot &= p.page_size - 1;
                            }
                            if (page_at) *reinterpret_cast<uint4 *>(page_at + (int64_t)slot * p.c_st) = val[u];
                        }
                    }
                    __syncwarp();
                }
            }
            if (!ok) break;
            const int e = g + 2 * item()->n_kv + part, q0 = item()->qb * tiles_per_block * kRows + part * sub_rows;
            if (!all_wait(&o_granted[ev], item_ph) || !all_wait(&o_staged[2 * ev + part], item_ph)) break;
            if (q0 + kRows <= item()->L && lane == 0) {
                const uint8_t *stage = ring + (size_t)(e % C::kSlots) * C::kTileBytes;
                int c1, c2, c3;
                order_coords(p.co, q0, item()->h + part * sub_heads, item()->b, c1, c2, c3);
#pragma unroll
                for (int hf = 0; hf < C::kHalves; ++hf) tma_store_4d(&tmap_o, stage + hf * kHalfBytes, hf * 64, c1, c2, c3);
                tma_store_commit();
                tma_store_wait_read_all();                         // shared memory must outlive the reads
            }
            if (lane == 0) mbar_arrive(&kv_empty[e % C::kSlots]);
        }
    } else if (warp == 9) {
        // ============================================================ MMA issuer
        constexpr uint32_t idesc_qk = make_idesc(kRows, false);
        constexpr uint32_t idesc_pv = make_idesc(D, true);
        const uint32_t tmem_s[2] = {tmem_base + C::kColS0, tmem_base + C::kColS1};
        const uint32_t tmem_o[2] = {tmem_base + C::kColO0, tmem_base + C::kColO1};
        const uint32_t q_addr = smem_u32(q_smem), ring_addr = smem_u32(ring);

        auto issue_qk = [&](int i, uint32_t k_addr) {
#pragma unroll
            for (int k = 0; k < D / 16; ++k) {
                const uint32_t off = (k >> 2) * kHalfBytes + (k & 3) * 32;
                tcgen05_mma_ss(tmem_s[i], make_smem_desc(q_addr + i * C::kTileBytes + off, 0),
                               make_smem_desc(k_addr + off, 0), idesc_qk, k > 0 ? 1u : 0u);
            }
        };
        auto issue_pv = [&](int i, uint32_t v_addr, bool first) {
#pragma unroll
            for (int k = 0; k < kRows / 16; ++k)
                tcgen05_mma_ts(tmem_o[i], tmem_s[i] + k * 8, make_smem_desc(v_addr + k * 2048, kHalfBytes), idesc_pv,
                               (first && k == 0) ? 0u : 1u);
        };

        uint32_t q_ph = 0, p_ph[2] = {0, 0};
        bool ok = true;
        while (ok && next_item()) {
            // (broadcast, so that the compiler knows them to be the same in all lanes)
            const int n_kv = __shfl_sync(0xffffffffu, item()->n_kv, 0), g = __shfl_sync(0xffffffffu, item()->g, 0);
            const int n_sub[2] = {__shfl_sync(0xffffffffu, item()->n_sub0, 0), __shfl_sync(0xffffffffu, item()->n_sub1, 0)};
            const int n_cache = __shfl_sync(0xffffffffu, item()->n_cache, 0), past = __shfl_sync(0xffffffffu, item()->past, 0);
            const int L = __shfl_sync(0xffffffffu, item()->L, 0);
            ok = all_wait(q_full, q_ph) && all_wait(&kv_full[g % C::kSlots], (g / C::kSlots) & 1u);
            q_ph ^= 1u;
            if (!ok) break;
            tcgen05_fence_after_sync();
            if (elect_one()) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (n_sub[i] > 0) {
                        issue_qk(i, ring_addr + (g % C::kSlots) * C::kTileBytes);
                        tcgen05_commit(&s_full[i]);
                    }
                tcgen05_commit(&kv_empty[g % C::kSlots]);
                if (n_kv == 1) tcgen05_commit(q_empty);
            }
            __syncwarp();
            for (int j = 0; j < n_kv; ++j) {
                const int iv = g + 2 * j + 1, ik = g + 2 * j + 2;
                const uint32_t sv = iv % C::kSlots, sk = ik % C::kSlots;
                ok = mbar_wait(&kv_full[sv], (iv / C::kSlots) & 1u, abort_flag);
                // V rows >= this hold no valid token (the partly filled last tile of the past, or of the new tokens)
                const int first_dead = j < n_cache ? past - j * kRows : L - (j - n_cache) * kRows;
                if (first_dead < kRows) {
                    // may hold any bits (NaN included): clear, so that a zero weight times garbage cannot appear
                    uint8_t *vt = ring + (size_t)sv * C::kTileBytes;
                    constexpr int kChunks = D / 8;
                    for (int i = lane; i < (kRows - first_dead) * kChunks; i += 32) {
                        const int r = first_dead + i / kChunks, ch = i % kChunks;
                        *reinterpret_cast<uint4 *>(vt + (ch >> 3) * kHalfBytes + r * 128 + ((ch & 7) << 4)) =
                            make_uint4(0u, 0u, 0u, 0u);
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                }
                const bool have_next = j + 1 < n_kv;
                if (have_next) ok = mbar_wait(&kv_full[sk], (ik / C::kSlots) & 1u, abort_flag) && ok;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if (j >= n_sub[i]) continue;
                    ok = mbar_wait(&p_full[i], p_ph[i], abort_flag) && ok;
                    __syncwarp();
                    p_ph[i] ^= 1u;
                    tcgen05_fence_after_sync();
                    if (elect_one()) {
                        issue_pv(i, ring_addr + sv * C::kTileBytes, j == 0);
                        if (j + 1 < n_sub[i]) {
                            issue_qk(i, ring_addr + sk * C::kTileBytes);
                            tcgen05_commit(&s_full[i]);
                        } else {
                            tcgen05_commit(&o_full[i]);
                        }
                    }
                    __syncwarp();
                }
                // (one vote for the waits of the iteration: after a dead one its products are garbage, which the status word says)
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (elect_one()) {
                    tcgen05_commit(&kv_empty[sv]);
                    if (have_next) tcgen05_commit(&kv_empty[sk]);
                    if (j + 2 == n_kv) tcgen05_commit(q_empty);
                }
                __syncwarp();
            }
        }
    }
    } else {
        setmaxnreg_inc<216>();
        // ============================================================ softmax + epilogue warpgroups
        const int i = warp >> 2;                                   // sub-tile
        const int t = threadIdx.x & 127;                           // row within the sub-tile == TMEM lane
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tmem_s = tmem_base + lane_base + (i ? C::kColS1 : C::kColS0);
        const uint32_t tmem_o = tmem_base + lane_base + (i ? C::kColO1 : C::kColO0);
        const float c = p.scale_log2e;
        uint32_t phases = 0;                                       // bit 0: of s_full, bit 1: of o_full
        bool ok = true;

        while (ok && next_item()) {
        const int n_mine = i ? item()->n_sub1 : item()->n_sub0;
        // Tiles that need a mask: the last tile of the past when it is partly filled (columns past its end, the same
        // for every row), and the sub-tile's diagonal tile among the new tokens (row t sees columns 0..t).
        const int j_ragged = (item()->past & (kRows - 1)) ? item()->n_cache - 1 : -1;
        const int j_diag = item()->n_cache + (pair ? item()->qb : 2 * item()->qb + i);
        float m = -INFINITY, l = 0.f;

        for (int j = 0; j < n_mine; ++j) {
            if (!mbar_wait(&s_full[i], phases & 1u, abort_flag)) { ok = false; break; }
            phases ^= 1u;
            tcgen05_fence_after_sync();
            uint32_t sr[4][32];
#pragma unroll
            for (int qd = 0; qd < 4; ++qd) tmem_ld_32x32b_x32(tmem_s + qd * 32, sr[qd]);
            tcgen05_wait_ld();

            // Row maximum of the scaled scores (log2 domain). Off the diagonal the maximum is taken over the
            // raw scores with independent 3-input max chains and scaled once (min for a negative scale);
            // on the diagonal tile the causal mask is applied to the scaled scores first.
            const bool diag = (j == j_ragged) || (j >= j_diag);
            float mx;
            if (diag) {
                const int lim = (j == j_ragged) ? (item()->past & (kRows - 1)) - 1 : t;   // columns > lim hold no visible key
                float a0 = -INFINITY, a1 = -INFINITY, a2 = -INFINITY, a3 = -INFINITY;
#pragma unroll
                for (int qd = 0; qd < 4; ++qd)
#pragma unroll
                    for (int e = 0; e < 32; e += 4) {
                        float x[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            x[u] = __uint_as_float(sr[qd][e + u]) * c;
                            x[u] = (qd * 32 + e + u > lim) ? -INFINITY : x[u];
                            sr[qd][e + u] = __float_as_uint(x[u]);
                        }
                        a0 = fmaxf(a0, x[0]); a1 = fmaxf(a1, x[1]); a2 = fmaxf(a2, x[2]); a3 = fmaxf(a3, x[3]);
                    }
                mx = fmaxf(fmaxf(a0, a1), fmaxf(a2, a3));
            } else if (c >= 0.f) {
                float a0 = -INFINITY, a1 = -INFINITY, a2 = -INFINITY, a3 = -INFINITY;
#pragma unroll
                for (int qd = 0; qd < 4; ++qd)
#pragma unroll
                    for (int e = 0; e < 32; e += 8) {
                        a0 = max3(a0, __uint_as_float(sr[qd][e + 0]), __uint_as_float(sr[qd][e + 1]));
                        a1 = max3(a1, __uint_as_float(sr[qd][e + 2]), __uint_as_float(sr[qd][e + 3]));
                        a2 = max3(a2, __uint_as_float(sr[qd][e + 4]), __uint_as_float(sr[qd][e + 5]));
                        a3 = max3(a3, __uint_as_float(sr[qd][e + 6]), __uint_as_float(sr[qd][e + 7]));
                    }
                mx = fmaxf(fmaxf(a0, a1), fmaxf(a2, a3)) * c;
            } else {
                float a0 = INFINITY, a1 = INFINITY, a2 = INFINITY, a3 = INFINITY;
#pragma unroll
                for (int qd = 0; qd < 4; ++qd)
#pragma unroll
                    for (int e = 0; e < 32; e += 4) {
                        a0 = fminf(a0, __uint_as_float(sr[qd][e + 0]));
                        a1 = fminf(a1, __uint_as_float(sr[qd][e + 1]));
                        a2 = fminf(a2, __uint_as_float(sr[qd][e + 2]));
                        a3 = fminf(a3, __uint_as_float(sr[qd][e + 3]));
                    }
                mx = fminf(fminf(a0, a1), fminf(a2, a3)) * c;
            }
            // lazy rescale: keep the old reference max unless the new one is much larger
            const bool grow = (mx > m + kRescaleThreshold) || (j == 0);
            float alpha = 1.f;
            if (grow) {
                const float m_new = (mx == -INFINITY) ? 0.f : mx;
                alpha = fast_exp2(m - m_new);                      // j == 0: exp2(-inf) = 0
                m = m_new;
                l *= alpha;
            }
            if (j > 0 && __any_sync(0xffffffffu, grow)) {
                // PV_{j-1} has completed (s_full is committed after it), PV_j is not issued before p_full
#pragma unroll
                for (int qd = 0; qd < D / 32; ++qd) {
                    uint32_t orr[32];
                    tmem_ld_32x32b_x32(tmem_o + qd * 32, orr);
                    tcgen05_wait_ld();
#pragma unroll
                    for (int e = 0; e < 32; ++e) orr[e] = __float_as_uint(__uint_as_float(orr[e]) * alpha);
                    tmem_st_32x32b_x32(tmem_o + qd * 32, orr);
                }
            }
            // p = 2^(x - m): packed fp32x2 FMA feeds the exp2 unit; sums in two independent packed chains
            const float fc = diag ? 1.f : c;                       // diagonal scores are already scaled
            const uint64_t c2 = pack_f32x2(fc, fc), nm2 = pack_f32x2(-m, -m);
            uint64_t sum_a = pack_f32x2(0.f, 0.f), sum_b = sum_a;
#pragma unroll
            for (int qd = 0; qd < 4; ++qd) {
                uint32_t pk[16];
#pragma unroll
                for (int e = 0; e < 16; e += 2) {
                    const uint64_t xa = fma_f32x2(pack_u32x2(sr[qd][2 * e], sr[qd][2 * e + 1]), c2, nm2);
                    const uint64_t xb = fma_f32x2(pack_u32x2(sr[qd][2 * e + 2], sr[qd][2 * e + 3]), c2, nm2);
                    float xa0, xa1, xb0, xb1;
                    unpack_f32x2(xa, xa0, xa1);
                    unpack_f32x2(xb, xb0, xb1);
                    const float pa0 = fast_exp2(xa0), pa1 = fast_exp2(xa1);
                    const float pb0 = fast_exp2(xb0), pb1 = fast_exp2(xb1);
                    sum_a = add_f32x2(sum_a, pack_f32x2(pa0, pa1));
                    sum_b = add_f32x2(sum_b, pack_f32x2(pb0, pb1));
                    pk[e] = pack_bf16x2(pa0, pa1);
                    pk[e + 1] = pack_bf16x2(pb0, pb1);
                }
                tmem_st_32x32b_x16(tmem_s + qd * 16, pk);
            }
            float sa0, sa1, sb0, sb1;
            unpack_f32x2(sum_a, sa0, sa1);
            unpack_f32x2(sum_b, sb0, sb1);
            const float sum = (sa0 + sa1) + (sb0 + sb1);
            l += sum;
            tcgen05_wait_st();
            tcgen05_fence_before_sync();
            mbar_arrive(&p_full[i]);
        }

        if (ok && n_mine > 0) {
            ok = mbar_wait(&o_full[i], phases >> 1, abort_flag);
            phases ^= 2u;
            if (!ok) break;
            tcgen05_fence_after_sync();
            const int q0 = item()->qb * tiles_per_block * kRows + i * sub_rows;         // first row of the sub-tile
            const int row = q0 + t, hq = item()->h + i * sub_heads;                      // this thread's query row, its query head
            const float inv = 1.f / l;
            const bool valid = row < item()->L;
            __nv_bfloat16 *orow = p.o + item()->b * p.o_sb + (int64_t)row * p.o_st + hq * p.o_sh;
            // A sub-tile whose 128 rows are all valid leaves through a slot of the ring and one TMA store per 64
            // columns (coalesced, asynchronous, issued by a helper warp). A ragged sub-tile writes its valid rows directly.
            const bool whole = q0 + kRows <= item()->L;
            uint8_t *stage = ring + (size_t)((item()->g + 2 * item()->n_kv + i) % C::kSlots) * C::kTileBytes;
            if (whole && !mbar_wait(&o_granted[(n_read - 1) & 1], ((n_read - 1) >> 1) & 1u, abort_flag)) { ok = false; break; }
#pragma unroll
            for (int qd = 0; qd < D / 32; ++qd) {
                uint32_t orr[32];
                tmem_ld_32x32b_x32(tmem_o + qd * 32, orr);
                tcgen05_wait_ld();
                if (whole) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        uint4 val;
                        val.x = pack_bf16x2(__uint_as_float(orr[8 * e + 0]) * inv, __uint_as_float(orr[8 * e + 1]) * inv);
                        val.y = pack_bf16x2(__uint_as_float(orr[8 * e + 2]) * inv, __uint_as_float(orr[8 * e + 3]) * inv);
                        val.z = pack_bf16x2(__uint_as_float(orr[8 * e + 4]) * inv, __uint_as_float(orr[8 * e + 5]) * inv);
                        val.w = pack_bf16x2(__uint_as_float(orr[8 * e + 6]) * inv, __uint_as_float(orr[8 * e + 7]) * inv);
                        const int ch = qd * 4 + e;                 // 16-byte chunk of the row
                        *reinterpret_cast<uint4 *>(stage + (ch >> 3) * kHalfBytes + swz128(t, ch & 7)) = val;
                    }
                } else if (valid) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        uint4 val;
                        val.x = pack_bf16x2(__uint_as_float(orr[8 * e + 0]) * inv, __uint_as_float(orr[8 * e + 1]) * inv);
                        val.y = pack_bf16x2(__uint_as_float(orr[8 * e + 2]) * inv, __uint_as_float(orr[8 * e + 3]) * inv);
                        val.z = pack_bf16x2(__uint_as_float(orr[8 * e + 4]) * inv, __uint_as_float(orr[8 * e + 5]) * inv);
                        val.w = pack_bf16x2(__uint_as_float(orr[8 * e + 6]) * inv, __uint_as_float(orr[8 * e + 7]) * inv);
                        *reinterpret_cast<uint4 *>(orow + qd * 32 + e * 8) = val;
                    }
                }
            }
            if (whole) fence_proxy_async_smem();                   // this thread's rows, for the TMA store
            if (valid && p.lse)
                p.lse[((size_t)item()->b * p.Hq + hq) * p.S_max + row] = (m + log2f(l)) * 0.6931471805599453f;
        }
        mbar_arrive(&o_staged[2 * ((n_read - 1) & 1) + i]);
        }
    }

    tcgen05_fence_before_sync();
    __syncthreads();
    if (warp == 9) {
        tcgen05_fence_after_sync();
        tmem_dealloc(tmem_base, C::kTmemCols);
    }
    if (threadIdx.x == 0 && *abort_flag) {
        if (atomicOr(p.status + kStatusErrWord, kErrPrefillWait) == 0u)
            p.status[kStatusInfoWord] = 0x20000u | (blockIdx.x & 0xffffu);
    }
}

bool pairs_heads(int G) { return G % 2 == 0; }
int row_blocks(int S_max, int G) { return pairs_heads(G) ? (S_max + kRows - 1) / kRows : (S_max + 2 * kRows - 1) / (2 * kRows); }

// Chunks over caches of different lengths: a row block's work is then set by the tokens cached ahead of it as much as by its
// place, and with the last row blocks first whatever their length the launch ends on a few heavy blocks. Five chunks of
// 180 to 676 tokens over 720 to 4590 in pages: 131.9 us by place, 115.1 by work; 32 chunks of up to 300 over up to 3000 236 and 216.
// One sequence needs no order, and launches of one or two blocks per SM have little to order (two chunks of up to 522 tokens, 160
// blocks: 21.8 us by place, 22.3 by work). Where a cache has room ahead of the chunk the pasts may still be equal, as
// for fresh prompts, and finding that out must cost nothing: with one sequence per lane it is a vote (16 prompts of 512 rotated
// and attended 118.9 us either way). Beyond 32 sequences it was not (40 prompts of up to 300 tokens 129.7 and 131.9 us, 100 of up to 200
// 209.5 and 213.7), for a gain of 2.6 % with 40 chunks and a loss of 1 % with 100. slots: token slots per sequence in the cache (0: no past).
bool row_blocks_by_work(int S_max, long long slots, int B, int Hq, int G)
{
    return slots - S_max >= kRows && B > 1 && B <= 32 &&
           (long long)row_blocks(S_max, G) * (pairs_heads(G) ? Hq / 2 : Hq) * B > 2 * sm_count();
}

// The order for tests: block g reports the (sequence, row block) that the blocks of group g of a ranked launch work on.
__global__ void row_block_order_kernel(const int32_t *past_lens, const int32_t *q_lens, int S_max, int B, int n_qblocks, bool pair, int2 *order)
{
    const int lane = threadIdx.x, g = blockIdx.x;
    int b = g % B, qb = n_qblocks - 1 - g / B;
    const int past = lane < B ? past_lens[lane] : 0, len = lane < B ? q_lens[lane] : 0, past_raw = past_lens[b];
    bool rows = true;
    if (!__all_sync(0xffffffffu, lane >= B || past == past_raw)) rows = row_block_by_work(len, past, S_max, pair ? 7 : 8, pair ? 0 : 1, g, b, qb);
    rows = rows && qb * (pair ? kRows : 2 * kRows) < min(q_lens[b], S_max);
    if (lane == 0) order[g] = rows ? make_int2(b, qb) : make_int2(-1, -1);
}

template <int D, bool kRanked>
l4l_status launch_t(const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv, const CUtensorMap &to,
                    const CUtensorMap &tkc, const CUtensorMap &tvc, const TcParams &p, cudaStream_t stream)
{
    using C = TcCfg<D>;
    static bool configured_on[kDeviceSlots] = {};
    const int slot = device_slot();
    if (slot < 0) return L4L_ERR_CUDA;
    {
        std::lock_guard<std::mutex> lock(setup_mutex());
        bool &configured = configured_on[slot];
        if (!configured) {
            if (cudaFuncSetAttribute(prefill_tc_kernel<D, kRanked>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)C::kSmemBytes) != cudaSuccess)
                return L4L_ERR_CUDA;
            configured = true;
        }
    }
    const long long grid = (long long)p.n_qblocks * (p.pair_heads ? p.Hq / 2 : p.Hq) * p.B;
    if (grid > 0x7fffffffll) return L4L_ERR_UNSUPPORTED;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = C::kSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, prefill_tc_kernel<D, kRanked>, tq, tk, tv, to, tkc, tvc, p) == cudaSuccess ? L4L_OK : L4L_ERR_CUDA;
}

}  // namespace

l4l_status launch_prefill_tc(const l4l_tensor4 &q, const l4l_tensor4 &o, const PrefillKV &kv, const int32_t *d_seq_lens,
                             const int32_t *d_past_lens, int S_max, int B, int Hq, int Hkv, int D, float scale,
                             float *d_lse, void *workspace, cudaStream_t stream)
{
    // A launch of at most one block per SM has nothing to claim (one of 2 blocks 6.8 us with a block per item, 7.1 without), and up to
    // 512 new tokens a block per item was ahead while one item copied all rows of a ragged or paged tile (figures in
    // l4l_prefill_blocks.cu). Since the items share that copy this kernel is ahead in part of that range too: 40 x 512 (32/8 x 128)
    // 192 us with a block per item, 145 here; 16 x 64..512 61 and 52; 12 x 17..64 over 64..500 27.3 and 29.1. Above: 4 x 300..540 with 40/8
    // 36.7 and 34, 8 x 520..640 (32/8) 58.6 and 48.5.
    const long long blocks = (long long)row_blocks(S_max, Hq / Hkv) * (pairs_heads(Hq / Hkv) ? Hq / 2 : Hq) * B;
    if (S_max <= 512 || blocks <= sm_count())
        return launch_prefill_blocks(q, o, kv, d_seq_lens, d_past_lens, S_max, B, Hq, Hkv, D, scale, d_lse, workspace, stream);
    CUtensorMap tq, tk, tv, to, tkc, tvc;
    TmapCoord cq, ck, cv, co, ckc, cvc;
    if (!make_tmap_bf16(&tq, &cq, q.ptr, D, S_max, Hq, B, q.stride_t, q.stride_h, q.stride_b, 64, kRows) ||
        !make_tmap_bf16(&to, &co, o.ptr, D, S_max, Hq, B, o.stride_t, o.stride_h, o.stride_b, 64, kRows) ||
        !make_tmap_bf16(&tk, &ck, kv.k_new.ptr, D, kv.new_extent, Hkv, B, kv.k_new.stride_t, kv.k_new.stride_h,
                        kv.k_new.stride_b, 64, kRows) ||
        !make_tmap_bf16(&tv, &cv, kv.v_new.ptr, D, kv.new_extent, Hkv, B, kv.v_new.stride_t, kv.v_new.stride_h,
                        kv.v_new.stride_b, 64, kRows))
        return L4L_ERR_CUDA;
    if (ck.pos_t != cv.pos_t || ck.pos_h != cv.pos_h || ck.pos_b != cv.pos_b) return L4L_ERR_UNSUPPORTED;
    TcParams p = {};
    // the tokens cached before: tiles of the cache (one box per tile), or of the page pool (one box per page if the
    // pages are smaller than a tile); without a past the kernel never touches these two maps
    tkc = tk; tvc = tv; ckc = ck;
    p.cache_box_t = kRows;
    if (kv.past) {
        const l4l_kv_cache &c = *kv.past;
        const int outer = kv.paged ? kv.paged->num_pages : B;
        if (kv.paged && c.max_len < kRows) p.cache_box_t = c.max_len;
        if (!make_tmap_bf16(&tkc, &ckc, c.k, D, c.max_len, Hkv, outer, c.stride_t, c.stride_h, c.stride_b, 64, p.cache_box_t) ||
            !make_tmap_bf16(&tvc, &cvc, c.v, D, c.max_len, Hkv, outer, c.stride_t, c.stride_h, c.stride_b, 64, p.cache_box_t))
            return L4L_ERR_CUDA;
    }
    p.o = static_cast<__nv_bfloat16 *>(o.ptr);
    p.o_sb = o.stride_b; p.o_st = o.stride_t; p.o_sh = o.stride_h;
    if (kv.write) {
        p.k_new = static_cast<const __nv_bfloat16 *>(kv.k_new.ptr);
        p.v_new = static_cast<const __nv_bfloat16 *>(kv.v_new.ptr);
        p.k_sb = kv.k_new.stride_b; p.k_st = kv.k_new.stride_t; p.k_sh = kv.k_new.stride_h;
        p.v_sb = kv.v_new.stride_b; p.v_st = kv.v_new.stride_t; p.v_sh = kv.v_new.stride_h;
        p.cache_k = static_cast<__nv_bfloat16 *>(kv.write->k);
        p.cache_v = static_cast<__nv_bfloat16 *>(kv.write->v);
        p.c_sb = kv.write->stride_b; p.c_sh = kv.write->stride_h; p.c_st = kv.write->stride_t;
        const long long slots = kv.paged ? (long long)kv.paged->table_stride * kv.write->max_len : kv.write->max_len;
        p.cache_slots = slots > 0x7fffffffll ? 0x7fffffff : (int)slots;
        // whole tiles of a contiguous cache leave by TMA (a cache whose strides no map can describe is written by the warps)
        const l4l_kv_cache &c = *kv.write;
        p.cache_tma = !kv.paged && (kv.past || (make_tmap_bf16(&tkc, &ckc, c.k, D, c.max_len, Hkv, B, c.stride_t, c.stride_h, c.stride_b, 64, kRows) &&
                                                make_tmap_bf16(&tvc, &cvc, c.v, D, c.max_len, Hkv, B, c.stride_t, c.stride_h, c.stride_b, 64, kRows)));
    }
    if (kv.paged) {
        const int page_size = kv.past ? kv.past->max_len : kv.write->max_len;
        p.block_table = kv.paged->block_table;
        p.table_stride = kv.paged->table_stride;
        p.num_pages = kv.paged->num_pages;
        p.page_size = page_size;
        while ((1 << p.page_shift) < page_size) ++p.page_shift;
    }
    p.new_at_past = kv.new_at_past ? 1 : 0;
    p.seq_lens = d_seq_lens;
    p.past_lens = d_past_lens;
    p.lse = d_lse;
    p.status = static_cast<unsigned *>(workspace);
    p.S_max = S_max; p.B = B; p.Hq = Hq; p.Hkv = Hkv; p.G = Hq / Hkv;
    p.pair_heads = pairs_heads(p.G) ? 1 : 0;
    p.n_qblocks = row_blocks(S_max, p.G);
    p.scale_log2e = scale * 1.4426950408889634f;
    p.claims = (long long)p.n_qblocks * (p.pair_heads ? Hq / 2 : Hq) * B > sm_count();
    p.cq = cq; p.ckv = ck; p.co = co; p.ckc = ckc;
    const long long slots = !kv.past ? 0 : kv.paged ? (long long)kv.paged->table_stride * kv.past->max_len : kv.past->max_len;
    const bool ranked = d_past_lens && row_blocks_by_work(S_max, slots, B, Hq, p.G);
    if (ranked)
        return D == 128 ? launch_t<128, true>(tq, tk, tv, to, tkc, tvc, p, stream) : launch_t<64, true>(tq, tk, tv, to, tkc, tvc, p, stream);
    return D == 128 ? launch_t<128, false>(tq, tk, tv, to, tkc, tvc, p, stream) : launch_t<64, false>(tq, tk, tv, to, tkc, tvc, p, stream);
}

int prefill_row_block_order(const int32_t *d_past_lens, const int32_t *d_q_lens, int S_max, long long slots, int B, int Hq, int Hkv,
                            int32_t *d_order, cudaStream_t stream)
{
    const int G = Hq / Hkv;
    if (!row_blocks_by_work(S_max, slots, B, Hq, G)) return 0;
    const int n = row_blocks(S_max, G) * B;
    if (d_order) {
        row_block_order_kernel<<<n, 32, 0, stream>>>(d_past_lens, d_q_lens, S_max, B, row_blocks(S_max, G), pairs_heads(G),
                                                     reinterpret_cast<int2 *>(d_order));
        if (cudaGetLastError() != cudaSuccess) return -1;
    }
    return n;
}

}  // namespace l4l
