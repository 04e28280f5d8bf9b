// Causal prefill on the 5th-generation tensor cores (tcgen05.mma, accumulators in tensor memory).
// A block per item, for launches of short sequences or of at most one block per SM; the longer ones go to l4l_prefill_tc.cu, whose CTAs
// take item after item. Here three warps copy a ragged or paged diagonal tile into the cache and nothing waits for them, there one warp
// per tensor does: 1 x 100 tokens (32/8 x 128) 9.1 us here, 13.3 there; 4 x 50..200 10.7 and 17.0; 16 x 50..100 18.1 and 25.3;
// 8 x 100..700 (64/8) 92.5 and 75.0; 3 x 300..1000 (40/8) 40.8 and 36.0.
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
//   warp  8     TMA producer: Q once, then K_j, V_j tiles (128 tokens, 128-byte swizzle) through a
//               ring of shared-memory slots; afterwards copies the block's diagonal K/V tiles from
//               shared memory into the KV cache (only for the first query head of a KV group)
//   warp  9     MMA issuer (one lane): S_i = Q_i K_j^T from shared memory, O_i += P_i V_j with P read
//               from TMEM and V as an MN-major shared-memory operand; owns the TMEM allocation
//   warps 10-11 help with the cache copy, which runs beside the last iterations
//
// The same kernel serves a chunk of new tokens over a populated cache. The key axis of a sequence is then two runs
// of 128-token tiles: the `past` tokens cached before (tiles of the cache, contiguous or paged, aligned to slot 0;
// every query row sees all of them, the last tile may be partly filled) followed by the new tokens (tiles aligned
// to the chunk's first token, so the causal diagonal sits exactly as in a fresh prompt, which is the case past = 0).
// The new tokens' K/V come from the caller's tensors (and are written to the cache in the same pass) or, when the
// caller has appended them already, from the cache itself at slot past + row.
// A whole sub-tile's output leaves through the shared memory that held its Q rows and TMA stores.
//
// TMEM columns: S0 [0,128) S1 [128,256) O0 [256,256+D) O1 [256+D,256+2D); P_i aliases the first 64
// columns of S_i. Causal tile skipping: sub-tile i only visits K/V tiles up to its diagonal.
// The tensor pipe executes one thread's MMAs in issue order, which is what makes the S/P aliasing
// safe: QK_{j+1} into S_i is issued after PV_j that reads P_i.
#include "l4l_prefill.cuh"

namespace l4l {

namespace {

template <int D>
struct BlocksCfg : TcCfg<D> {
    using TcCfg<D>::kSlots, TcCfg<D>::kTileBytes;
    static constexpr int kNumBars = 1 + 2 * kSlots + 8;
    static constexpr size_t kSmemBytes = 1024 + 2 * kTileBytes + (size_t)kSlots * kTileBytes + kNumBars * 8 + 64;
};

// kRanked: row blocks in the order of their work, not of their place in the sequence (an instantiation of its own: fresh
// prompts do not pay for it)
template <int D, bool kRanked>
__global__ void __launch_bounds__(kThreads, 1)
prefill_blocks_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                  const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_o,
                  const __grid_constant__ CUtensorMap tmap_kc, const __grid_constant__ CUtensorMap tmap_vc,
                  const TcParams p)
{
    using C = BlocksCfg<D>;
    // ---- which block: heaviest (longest causal span) blocks first, heads of a KV group adjacent
    grid_dependency_wait();                       // seq_lens may have been written by the previous kernel
    // pair mode: sub-tile i is query head h + i at rows q0 ..; else: head h at rows q0 + 128 i ..
    const bool pair = p.pair_heads != 0;
    const int heads = pair ? p.Hq / 2 : p.Hq;
    const int per_block = heads * p.B;
    int qb = p.n_qblocks - 1 - (int)(blockIdx.x / per_block);           // block of 128 (pair mode) or 256 rows
    const int hb = blockIdx.x % per_block;
    const int h = pair ? 2 * (hb % heads) : hb % heads;
    int b = hb / heads;
    const int kvh = h / p.G;
    const int sub_rows = pair ? 0 : kRows;                // rows between the two sub-tiles
    const int sub_heads = pair ? 1 : 0;                   // heads between them
    // The two lengths are requested now and first looked at after the barrier / TMEM set-up below, so that
    // their latency is hidden behind it.
    int L_raw = __ldg(p.seq_lens + b);
    int past_raw = p.past_lens ? __ldg(p.past_lens + b) : 0;
    // Ranked row blocks: the lengths of all sequences (at most 32), requested with them.
    int len_of = 0, past_of = 0;
    if (kRanked && (int)(threadIdx.x & 31) < p.B) {
        len_of = __ldg(p.seq_lens + (threadIdx.x & 31));
        past_of = __ldg(p.past_lens + (threadIdx.x & 31));
    }

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    uint8_t *q_smem = smem;                                       // 2 sub-tiles
    uint8_t *ring = smem + 2 * C::kTileBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(ring + (size_t)C::kSlots * C::kTileBytes);
    uint64_t *q_full = bars;
    uint64_t *kv_full = bars + 1;
    uint64_t *kv_empty = kv_full + C::kSlots;
    uint64_t *s_full = kv_empty + C::kSlots;      // [2]
    uint64_t *p_full = s_full + 2;                // [2]
    uint64_t *o_full = p_full + 2;                // [2]
    uint64_t *o_staged = o_full + 2;              // [2] a sub-tile's output rows are in shared memory
    uint32_t *tmem_base_smem = reinterpret_cast<uint32_t *>(o_staged + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_base_smem + 1);
    volatile int *copy_go = abort_flag + 1;       // producer -> helper warps: all loads issued

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // The producer's lane sets the barriers up itself, so that it can start the first loads right away, while
    // the other warps are still on their way to the block-wide barrier below (TMEM allocation included).
    const bool producer_lane = threadIdx.x == 8 * 32;
    if (producer_lane) {
        mbar_init(q_full, 1);
        for (int s = 0; s < C::kSlots; ++s) {
            mbar_init(&kv_full[s], 1);
            mbar_init(&kv_empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&s_full[i], 1);
            mbar_init(&p_full[i], kRows);
            mbar_init(&o_full[i], 1);
            mbar_init(&o_staged[i], kRows);
        }
        *abort_flag = 0;
        *copy_go = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
    }
    // Ranked row blocks. With equal pasts (every fresh prompt) the order of places is the order of work, and this vote is all that
    // the block pays for.
    if (kRanked && __builtin_expect(!__all_sync(0xffffffffu, lane >= p.B || past_of == past_raw), 0)) {
        if (!row_block_by_work(len_of, past_of, p.S_max, pair ? 7 : 8, pair ? 0 : 1, (int)(blockIdx.x / heads), b, qb)) return;
        L_raw = __shfl_sync(0xffffffffu, len_of, b);
        past_raw = __shfl_sync(0xffffffffu, past_of, b);
        b = __shfl_sync(0xffffffffu, b, 0);                  // the same in every lane: in registers of the warp
        qb = __shfl_sync(0xffffffffu, qb, 0);
    }
    const int q0 = qb * (pair ? kRows : 2 * kRows);
    const int diag0 = pair ? qb : 2 * qb;                 // tile (among the new tokens) of sub-tile 0's diagonal
    // first use of the lengths. A block past the end of its sequence has nothing to do (decided before any
    // TMEM is taken).
    const int L = L_raw < 0 ? 0 : (L_raw > p.S_max ? p.S_max : L_raw);
    if (q0 >= L) return;
    // Tokens already in the cache ahead of these (0 for a fresh prompt): n_cache tiles, seen by every row.
    const int past = past_raw < 0 ? 0 : past_raw;
    const int n_cache = (past + kRows - 1) / kRows;
    // sub-tile i (rows q0 + 128 i ..) visits the tiles of the past and the new tokens' tiles up to its diagonal
    int n_sub[2];
    n_sub[0] = n_cache + min(q0 + kRows - 1, L - 1) / kRows + 1;
    n_sub[1] = (q0 + sub_rows < L) ? n_cache + min(q0 + sub_rows + kRows - 1, L - 1) / kRows + 1 : 0;
    const int n_kv = max(n_sub[0], n_sub[1]);
    // Q and the first ring-ful of K/V tiles need no waiting: requested before the block-wide barrier
    const int n_pre = min(2 * n_kv, C::kSlots);
    auto request_tile = [&](int idx) {
        const uint32_t s = idx % C::kSlots;
        mbar_arrive_expect_tx(&kv_full[s], C::kTileBytes);
        load_kv_tile<D>(p, tmap_k, tmap_v, tmap_kc, tmap_vc, b, kvh, past, n_cache, idx, ring + (size_t)s * C::kTileBytes, &kv_full[s]);
    };
    if (producer_lane) {
        tma_prefetch_desc(&tmap_q);
        tma_prefetch_desc(&tmap_k);
        tma_prefetch_desc(&tmap_v);
        if (n_cache > 0) {
            tma_prefetch_desc(&tmap_kc);
            tma_prefetch_desc(&tmap_vc);
        }
        int c1, c2, c3;
        mbar_arrive_expect_tx(q_full, 2 * C::kTileBytes);
        order_coords(p.cq, q0, h, b, c1, c2, c3);
#pragma unroll
        for (int hf = 0; hf < C::kHalves; ++hf) tma_load_4d(q_smem + hf * kHalfBytes, &tmap_q, q_full, hf * 64, c1, c2, c3);
        request_tile(0);                                   // K_0 right behind Q_0: the first product needs both
        order_coords(p.cq, q0 + sub_rows, h + sub_heads, b, c1, c2, c3);
#pragma unroll
        for (int hf = 0; hf < C::kHalves; ++hf)
            tma_load_4d(q_smem + C::kTileBytes + hf * kHalfBytes, &tmap_q, q_full, hf * 64, c1, c2, c3);
        for (int idx = 1; idx < n_pre; ++idx) request_tile(idx);
    }
    if (warp == 9) {
        tmem_alloc(tmem_base_smem, C::kTmemCols);
        tmem_relinquish_alloc_permit();
    }
    // Programmatic dependent launch: the next kernel of the stream may start its own prologue now.
    grid_launch_dependents();
    tcgen05_fence_before_sync();
    __syncthreads();
    tcgen05_fence_after_sync();
    const uint32_t tmem_base = *tmem_base_smem;

    // The block's diagonal K/V tiles (one or two tiles of the new tokens, from diag0 on) go to the cache, at slot past + row
    // (first query head of a KV group only, so each row is written once). They are the last tiles loaded, so their
    // ring slots are never refilled; the copy runs beside the last iterations, shared by three warps. Rows >= L
    // and slots the cache does not have are not written.
    const bool writes_cache = p.cache_k != nullptr && (h % p.G) == 0;
    auto copy_diagonal_tiles = [&](int part) {
        if (!writes_cache) return;
        for (int j = n_cache + diag0; j < n_kv; ++j) {
            const int r_base = (j - n_cache) * kRows;              // first row of the tile among the new tokens
            for (int kv = 0; kv < 2; ++kv) {
                const int idx = 2 * j + kv;
                const uint32_t s = idx % C::kSlots, ph = (idx / C::kSlots) & 1u;
                if (!mbar_wait(&kv_full[s], ph, abort_flag)) return;
                const uint8_t *src = ring + (size_t)s * C::kTileBytes;
                __nv_bfloat16 *dst_all = kv ? p.cache_v : p.cache_k;
                constexpr int kChunks = D / 8;
                const int rows = min(min(kRows, L - r_base), p.cache_slots - past - r_base);
                for (int i = part * 32 + lane; i < rows * kChunks; i += 96) {
                    const int r = i / kChunks, ch = i % kChunks;
                    const int slot = past + r_base + r;
                    __nv_bfloat16 *dst;
                    if (p.block_table == nullptr) {
                        dst = dst_all + b * p.c_sb + kvh * p.c_sh + (int64_t)slot * p.c_st;
                    } else {
                        const int page = __ldg(p.block_table + (size_t)b * p.table_stride + (slot >> p.page_shift));
                        if (page < 0 || page >= p.num_pages) continue;          // no page behind this slot
                        dst = dst_all + (int64_t)page * p.c_sb + kvh * p.c_sh + (int64_t)(slot & (p.page_size - 1)) * p.c_st;
                    }
                    const uint4 val = *reinterpret_cast<const uint4 *>(src + (ch >> 3) * kHalfBytes + swz128(r, ch & 7));
                    *reinterpret_cast<uint4 *>(dst + ch * 8) = val;
                }
            }
        }
    };

    // Register reallocation: the data-movement warpgroup gives registers to the softmax warpgroups,
    // whose threads hold a whole 128-column score row.
    if (warp >= 8) {
    setmaxnreg_dec<64>();
    if (warp == 8) {
        // ============================================================ TMA producer (+ cache copy)
        if (lane == 0) {
            for (int idx = n_pre; idx < 2 * n_kv; ++idx) {
                const uint32_t s = idx % C::kSlots, ph = (idx / C::kSlots) & 1u;
                if (!mbar_wait(&kv_empty[s], ph ^ 1u, abort_flag)) break;
                request_tile(idx);
            }
        }
        // all loads are issued: the diagonal tiles' slots are in their last phase, the copy may start
        if (lane == 0) {
            __threadfence_block();
            *copy_go = 1;
        }
        __syncwarp();
        copy_diagonal_tiles(0);
    } else if (warp == 10 || warp == 11) {
        // otherwise idle warps. First: if an earlier CTA of this launch already reported a dead wait, do
        // not repeat its time-out in every remaining CTA. Then: help the producer warp copy the diagonal
        // tiles to the cache.
        if (warp == 10 && lane == 0 && *reinterpret_cast<volatile unsigned *>(p.status + kStatusErrWord) != 0u)
            *abort_flag = 1;
        if (writes_cache) {
            const long long t0 = clock64();
            bool go = true;
            while (*copy_go == 0) {
                if (*abort_flag || clock64() - t0 > kWaitCycleBudget) { go = false; break; }
                __nanosleep(128);
            }
            __threadfence_block();
            if (go) copy_diagonal_tiles(warp - 9);
        }
    } else if (warp == 9) {
        // ============================================================ MMA issuer
        const uint32_t tmem_s[2] = {tmem_base + C::kColS0, tmem_base + C::kColS1};
        const uint32_t tmem_o[2] = {tmem_base + C::kColO0, tmem_base + C::kColO1};
        const uint32_t q_addr = smem_u32(q_smem), ring_addr = smem_u32(ring);

        bool ok = mbar_wait(q_full, 0, abort_flag) && mbar_wait(&kv_full[0], 0, abort_flag);
        if (ok) {
            tcgen05_fence_after_sync();
            if (lane == 0) {
                for (int i = 0; i < 2; ++i)
                    if (n_sub[i] > 0) {
                        issue_qk<D>(tmem_s[i], q_addr + i * C::kTileBytes, ring_addr);
                        tcgen05_commit(&s_full[i]);
                    }
                tcgen05_commit(&kv_empty[0]);
            }
            __syncwarp();
        }
        for (int j = 0; ok && j < n_kv; ++j) {
            const int iv = 2 * j + 1, ik = 2 * j + 2;
            const uint32_t sv = iv % C::kSlots, sk = ik % C::kSlots;
            if (!mbar_wait(&kv_full[sv], (iv / C::kSlots) & 1u, abort_flag)) { ok = false; break; }
            clear_dead_rows<D>(ring + (size_t)sv * C::kTileBytes, j < n_cache ? past - j * kRows : L - (j - n_cache) * kRows, lane);
            const bool have_next = j + 1 < n_kv;
            if (have_next && !mbar_wait(&kv_full[sk], (ik / C::kSlots) & 1u, abort_flag)) { ok = false; break; }
            for (int i = 0; i < 2 && ok; ++i) {
                if (j >= n_sub[i]) continue;
                if (!mbar_wait(&p_full[i], j & 1u, abort_flag)) { ok = false; break; }
                tcgen05_fence_after_sync();
                if (lane == 0) {
                    issue_pv<D>(tmem_o[i], tmem_s[i], ring_addr + sv * C::kTileBytes, j == 0);
                    if (j + 1 < n_sub[i]) {
                        issue_qk<D>(tmem_s[i], q_addr + i * C::kTileBytes, ring_addr + sk * C::kTileBytes);
                        tcgen05_commit(&s_full[i]);
                    } else {
                        tcgen05_commit(&o_full[i]);
                    }
                }
                __syncwarp();
            }
            if (ok && lane == 0) {
                tcgen05_commit(&kv_empty[sv]);
                if (have_next) tcgen05_commit(&kv_empty[sk]);
            }
            __syncwarp();
        }
    }
    } else {
        setmaxnreg_inc<216>();
        // ============================================================ softmax + epilogue warpgroups
        const int i = warp >> 2;                                   // sub-tile
        const int t = threadIdx.x & 127;                           // row within the sub-tile == TMEM lane
        const int row = q0 + i * sub_rows + t;                     // token index of this thread's query row
        const int hq = h + i * sub_heads;                          // ... and its query head
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tmem_s = tmem_base + lane_base + (i ? C::kColS1 : C::kColS0);
        const uint32_t tmem_o = tmem_base + lane_base + (i ? C::kColO1 : C::kColO0);
        const int n_mine = n_sub[i];
        // Tiles that need a mask: the last tile of the past when it is partly filled (columns past its end, the same
        // for every row), and the sub-tile's diagonal tile among the new tokens (row t sees columns 0..t).
        const int j_ragged = (past & (kRows - 1)) ? n_cache - 1 : -1;
        const int j_diag = n_cache + (pair ? diag0 : diag0 + i);
        const float c = p.scale_log2e;
        float m = -INFINITY, l = 0.f;
        bool ok = true;

        for (int j = 0; j < n_mine; ++j) {
            if (!mbar_wait(&s_full[i], j & 1u, abort_flag)) { ok = false; break; }
            tcgen05_fence_after_sync();
            softmax_tile<D>(tmem_s, tmem_o, c, j == 0, j == j_ragged || j >= j_diag, [&] { return j == j_ragged ? (past & (kRows - 1)) - 1 : t; }, m, l);
            mbar_arrive(&p_full[i]);
        }

        if (ok && n_mine > 0 && mbar_wait(&o_full[i], 0, abort_flag)) {
            tcgen05_fence_after_sync();
            const float inv = 1.f / l;
            const bool valid = row < L;
            __nv_bfloat16 *orow = p.o + b * p.o_sb + (int64_t)row * p.o_st + hq * p.o_sh;
            // A sub-tile whose 128 rows are all valid leaves through shared memory and one TMA store per 64
            // columns (coalesced, asynchronous): the rows are staged where Q_i was, which no MMA reads any more
            // (o_full follows the last of them). A ragged sub-tile writes its valid rows directly.
            const bool whole = q0 + i * sub_rows + kRows <= L;
            uint8_t *stage = q_smem + i * C::kTileBytes;
            put_row<D>(tmem_o, inv, whole, stage, t, valid, orow);
            if (whole) {
                mbar_arrive(&o_staged[i]);
                if (t == 0 && mbar_wait(&o_staged[i], 0, abort_flag)) {
                    int c1, c2, c3;
                    order_coords(p.co, q0 + i * sub_rows, hq, b, c1, c2, c3);
#pragma unroll
                    for (int hf = 0; hf < C::kHalves; ++hf) tma_store_4d(&tmap_o, stage + hf * kHalfBytes, hf * 64, c1, c2, c3);
                    tma_store_commit();
                    tma_store_wait_read_all();                     // shared memory must outlive the reads
                }
            }
            if (valid && p.lse)
                p.lse[((size_t)b * p.Hq + hq) * p.S_max + row] = (m + log2f(l)) * 0.6931471805599453f;
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

template <int D>
l4l_status launch_blocks(const PrefillMaps &m, const TcParams &p, bool ranked, cudaStream_t stream)
{
    constexpr size_t smem = BlocksCfg<D>::kSmemBytes;
    return ranked ? launch_prefill_kernel<prefill_blocks_kernel<D, true>, smem>(m, p, stream)
                  : launch_prefill_kernel<prefill_blocks_kernel<D, false>, smem>(m, p, stream);
}

}  // namespace

l4l_status launch_prefill_blocks(const PrefillMaps &m, const TcParams &p, int D, bool ranked, cudaStream_t stream)
{
    return D == 128 ? launch_blocks<128>(m, p, ranked, stream) : launch_blocks<64>(m, p, ranked, stream);
}

}  // namespace l4l
