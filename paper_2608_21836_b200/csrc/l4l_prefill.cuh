// What the two forms of the causal prefill on the 5th-generation tensor cores share: a block per item (l4l_prefill_blocks.cu) and
// CTAs that take item after item (l4l_prefill_tc.cu, which describes the algorithm and the roles of the warps).
#pragma once
#include "l4l_internal.h"
#include "l4l_ptx.cuh"

namespace l4l {

constexpr int kRows = 128;                     // rows per sub-tile == tokens per K/V tile
constexpr int kThreads = 384;                  // 3 warpgroups: softmax 0, softmax 1, {producer, MMA, 2 that move rows to the cache and out}
constexpr uint32_t kHalfBytes = kRows * 128;   // [128 rows][64 bf16], 128-byte swizzled
constexpr float kRescaleThreshold = 8.f;       // log2 domain: O is rescaled only if the max grew by > 2^8

template <int D>
struct TcCfg {
    static constexpr int kHalves = D / 64;
    static constexpr uint32_t kTileBytes = kHalves * kHalfBytes;        // one Q sub-tile, K tile or V tile
    static constexpr int kSlots = (D == 128) ? 5 : 8;                    // ring of K/V tiles
    static constexpr uint32_t kTmemCols = 512;
    static constexpr uint32_t kColS0 = 0, kColS1 = 128, kColO0 = 256, kColO1 = 256 + D;
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

// The descriptors of a launch.
struct PrefillMaps {
    CUtensorMap q, k, v, o, kc, vc;
};

// Asks for K (idx even) or V (odd) of key tile j = idx / 2 into a slot of the ring.
template <int D>
__device__ __forceinline__ void load_kv_tile(const TcParams &p, const CUtensorMap &tmap_k, const CUtensorMap &tmap_v, const CUtensorMap &tmap_kc,
                                             const CUtensorMap &tmap_vc, int b, int kvh, int past, int n_cache, int idx, uint8_t *dst, uint64_t *bar)
{
    const int j = idx >> 1;
    int c1, c2, c3;
    if (j >= n_cache) {
        // a tile of the new tokens
        order_coords(p.ckv, (p.new_at_past ? past : 0) + (j - n_cache) * kRows, kvh, b, c1, c2, c3);
        const CUtensorMap *tm = (idx & 1) ? &tmap_v : &tmap_k;
#pragma unroll
        for (int hf = 0; hf < TcCfg<D>::kHalves; ++hf) tma_load_4d(dst + hf * kHalfBytes, tm, bar, hf * 64, c1, c2, c3);
    } else if (p.block_table == nullptr) {
        // a tile of the tokens cached before, contiguous cache
        order_coords(p.ckc, j * kRows, kvh, b, c1, c2, c3);
        const CUtensorMap *tm = (idx & 1) ? &tmap_vc : &tmap_kc;
#pragma unroll
        for (int hf = 0; hf < TcCfg<D>::kHalves; ++hf) tma_load_4d(dst + hf * kHalfBytes, tm, bar, hf * 64, c1, c2, c3);
    } else {
        // ... paged cache: one box per page that the tile touches (a page never straddles tiles or boxes), four look-ups at a
        // time. A table entry outside the pool becomes an out-of-range coordinate, which reads zeros.
        const CUtensorMap *tm = (idx & 1) ? &tmap_vc : &tmap_kc;
        const int32_t *row = p.block_table + (size_t)b * p.table_stride;
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
                order_coords(p.ckc, (j * kRows + r0) & (p.page_size - 1), kvh, page[u] < 0 || page[u] >= p.num_pages ? p.num_pages : page[u], c1, c2, c3);
#pragma unroll
                for (int hf = 0; hf < TcCfg<D>::kHalves; ++hf)
                    tma_load_4d(dst + hf * kHalfBytes + r0 * 128, tm, bar, hf * 64, c1, c2, c3);
            }
        }
    }
}

// S_i = Q_i K_j^T, both operands in shared memory; O_i += P_i V_j, P in tensor memory over S_i.
template <int D>
__device__ __forceinline__ void issue_qk(uint32_t tmem_s, uint32_t q_addr, uint32_t k_addr)
{
#pragma unroll
    for (int k = 0; k < D / 16; ++k) {
        const uint32_t off = (k >> 2) * kHalfBytes + (k & 3) * 32;
        tcgen05_mma_ss(tmem_s, make_smem_desc(q_addr + off, 0), make_smem_desc(k_addr + off, 0), make_idesc(kRows, false), k > 0 ? 1u : 0u);
    }
}

template <int D>
__device__ __forceinline__ void issue_pv(uint32_t tmem_o, uint32_t tmem_s, uint32_t v_addr, bool first)
{
#pragma unroll
    for (int k = 0; k < kRows / 16; ++k)
        tcgen05_mma_ts(tmem_o, tmem_s + k * 8, make_smem_desc(v_addr + k * 2048, kHalfBytes), make_idesc(D, true), (first && k == 0) ? 0u : 1u);
}

// V rows from first_dead on hold no valid token (the partly filled last tile of the past, or of the new tokens) and may hold any
// bits, NaN included: cleared, so that a zero weight times garbage cannot appear. A whole warp calls this.
template <int D>
__device__ __forceinline__ void clear_dead_rows(uint8_t *vt, int first_dead, int lane)
{
    if (first_dead >= kRows) return;
    constexpr int kChunks = D / 8;
    for (int i = lane; i < (kRows - first_dead) * kChunks; i += 32) {
        const int r = first_dead + i / kChunks, ch = i % kChunks;
        *reinterpret_cast<uint4 *>(vt + (ch >> 3) * kHalfBytes + r * 128 + ((ch & 7) << 4)) = make_uint4(0u, 0u, 0u, 0u);
    }
    fence_proxy_async_smem();
    __syncwarp();
}

// One key tile of one query row (a thread): scores from tensor memory, running maximum m and sum l, weights P back over S, O rescaled
// where the maximum grew. masked: columns past limit() hold no visible key. A whole warp calls this; P is complete behind it.
template <int D, class Limit>
__device__ __forceinline__ void softmax_tile(uint32_t tmem_s, uint32_t tmem_o, float c, bool first, bool masked, Limit limit, float &m, float &l)
{
    uint32_t sr[4][32];
#pragma unroll
    for (int qd = 0; qd < 4; ++qd) tmem_ld_32x32b_x32(tmem_s + qd * 32, sr[qd]);
    tcgen05_wait_ld();

    // Row maximum of the scaled scores (log2 domain). Off the diagonal the maximum is taken over the
    // raw scores with independent 3-input max chains and scaled once (min for a negative scale);
    // on the diagonal tile the causal mask is applied to the scaled scores first.
    float mx;
    if (masked) {
        const int lim = limit();                               // columns > lim hold no visible key
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
    const bool grow = (mx > m + kRescaleThreshold) || first;
    float alpha = 1.f;
    if (grow) {
        const float m_new = (mx == -INFINITY) ? 0.f : mx;
        alpha = fast_exp2(m - m_new);                      // first: exp2(-inf) = 0
        m = m_new;
        l *= alpha;
    }
    if (!first && __any_sync(0xffffffffu, grow)) {
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
    const float fc = masked ? 1.f : c;                       // diagonal scores are already scaled
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
}

// A row of O, times inv, as bf16: into its place in the staged sub-tile (whole: one TMA store per 64 columns takes it from there) or, if valid,
// to its place in the output.
template <int D>
__device__ __forceinline__ void put_row(uint32_t tmem_o, float inv, bool whole, uint8_t *stage, int t, bool valid, __nv_bfloat16 *orow)
{
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
}

inline bool pairs_heads(int G) { return G % 2 == 0; }
inline int row_blocks(int S_max, int G) { return pairs_heads(G) ? (S_max + kRows - 1) / kRows : (S_max + 2 * kRows - 1) / (2 * kRows); }

// A launch of either kernel.
template <auto kKernel, size_t kSmemBytes>
l4l_status launch_prefill_kernel(const PrefillMaps &m, const TcParams &p, cudaStream_t stream)
{
    static bool configured_on[kDeviceSlots] = {};
    const int slot = device_slot();
    if (slot < 0) return L4L_ERR_CUDA;
    {
        std::lock_guard<std::mutex> lock(setup_mutex());
        bool &configured = configured_on[slot];
        if (!configured) {
            if (cudaFuncSetAttribute(kKernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes) != cudaSuccess) return L4L_ERR_CUDA;
            configured = true;
        }
    }
    const long long grid = (long long)p.n_qblocks * (p.pair_heads ? p.Hq / 2 : p.Hq) * p.B;
    if (grid > 0x7fffffffll) return L4L_ERR_UNSUPPORTED;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kKernel, m.q, m.k, m.v, m.o, m.kc, m.vc, p) == cudaSuccess ? L4L_OK : L4L_ERR_CUDA;
}

// The launch with a block per item.
l4l_status launch_prefill_blocks(const PrefillMaps &m, const TcParams &p, int D, bool ranked, cudaStream_t stream);

}  // namespace l4l
