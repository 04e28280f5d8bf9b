// Warp-level building blocks of the decode kernels on the legacy tensor path (mma.sync m16n8k16, 16-bit inputs -> fp32):
// one warp holds the query heads of one KV group and consumes 16 tokens of K and V at a time from a shared-memory tile
// with the 128-byte swizzle. (Prefill runs on tcgen05 instead: see l4l_prefill_tc.cu.)
//
// The products are taken transposed: S^T = K Q^T with the TOKENS as the M = 16 rows and the group's query heads as the
// N = 8 columns, then O^T = V^T P^T with the head dims as rows. A group of 4 heads fills half of the 8 columns, where as
// rows it would fill a quarter of 16: half the MMAs, half the exponentials, and the output accumulators of a 128-wide
// head are 32 registers instead of 64 (NB = 2 blocks of 8 heads, for groups of 9 to 16, are as before). P^T is the B operand of
// the second product: an 8 x 8 transpose of the score fragment (movmatrix). Measured, us, heads as rows -> as columns: e4m3
// cache, B = 32 ragged 37.0 -> 31.7; B = 512 x 64..256 tokens 65.1 -> 62.4; bf16 caches of large batches are bound by HBM, 46.2
// either way. Every sum has the order that it has with the heads as rows, so that the results are the same bit for bit: one
// accumulator per score, and denominators summed from the transposed weights. (Two accumulators for even and odd k-steps and
// sums ahead of the transpose would save one sequence of 2304 tokens 8.58 against 8.70 us, 512 short ones 62.2 against 62.4.)
//
// Tile layout in shared memory: D/64 "halves", each [tile_tokens][64] bf16 (128-byte rows,
// swizzled), half h covering head_dim [64h, 64h+64). Over pages of 16 or 32 tokens at head_dim 128 one load brings
// both halves of a page, and the tile is a row of pages, each [half][page tokens][64] (TileRows).
#pragma once

#include "l4l_ptx.cuh"

namespace l4l {

// Where the token rows of a tile lie: `half_bytes` between the halves, and `group` (the negative of the tokens per page;
// 0: one group) for tiles made of pages that hold both halves each. A 16-token block never straddles groups.
struct TileRows {
    uint32_t half_bytes, group;
    // offset of a token's row in half 0, without the swizzle of its chunks
    __device__ __forceinline__ uint32_t row(uint32_t token) const { return (token + (token & group)) * 128u; }
    // 16-byte chunk `ch` of a token's row (bf16: 16 chunks at head_dim 128)
    __device__ __forceinline__ uint32_t chunk(uint32_t token, uint32_t ch) const
    {
        return (ch >> 3) * half_bytes + row(token) + (((ch ^ token) & 7u) << 4);
    }
};

// Fragment positions of a lane: r = lane / 4, c = lane % 4. Heads of block n: column 2c, 2c + 1 -> heads 8n + 2c + {0, 1}.
template <int D, int NB>
struct WarpAttnState {
    float m[NB][2];          // running maximum (log2 domain) of this lane's two heads of each block
    float l[NB];             // this lane's share of the running sum of head 8n + r (tokens 2c, 2c + 1 of every 8)
    float o[D / 16][NB][4];  // O^T, unnormalised: 16 head dims per tile; [e] dim row r, [2 + e] dim row r + 8 of head 2c + e

    __device__ __forceinline__ void reset()
    {
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            m[n][0] = m[n][1] = -INFINITY;
            l[n] = 0.f;
#pragma unroll
            for (int i = 0; i < D / 16; ++i) o[i][n][0] = o[i][n][1] = o[i][n][2] = o[i][n][3] = 0.f;
        }
    }
    // the sums over all tokens (every lane of the warp must call this)
    __device__ __forceinline__ void finish_sums()
    {
#pragma unroll
        for (int n = 0; n < NB; ++n)
#pragma unroll
            for (int off = 1; off <= 2; off <<= 1) l[n] += __shfl_xor_sync(0xffffffffu, l[n], off);
    }
};

__device__ __forceinline__ uint32_t bf16x2_to_f16x2(uint32_t v)
{
    return pack_f16x2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}

// The group's query rows (bf16, [G][D] in shared memory) as B fragments: qf[k-step][block] = head 8n + r, columns
// 16 ks + 2c + {0, 1} and + 8. kF16 (e4m3 caches): as f16, with the k index permuted the way the K bytes arrive (below).
template <int D, int NB, bool kF16>
__device__ __forceinline__ void load_q_fragments(uint32_t (&qf)[D / 16][NB][2], const uint32_t *q_rows, int G)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
        const int head = 8 * n + (lane >> 2);
        const uint32_t *row = q_rows + (size_t)head * (D / 2);
        const bool valid = head < G;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
            const int w = kF16 ? ks * 8 + 2 * (lane & 3) : ks * 8 + (lane & 3);
            const uint32_t a = valid ? row[w] : 0u, b = valid ? row[w + (kF16 ? 1 : 4)] : 0u;
            qf[ks][n][0] = kF16 ? bf16x2_to_f16x2(a) : a;
            qf[ks][n][1] = kF16 ? bf16x2_to_f16x2(b) : b;
        }
    }
}

// S^T (16 tokens x 8 NB heads) = K(tokens row0 .. row0 + 15) . Q^T. s[n]: [e] token row0 + r, [2 + e] token row0 + r + 8 of
// head 8n + 2c + e. One accumulator per score, the k-steps in their order; several blocks of 16 tokens (block u at k_tile[u], rows from
// row0 on) are so many independent chains, issued in turn.
template <int D, int NB, int NT>
__device__ __forceinline__ void warp_qk(const uint32_t (&qf)[D / 16][NB][2], const uint32_t (&k_tile)[NT], uint32_t half_bytes,
                                        float (&s)[NT][NB][4])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < NT; ++u)
#pragma unroll
        for (int n = 0; n < NB; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[u][n][e] = 0.f;
    const uint32_t row = lane & 15;                                 // matrices 1, 3: tokens + 8
    const uint32_t csel = lane >> 4;                                // matrices 2, 3: head dims + 8
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
        const uint32_t chunk = 2 * ks + csel;                       // 16-byte chunk of the full row
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            uint32_t a[4];
            ldmatrix_x4(k_tile[u] + (chunk >> 3) * half_bytes + swz128(row, chunk & 7), a[0], a[1], a[2], a[3]);
#pragma unroll
            for (int n = 0; n < NB; ++n) mma_bf16_16816(s[u][n], a, qf[ks][n][0], qf[ks][n][1]);
        }
    }
}

// O^T += V(tokens row0 .. row0 + 15)^T . P^T
template <int D, int NB>
__device__ __forceinline__ void warp_pv(WarpAttnState<D, NB> &st, const uint32_t (&pb)[NB][2], uint32_t v_tile,
                                        uint32_t half_bytes, int row0)
{
    const int lane = threadIdx.x & 31;
    const uint32_t row = row0 + ((lane >> 4) << 3) + (lane & 7);    // matrices 2, 3: tokens + 8
    const uint32_t csel = (lane >> 3) & 1;                          // matrices 1, 3: head dims + 8
#pragma unroll
    for (int mt = 0; mt < D / 16; ++mt) {
        const uint32_t chunk = 2 * mt + csel;
        uint32_t a[4];
        ldmatrix_x4_trans(v_tile + (chunk >> 3) * half_bytes + swz128(row, chunk & 7), a[0], a[1], a[2], a[3]);
#pragma unroll
        for (int n = 0; n < NB; ++n) mma_bf16_16816(st.o[mt][n], a, pb[n][0], pb[n][1]);
    }
}

// Tokens from `nvalid` on (of the 16 * NT in s) get no weight.
template <int NB, int NT>
__device__ __forceinline__ void warp_mask(float (&s)[NT][NB][4], int nvalid)
{
    const int r = (threadIdx.x & 31) >> 2;
#pragma unroll
    for (int u = 0; u < NT; ++u)
#pragma unroll
        for (int n = 0; n < NB; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (16 * u + r + 8 * (e >> 1) >= nvalid) s[u][n][e] = -INFINITY;
}

// Online-softmax update over NT blocks of 16 tokens. Scores arrive already multiplied by scale*log2(e), masked positions
// at -inf. A step in which no score exceeds the running maxima of its heads (most of them, after the first tiles) needs one
// vote and neither shuffles nor a rescale. (The maxima stay exact: a reference left up to 2^8 behind would save the rest of
// the shuffles, but then the largest weights are rounded too, and the log-sum-exp was off by 2.5e-3 instead of 2e-3.)
// pb[u]: B fragments of P^T, weights as bf16, or as f16 for the MMAs of the e4m3 path. The denominators are summed from them:
// once transposed, a lane's weights are all of one head. kInRow: the four weights of a 16-token block one after the other, else by pairs.
template <int D, int NB, bool kF16, int NT, bool kInRow>
__device__ __forceinline__ void warp_softmax(WarpAttnState<D, NB> &st, const float (&s)[NT][NB][4], uint32_t (&pb)[NT][NB][2])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
        float mx[2], corr_l = 1.f;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            mx[e] = fmaxf(s[0][n][e], s[0][n][2 + e]);
#pragma unroll
            for (int u = 1; u < NT; ++u) mx[e] = fmaxf(mx[e], fmaxf(s[u][n][e], s[u][n][2 + e]));
        }
        if (__any_sync(0xffffffffu, mx[0] > st.m[n][0] || mx[1] > st.m[n][1])) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
                for (int off = 4; off <= 16; off <<= 1) mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], off));
                const float m_new = fmaxf(st.m[n][e], mx[e]);
                const float corr = fast_exp2(st.m[n][e] - ((m_new == -INFINITY) ? 0.f : m_new));
                st.m[n][e] = m_new;
                const float of_row = __shfl_sync(0xffffffffu, corr, lane >> 3);      // lane r / 2 holds heads r - r % 2 + {0, 1}
                if (((lane >> 2) & 1) == e) corr_l = of_row;
#pragma unroll
                for (int mt = 0; mt < D / 16; ++mt) {
                    st.o[mt][n][e] *= corr;
                    st.o[mt][n][2 + e] *= corr;
                }
            }
        }
        const float m0 = (st.m[n][0] == -INFINITY) ? 0.f : st.m[n][0], m1 = (st.m[n][1] == -INFINITY) ? 0.f : st.m[n][1];
        float sum = 0.f;
#pragma unroll
        for (int u = 0; u < NT; ++u)
#pragma unroll
            for (int h = 0; h < 2; ++h) {                           // token rows r and r + 8
                const float e0 = fast_exp2(s[u][n][2 * h] - m0), e1 = fast_exp2(s[u][n][2 * h + 1] - m1);
                const uint32_t pk = movmatrix_trans(kF16 ? pack_f16x2(e0, e1) : pack_bf16x2(e0, e1));
                pb[u][n][h] = pk;
                // the denominator sums exactly the rounded weights that multiply V
                float w0, w1;
                if constexpr (kF16) unpack_f16x2(pk, w0, w1);
                else w0 = __uint_as_float(pk << 16), w1 = __uint_as_float(pk & 0xffff0000u);
                sum = kInRow ? sum + w0 + w1 : sum + (w0 + w1);
            }
        st.l[n] = fmaf(st.l[n], corr_l, sum);
    }
}

// ----------------------------------------------------------------------------- fp8 (e4m3) K/V tiles
// A tile is rows of 128 bytes, 128-byte swizzled: one token per row at D = 128, TWO consecutive tokens per row at
// D = 64 (token 2r in bytes 0..63 of row r, token 2r+1 in bytes 64..127: a dense cache of 64-byte token rows seen as
// rows of 128). tok_chunk_f8 gives the address of 16-byte chunk c (16 head dims) of a token either way. The values are
// widened to f16 in registers (exact) and multiplied with f16 MMAs. ldmatrix moves 16-bit units, so a
// thread receives 4 consecutive head-dim bytes of a K row where the MMA wants two separate pairs: the
// k index of QK^T is therefore permuted (MMA slots 2c, 2c+1, 2c+8, 2c+9 of a 16-block hold head dims
// 4c .. 4c+3), and the q fragments are built with the same permutation. For V the
// transposing ldmatrix delivers, per thread, two tokens of an EVEN and an ODD head dim: rows r of a 16-dim tile of O^T
// are the even dims (2r), rows r + 8 the odd ones (2r + 1).

// Shared-memory address of head dims [16c, 16c+16) of token `tok` of an fp8 tile.
template <int D>
__device__ __forceinline__ uint32_t tok_chunk_f8(uint32_t tile, uint32_t tok, uint32_t c)
{
    static_assert(D == 128 || D == 64, "one or two tokens per 128-byte row");
    if constexpr (D == 128) return tile + swz128(tok, c);
    else return tile + swz128(tok >> 1, ((tok & 1u) << 2) + c);
}

template <int D, int NB, int NT>
__device__ __forceinline__ void warp_qk_f8(const uint32_t (&qf)[D / 16][NB][2], uint32_t k_tile, int row0, float (&s)[NT][NB][4])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < NT; ++u)
#pragma unroll
        for (int n = 0; n < NB; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[u][n][e] = 0.f;
    const uint32_t row = row0 + (lane & 15);                        // matrices 1, 3: tokens + 8
    const uint32_t csel = lane >> 4;                                // matrices 2, 3: next 16 head dims
#pragma unroll
    for (int qd = 0; qd < D / 32; ++qd) {
        uint32_t r[NT][4];
#pragma unroll
        for (int u = 0; u < NT; ++u)
            ldmatrix_x4(tok_chunk_f8<D>(k_tile, row + 16 * u, 2 * qd + csel), r[u][0], r[u][1], r[u][2], r[u][3]);
#pragma unroll
        for (int h = 0; h < 2; ++h)                                 // head dims 32 qd + 16 h ..
#pragma unroll
            for (int u = 0; u < NT; ++u) {
                const uint32_t lo = r[u][2 * h], hi = r[u][2 * h + 1];
                const uint32_t a[4] = {e4m3x2_to_f16x2(lo), e4m3x2_to_f16x2(hi), e4m3x2_to_f16x2(lo >> 16), e4m3x2_to_f16x2(hi >> 16)};
#pragma unroll
                for (int n = 0; n < NB; ++n) mma_f16_16816(s[u][n], a, qf[2 * qd + h][n][0], qf[2 * qd + h][n][1]);
            }
    }
}

template <int D, int NB>
__device__ __forceinline__ void warp_pv_f8(WarpAttnState<D, NB> &st, const uint32_t (&pb)[NB][2], uint32_t v_tile, int row0)
{
    const int lane = threadIdx.x & 31;
    const uint32_t row = row0 + (lane & 15);                        // matrices 1, 3: tokens + 8
    const uint32_t csel = lane >> 4;                                // matrices 2, 3: next 16 head dims
    // bytes (tok, even) (tok, odd) (tok+1, even) (tok+1, odd) -> (tok, even) (tok+1, even) | (tok, odd) (tok+1, odd)
    auto tile = [&](int mt, uint32_t lo, uint32_t hi) {
        const uint32_t x = __byte_perm(lo, 0u, 0x3120), y = __byte_perm(hi, 0u, 0x3120);
        const uint32_t a[4] = {e4m3x2_to_f16x2(x), e4m3x2_to_f16x2(x >> 16), e4m3x2_to_f16x2(y), e4m3x2_to_f16x2(y >> 16)};
#pragma unroll
        for (int n = 0; n < NB; ++n) mma_f16_16816(st.o[mt][n], a, pb[n][0], pb[n][1]);
    };
#pragma unroll
    for (int qd = 0; qd < D / 32; ++qd) {
        uint32_t r0, r1, r2, r3;
        ldmatrix_x4_trans(tok_chunk_f8<D>(v_tile, row, 2 * qd + csel), r0, r1, r2, r3);
        tile(2 * qd, r0, r1);
        tile(2 * qd + 1, r2, r3);
    }
}

// ----------------------------------------------------------------------------- leaving the accumulators
// One block's O^T tile mt, scaled per head, as bf16 rows: lane (r, c) gets two words of head 8n + r, and word_dim says which
// head dims they hold: bf16 caches 16 mt + 2c + {0, 1} and + 8, e4m3 caches 16 mt + 4c + {0, 1} and {2, 3}.
template <int D, int NB, bool F8>
__device__ __forceinline__ uint2 output_words(const WarpAttnState<D, NB> &st, int mt, int n, float f0, float f1)
{
    const uint32_t a = movmatrix_trans(pack_bf16x2(st.o[mt][n][0] * f0, st.o[mt][n][1] * f1));
    const uint32_t b = movmatrix_trans(pack_bf16x2(st.o[mt][n][2] * f0, st.o[mt][n][3] * f1));
    if constexpr (F8) return make_uint2(__byte_perm(a, b, 0x5410), __byte_perm(a, b, 0x7632));
    else return make_uint2(a, b);
}
// Stores them into a row of bf16 (16-byte aligned).
template <bool F8>
__device__ __forceinline__ void store_output_words(void *row, int mt, int lane, uint2 w)
{
    uint32_t *dst = reinterpret_cast<uint32_t *>(row) + mt * 8;
    if constexpr (F8) {
        *reinterpret_cast<uint2 *>(dst + 2 * (lane & 3)) = w;
    } else {
        dst[lane & 3] = w.x;
        dst[4 + (lane & 3)] = w.y;
    }
}

// This warp's share of a piece as rows of fp32 O, maximum and sum for the merge over warps: row(head) gives the row of a
// head, the maximum sits at off_m bytes, the sum behind it. finish_sums() has been called.
template <int D, int NB, bool F8, class RowOf>
__device__ __forceinline__ void dump_rows_f32(const WarpAttnState<D, NB> &st, int G, float vs, int off_m, RowOf row)
{
    const int lane = threadIdx.x & 31, r = lane >> 2;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
        if ((lane & 3) == 0 && 8 * n + r < G) *reinterpret_cast<float *>(row(8 * n + r) + off_m + 4) = st.l[n];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int head = 8 * n + 2 * (lane & 3) + e;
            if (head >= G) continue;
            uint8_t *rowb = row(head);
            float *o = reinterpret_cast<float *>(rowb);
            if (r == 0) *reinterpret_cast<float *>(rowb + off_m) = st.m[n][e];
#pragma unroll
            for (int mt = 0; mt < D / 16; ++mt) {
                if constexpr (F8) {
                    *reinterpret_cast<float2 *>(o + mt * 16 + 2 * r) = make_float2(st.o[mt][n][e] * vs, st.o[mt][n][2 + e] * vs);
                } else {
                    o[mt * 16 + r] = st.o[mt][n][e];
                    o[mt * 16 + 8 + r] = st.o[mt][n][2 + e];
                }
            }
        }
    }
}

}  // namespace l4l
