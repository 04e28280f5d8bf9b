// Gated linear recurrence of the RecurrentGemma block (RG-LRU): gates, normalisation, reset handling and
// the scan over the sequence in one kernel and one pass over the data; the state is handed from tile to
// tile on chip and written once at the end.
//
// The recurrence is sequential in time and independent across (sequence, channel). A CTA owns 64 channels
// of one sequence (two per lane, packed fp32x2 arithmetic) and walks the time axis in tiles of 16 steps,
// its 8 warps taking the tiles in turn (warp w: tiles w, w + 8, ...). Per tile a warp
//   1. has the tile's x, gate_x and gate_a in shared memory (its own TMA double buffer: as soon as a tile's
//      values are in registers the buffer is refilled with the warp's tile after next),
//   2. evaluates a_t and b_t of all 16 steps (independent of the state, so MUFU and FMA latencies overlap)
//      and, by linearity, the tile's aggregate: A = prod a_t and E = the end state from a zero start,
//   3. waits for the state at the start of the tile from the warp that owns the previous tile (shared
//      memory), hands A h + E on to the next warp at once,
//   4. and only then runs the recurrence proper from its start state and stores y.
// Only step 3 is serial along the sequence (a hand-off of 64 floats through shared memory per 16 steps);
// everything else runs 8 tiles at a time, which is what lets ONE sequence of 64 channels stream at a
// rate near an SM's share of HBM instead of at the latency of one warp.
// 8 bytes per (step, channel) move through HBM (3 bf16 read, 1 written) against 4 MUFU operations per
// channel (two tanh.approx sigmoids, ex2.approx, sqrt.approx) and about 25 issued instructions per channel
// pair and step.
//
// Narrow strips (template parameter kSplit = 2 or 4). A strip is one serial chain, so a launch is as long as the
// most loaded SM's chains: 160 strips on 148 SMs put two on twelve SMs and take twice the time of 148. For such
// launches the strips are made 32 or 16 channels wide, and a warp then owns kSplit CONSECUTIVE time tiles at once:
// lane = (sub-tile, channel pair), so every instruction still does 32 lanes' worth of work. Everything per lane is
// unchanged; the start states of a warp's later sub-tiles come from the earlier ones by kSplit - 1 shuffles
// (h <- A h + E) inside step 3. Twice or four times as many CTAs of half or a quarter of the work spread evenly.
//
// Segments. Where the strips fill the GPU more than once, a last round of a few strips leaves most SMs idle (320 strips of 32
// channels on 296 places: 181 us). The time axis is then cut as well: a CTA per (strip, segment), all first segments ahead of all
// second ones, the state passing through its place in global memory behind a counter per strip (release / acquire). Blocks
// start in the order of their indexes, so by the time a later segment gets a place its predecessor has long finished and nothing
// waits (the wait is bounded like every other): 135 us in four segments.
#include <type_traits>

#include "l4l_internal.h"
#include "l4l_ptx.cuh"

namespace l4l {

namespace {

constexpr int kTb = 16;          // time steps per tile
constexpr int kCb = 64;          // channels per CTA at kSplit = 1 (two per lane); kCb / kSplit otherwise
constexpr int kStages = 2;       // TMA buffers per warp
constexpr uint32_t kArrayBytes = kTb * kCb * 2;   // one array of a warp's tile: (kTb * kSplit) steps x (kCb / kSplit) channels
constexpr uint32_t kStageBytes = 3 * kArrayBytes;
// kTeam warps per CTA, each taking every kTeam-th tile: 8 for sequences, 16 when the launch has no more strips
// than the GPU has SMs (one CTA per SM then, and a strip's rate is set by how many tiles it has in flight)
constexpr size_t smem_bytes(int team)
{
    return 128 + (size_t)team * kStages * kStageBytes + (team * kStages + team) * 8 + 2 * kCb * 4 + 64;
}

struct RglruParams {
    const float *a_param;        // [W]
    const int32_t *position;     // [B, T] or null
    const int32_t *seq_lens;     // [B] or null
    float *state;                // [B, W] in/out
    __nv_bfloat16 *y;            // [B, T, W]
    unsigned *status;
    int *progress;               // [B, strips] segments of the strip that are done (null: one segment); zero between calls
    int seg_tiles;               // tiles (of kSteps steps) per segment
    int B, T, W;
};

__device__ __forceinline__ float tanh_approx(float x)
{
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sqrt_approx(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// two bf16 in one word -> packed fp32x2 (low half first)
__device__ __forceinline__ uint64_t widen2(uint32_t w) { return pack_u32x2(w << 16, w & 0xffff0000u); }

// The constants of a step's gates for two channels.
struct GateConsts {
    uint64_t k2h;                        // -4 softplus(a_param) log2(e)
    uint64_t half2, quarter2, nquarter2, s1c, s2c, s3c, s4c;
};

__device__ __forceinline__ GateConsts gate_consts(const float *a_param, int c, bool live)
{
    // (1 - a^2) / 4 = -expm1(z) / 4 with z = w log2(a), w = 2 ln 2: series coefficients in log2(a), the quarter (which
    // the square root turns into the half of sigmoid = 0.5 tanh + 0.5) folded in
    constexpr float kW = 1.3862943611198906f;
    GateConsts g;
    uint64_t k2 = pack_f32x2(0.f, 0.f);                  // -8 softplus(a_param) log2(e)
    if (live) {
        const float2 lam = *reinterpret_cast<const float2 *>(a_param + c);
        const float sp0 = lam.x > 15.f ? lam.x : log1pf(expf(lam.x));
        const float sp1 = lam.y > 15.f ? lam.y : log1pf(expf(lam.y));
        k2 = pack_f32x2(-8.f * 1.4426950408889634f * sp0, -8.f * 1.4426950408889634f * sp1);
    }
    g.half2 = pack_f32x2(0.5f, 0.5f);
    g.k2h = mul_f32x2(k2, g.half2);
    g.quarter2 = pack_f32x2(0.25f, 0.25f);
    g.nquarter2 = pack_f32x2(-0.25f, -0.25f);
    g.s1c = pack_f32x2(-kW / 4, -kW / 4);
    g.s2c = pack_f32x2(-kW * kW / 8, -kW * kW / 8);
    g.s3c = pack_f32x2(-kW * kW * kW / 24, -kW * kW * kW / 24);
    g.s4c = pack_f32x2(-kW * kW * kW * kW / 96, -kW * kW * kW * kW / 96);
    return g;
}

// A step's gates from the words of gate_x and gate_a: tanh(gate_x / 2), a and m / 2 of two channels.
__device__ __forceinline__ void gates_of(const GateConsts &g, uint32_t gx, uint32_t ga, uint64_t &th_x, uint64_t &a, float &m0, float &m1)
{
    constexpr float kW = 1.3862943611198906f, kNearOne = -0.0625f / kW;
    float g0, g1, r0, r1;
    unpack_f32x2(mul_f32x2(widen2(gx), g.half2), g0, g1);
    unpack_f32x2(mul_f32x2(widen2(ga), g.half2), r0, r1);
    th_x = pack_f32x2(tanh_approx(g0), tanh_approx(g1));                       // sigmoid = 0.5 tanh(z/2) + 0.5
    const uint64_t th_a = pack_f32x2(tanh_approx(r0), tanh_approx(r1));
    const uint64_t la2 = fma_f32x2(th_a, g.k2h, g.k2h);                        // log2(a) = k2 * sigmoid(gate_a)
    float l0, l1;
    unpack_f32x2(la2, l0, l1);
    a = pack_f32x2(fast_exp2(l0), fast_exp2(l1));
    // m / 2 = sqrt((1 - a^2) / 4): a short series when a is close to 1, where 1 - a*a cancels
    const uint64_t series = fma_f32x2(la2, fma_f32x2(la2, fma_f32x2(la2, g.s4c, g.s3c), g.s2c), g.s1c);
    float s0, s1, d0, d1;
    unpack_f32x2(mul_f32x2(la2, series), s0, s1);
    unpack_f32x2(fma_f32x2(mul_f32x2(a, g.nquarter2), a, g.quarter2), d0, d1);
    m0 = sqrt_approx(l0 > kNearOne ? s0 : d0);
    m1 = sqrt_approx(l1 > kNearOne ? s1 : d1);
}

// kSeg: the launch is cut along the time axis (an instantiation of its own: the other launches are 8 % faster without its code)
template <int kTeam, int kSplit, bool kSeg>
__global__ void __launch_bounds__(kTeam * 32)
rglru_scan_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_gx,
                  const __grid_constant__ CUtensorMap tmap_ga, const RglruParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    uint8_t *stages = smem;                                                    // [warp][stage][3 arrays]
    uint64_t *full = reinterpret_cast<uint64_t *>(stages + (size_t)kTeam * kStages * kStageBytes);   // [warp][stage]
    uint64_t *handed = full + kTeam * kStages;                                 // [warp]: the start state of its next tile is there
    float *carry = reinterpret_cast<float *>(handed + kTeam);                  // [2][kCb]: start state of tile j in slot j & 1
    volatile int *abort_flag = reinterpret_cast<volatile int *>(carry + 2 * kCb);

    constexpr int kCw = kCb / kSplit;                    // channels of this CTA's strip
    constexpr int kPairs = kCw / 2;                      // lanes per sub-tile (one channel pair each)
    constexpr int kSteps = kTb * kSplit;                 // time steps a warp owns at a time (kSplit sub-tiles of kTb)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / kPairs, cp = lane % kPairs;   // this lane's sub-tile and channel pair
    const int b = blockIdx.y, c0 = blockIdx.x * kCw;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kTeam * kStages; ++s) mbar_init(&full[s], 1);
        for (int w = 0; w < kTeam; ++w) mbar_init(&handed[w], 1);
        *abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
    }
    // everything above overlaps the tail of the kernel before; nothing is read before that has completed
    grid_dependency_wait();
    grid_launch_dependents();
    int L = p.seq_lens ? p.seq_lens[b] : p.T;
    L = L < 0 ? 0 : (L > p.T ? p.T : L);
    // this block's segment of the time axis: tiles [tile0, n_tiles) of the n_all tiles that the sequence has
    const int n_all = (L + kSteps - 1) / kSteps;
    const int segment = kSeg ? (int)blockIdx.z : 0, tile0 = kSeg ? segment * p.seg_tiles : 0;
    const int n_tiles = kSeg ? min(n_all, tile0 + p.seg_tiles) : n_all;
    if (kSeg && tile0 >= n_tiles) return;
    const int c = c0 + 2 * cp;
    const bool live = c < p.W;                           // W is even: both channels or neither

    if (warp == 0 && sub == 0) {
        // slot 0: the state that the block's first tile starts from (a later segment's: below)
        const float2 st = live && segment == 0 ? *reinterpret_cast<const float2 *>(p.state + (size_t)b * p.W + c) : make_float2(0.f, 0.f);
        *reinterpret_cast<float2 *>(carry + 2 * cp) = st;
    }
    __syncthreads();
    if (threadIdx.x == 0 && segment == 0) mbar_arrive(&handed[0]);

    uint8_t *my_stages = stages + (size_t)warp * kStages * kStageBytes;
    uint64_t *my_full = full + warp * kStages;
    // lane 0 requests this warp's k-th tile (tile tile0 + warp + k * kTeam) into its buffer k % kStages
    // (rows past T arrive as zeros and still count)
    auto request = [&](int k) {
        const int tile = tile0 + warp + k * kTeam;
        if (lane == 0 && tile < n_tiles) {
            const uint32_t s = k % kStages;
            mbar_arrive_expect_tx(&my_full[s], kStageBytes);
            uint8_t *dst = my_stages + s * kStageBytes;
            tma_load_3d(dst, &tmap_x, &my_full[s], c0, tile * kSteps, b);
            tma_load_3d(dst + kArrayBytes, &tmap_gx, &my_full[s], c0, tile * kSteps, b);
            tma_load_3d(dst + 2 * kArrayBytes, &tmap_ga, &my_full[s], c0, tile * kSteps, b);
        }
    };
    if (lane == 0) {
        tma_prefetch_desc(&tmap_x);
        tma_prefetch_desc(&tmap_gx);
        tma_prefetch_desc(&tmap_ga);
    }
    for (int k = 0; k < kStages; ++k) request(k);

    const GateConsts consts = gate_consts(p.a_param, c, live);
    const uint64_t one2 = pack_f32x2(1.f, 1.f), zero2 = pack_f32x2(0.f, 0.f);
    uint32_t *yrow = reinterpret_cast<uint32_t *>(p.y + (size_t)b * p.T * p.W + c);
    const size_t y_step = (size_t)p.W / 2;               // 32-bit words between time steps
    // Positions of a tile's steps, one per lane and part, as loaded: the vote that turns them into a mask comes a whole
    // tile later. (Voting right behind the load stalled every tile for an L2 round trip: B=4 x 8192 x 2560 with
    // positions 184 us, without them 140 us.)
    constexpr int kPosParts = (kSteps + 31) / 32;
    int pos_next[kPosParts];
    auto request_positions = [&](int tile) {
#pragma unroll
        for (int part = 0; part < kPosParts; ++part) {
            const int t = tile * kSteps + part * 32 + lane;
            pos_next[part] = (p.position && tile < n_tiles && part * 32 + lane < kSteps && t < L)
                                 ? __ldg(p.position + (size_t)b * p.T + t) : 1;
        }
    };
    auto resets_requested = [&]() -> unsigned {
        // bit t: step t of THIS LANE'S sub-tile is the first token of a segment (position 0). Nearly every tile has none.
        bool any = pos_next[0] == 0;
#pragma unroll
        for (int part = 1; part < kPosParts; ++part) any = any || pos_next[part] == 0;
        unsigned mine = 0u;
        if (!__any_sync(0xffffffffu, any)) return mine;
#pragma unroll
        for (int part = 0; part < kPosParts; ++part) {
            const unsigned bits = __ballot_sync(0xffffffffu, pos_next[part] == 0);
            if ((sub * kTb) / 32 == part) mine = (bits >> ((sub * kTb) % 32)) & 0xffffu;
        }
        return mine;
    };
    request_positions(tile0 + warp);

    int *progress = kSeg ? p.progress + (size_t)b * gridDim.x + blockIdx.x : nullptr;
    if (kSeg && warp == 0 && segment != 0) {
        // a later segment starts from the state that the strip's previous segment left in global memory
        if (lane == 0) {
            const long long w0 = clock64();
            while (ld_acquire_gpu(progress) != segment) {
                if (*abort_flag || clock64() - w0 > kWaitCycleBudget) {
                    *abort_flag = 1;
                    break;
                }
                __nanosleep(64);
            }
        }
        __syncwarp();
        if (sub == 0 && live) *reinterpret_cast<float2 *>(carry + 2 * cp) = __ldcg(reinterpret_cast<const float2 *>(p.state + (size_t)b * p.W + c));
        __syncwarp();
        if (lane == 0) mbar_arrive(&handed[0]);
    }
    for (int k = 0, tile = tile0 + warp; tile < n_tiles; ++k, tile += kTeam) {
        const uint32_t s = k % kStages, ph = (k / kStages) & 1u;
        const unsigned resets = resets_requested();
        request_positions(tile + kTeam);                 // in flight while this tile is processed
        if (!mbar_wait(&my_full[s], ph, abort_flag)) break;
        // the tile in shared memory: kSteps rows of kPairs words; this lane reads rows sub * kTb .. of column cp
        const uint32_t *xs = reinterpret_cast<const uint32_t *>(my_stages + s * kStageBytes) + sub * kTb * kPairs + cp;
        const uint32_t *gxs = xs + kTb * kCb / 2, *gas = gxs + kTb * kCb / 2;
        const int t0 = tile * kSteps + sub * kTb;            // first step of this lane's sub-tile
        const int n = max(0, min(kTb, L - t0));
        // ---- a_t and b_t = m_t i_t x_t of all steps of the tile (independent of the state). Tiles without a
        // reset and without a ragged end (nearly all) take the version without the per-step selects.
        uint64_t av[kTb], bv[kTb];
        auto gates = [&](auto plain_tag) {
            constexpr bool kPlain = decltype(plain_tag)::value;
#pragma unroll
            for (int t = 0; t < kTb; ++t) {
                const uint64_t xv = widen2(xs[t * kPairs]);
                uint64_t th_x, a;
                float m0, m1;
                gates_of(consts, gxs[t * kPairs], gas[t * kPairs], th_x, a, m0, m1);
                if constexpr (!kPlain) {
                    if ((resets >> t) & 1u) {                                          // uniform across a sub-tile's lanes
                        a = zero2;
                        m0 = m1 = 0.5f;
                    }
                    if (t >= n) {                                                      // past the end: the identity step
                        a = one2;
                        m0 = m1 = 0.f;
                    }
                }
                av[t] = a;
                const uint64_t mxh = mul_f32x2(pack_f32x2(m0, m1), xv);                    // m x / 2
                bv[t] = fma_f32x2(th_x, mxh, mxh);                                         // m x sigmoid(gate_x)
                if constexpr (!kPlain) {
                    // rows past the end are caller memory that may hold anything (0 * NaN is NaN): select, not multiply
                    if (t >= n) bv[t] = zero2;
                }
            }
        };
        if (__all_sync(0xffffffffu, resets == 0u && n == kTb))
            gates(std::true_type{});
        else
            gates(std::false_type{});
        // every lane has its values of this tile in registers: the buffer can take this warp's tile after next
        __syncwarp();
        request(k + kStages);
        // ---- the tile's aggregate: h_end = A h_start + E
        uint64_t A = one2, E = zero2;
#pragma unroll
        for (int t = 0; t < kTb; ++t) {
            E = fma_f32x2(av[t], E, bv[t]);
            A = mul_f32x2(A, av[t]);
        }
        // ---- the start state, from the owner of the previous tile (bounded wait); pass the end state on at once.
        // Every warp has its own barrier, completed once per tile it owns by the owner of the tile before; that
        // warp cannot reach its next arrival here before this warp has handed the present tile on, so the
        // phases are seen one by one.
        if (!mbar_wait(&handed[warp], k & 1u, abort_flag)) break;
        const int slot = (tile - tile0) & 1;
        const float2 hs = *reinterpret_cast<const float2 *>(carry + slot * kCb + 2 * cp);
        uint64_t h2 = pack_f32x2(hs.x, hs.y);                                  // start state of the warp's first sub-tile
        {
            // start states of the later sub-tiles, and the end state of the warp's steps: h <- A h + E along the
            // sub-tiles, the state travelling kPairs lanes up at each step
            float e0, e1;
            unpack_f32x2(fma_f32x2(A, h2, E), e0, e1);
#pragma unroll
            for (int u = 1; u < kSplit; ++u) {
                const float i0 = __shfl_up_sync(0xffffffffu, e0, kPairs), i1 = __shfl_up_sync(0xffffffffu, e1, kPairs);
                if (sub == u) {
                    h2 = pack_f32x2(i0, i1);
                    unpack_f32x2(fma_f32x2(A, h2, E), e0, e1);
                }
            }
            if (sub == kSplit - 1) *reinterpret_cast<float2 *>(carry + (slot ^ 1) * kCb + 2 * cp) = make_float2(e0, e1);
            __syncwarp();
            if (lane == 0) mbar_arrive(&handed[(warp + 1) % kTeam]);           // release: the slot is written
            if (tile + 1 == n_tiles && live && sub == kSplit - 1)              // the sequence, or its segment, ends here
                *reinterpret_cast<float2 *>(p.state + (size_t)b * p.W + c) = make_float2(e0, e1);
        }
        // ---- the recurrence proper, one packed FMA per step, and the outputs
#pragma unroll
        for (int t = 0; t < kTb; ++t) {
            if (t < n) {                                                       // uniform across a sub-tile's lanes
                h2 = fma_f32x2(av[t], h2, bv[t]);
                float h0, h1;
                unpack_f32x2(h2, h0, h1);
                if (live) yrow[(size_t)(t0 + t) * y_step] = pack_bf16x2(h0, h1);
            }
        }
    }
    if (kSeg && warp == (n_tiles - 1 - tile0) % kTeam && !*abort_flag) {
        // this warp stored the segment's end state: on to the next segment (the last one leaves the counter at zero for the
        // next call)
        __threadfence();
        __syncwarp();
        if (lane == 0) st_release_gpu(progress, n_tiles == n_all ? 0 : segment + 1);
    }
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) atomicOr(p.status + kStatusErrWord, kErrScanWait);
}

// A few steps (decode, T <= kTb): a thread per channel pair walks them, straight from global memory. There is too little
// work for a ring; the launch is one round trip to memory and a chain of gates. Against one warp and one TMA tile per 64
// channels, which worked out sixteen steps whatever T was (launches back to back): 64 x 1 x 4096 10.3 -> 4.5 us, 16 x 1 x 2560
// 6.2 -> 3.2, 8 x 16 x 2560 6.2 -> 3.8, 64 x 16 x 4096 12.3 -> 9.9, so it is taken up to sixteen steps.
struct RglruStepParams {
    const uint32_t *x, *gate_x, *gate_a;
    const float *a_param;
    const int32_t *position, *seq_lens;
    float *state;
    uint32_t *y;
    int T, W;
};

template <int kAtOnce>
__global__ void __launch_bounds__(128) rglru_steps_kernel(const RglruStepParams p)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const int b = blockIdx.y, pair = blockIdx.x * 128 + threadIdx.x, pairs = p.W / 2;
    if (pair >= pairs) return;
    const size_t row0 = (size_t)b * p.T;
    int L = p.seq_lens ? __ldg(p.seq_lens + b) : p.T;
    float2 *state = reinterpret_cast<float2 *>(p.state + (size_t)b * p.W) + pair;
    const float2 st = *state;
    uint64_t h = pack_f32x2(st.x, st.y);
    const GateConsts consts = gate_consts(p.a_param, 2 * pair, true);
    for (int t0 = 0; t0 < p.T; t0 += kAtOnce) {
        // asked for together with the length (rows past it may hold anything, and are not used)
        uint32_t xw[kAtOnce], gx[kAtOnce], ga[kAtOnce];
        int pos[kAtOnce];
#pragma unroll
        for (int t = 0; t < kAtOnce; ++t) {
            if (t0 + t < p.T) {
                const size_t at = (row0 + t0 + t) * pairs + pair;
                xw[t] = p.x[at];
                gx[t] = p.gate_x[at];
                ga[t] = p.gate_a[at];
                pos[t] = p.position ? __ldg(p.position + row0 + t0 + t) : 1;
            }
        }
#pragma unroll
        for (int t = 0; t < kAtOnce; ++t) {
            if (t0 + t < min(L, p.T)) {
                uint64_t th_x, a;
                float m0, m1;
                gates_of(consts, gx[t], ga[t], th_x, a, m0, m1);
                if (pos[t] == 0) {                                             // the first token of a segment
                    a = pack_f32x2(0.f, 0.f);
                    m0 = m1 = 0.5f;
                }
                const uint64_t mxh = mul_f32x2(pack_f32x2(m0, m1), widen2(xw[t]));
                h = fma_f32x2(a, h, fma_f32x2(th_x, mxh, mxh));
                float h0, h1;
                unpack_f32x2(h, h0, h1);
                p.y[(row0 + t0 + t) * pairs + pair] = pack_bf16x2(h0, h1);
            }
        }
    }
    if (L > 0) {
        float h0, h1;
        unpack_f32x2(h, h0, h1);
        *state = make_float2(h0, h1);
    }
}

}  // namespace

// the status block and one counter per strip (of the narrowest width) where they fit the region that decode calls on
// the same workspace leave at zero; a workspace of the status block alone is enough, the time axis is not cut then
size_t rglru_workspace_bytes(int B, int, int W)
{
    const size_t counters = (size_t)B * ((W + 15) / 16) * sizeof(int);
    return kStatusBytes + (counters <= kCounterBytes ? counters : 0);
}

namespace {

int tiles_of(int T, int split) { return (T + kTb * split - 1) / (kTb * split); }
int tiles_per_segment(int tiles, int segments, int team) { return (tiles + segments * team - 1) / (segments * team) * team; }   // whole rounds of the team

// A launch whose blocks may set themselves up under the tail of the kernel before: launches back to back 4 x 64 x 2560 6.2 -> 4.6 us,
// 16 x 300 x 1024 14.4 -> 13.2, 64 x 100 x 2560 46.7 -> 44.5; nothing on 4 x 8192 x 2560 (147 us).
struct Launch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr = {};
    Launch(dim3 grid, int threads, size_t smem, cudaStream_t stream)
    {
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cfg.gridDim = grid;
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
    }
    Launch(const Launch &) = delete;
};

template <int kTeam, int kSplit, bool kSeg = false>
l4l_status launch_shape(const void *x, const void *gate_x, const void *gate_a, RglruParams p, int segments, cudaStream_t stream)
{
    // one opt-in per instantiation and device
    static bool configured_on[kDeviceSlots] = {};
    const int slot = device_slot();
    if (slot < 0) return L4L_ERR_CUDA;
    {
        std::lock_guard<std::mutex> lock(setup_mutex());
        if (!configured_on[slot]) {
            if (cudaFuncSetAttribute(rglru_scan_kernel<kTeam, kSplit, kSeg>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem_bytes(kTeam)) != cudaSuccess)
                return L4L_ERR_CUDA;
            configured_on[slot] = true;
        }
    }
    constexpr int kCw = kCb / kSplit;
    CUtensorMap tx, tgx, tga;
    if (!make_tmap_rows_bf16(&tx, x, p.W, p.T, p.B, p.W, (int64_t)p.T * p.W, kCw, kTb * kSplit) ||
        !make_tmap_rows_bf16(&tgx, gate_x, p.W, p.T, p.B, p.W, (int64_t)p.T * p.W, kCw, kTb * kSplit) ||
        !make_tmap_rows_bf16(&tga, gate_a, p.W, p.T, p.B, p.W, (int64_t)p.T * p.W, kCw, kTb * kSplit))
        return L4L_ERR_CUDA;
    const int strips = (p.W + kCw - 1) / kCw, tiles = tiles_of(p.T, kSplit);
    p.seg_tiles = kSeg ? tiles_per_segment(tiles, segments, kTeam) : tiles;
    const dim3 grid(strips, p.B, (tiles + p.seg_tiles - 1) / p.seg_tiles);
    const Launch launch(grid, kTeam * 32, smem_bytes(kTeam), stream);
    return cudaLaunchKernelEx(&launch.cfg, rglru_scan_kernel<kTeam, kSplit, kSeg>, tx, tgx, tga, p) == cudaSuccess ? L4L_OK : L4L_ERR_CUDA;
}

}  // namespace

l4l_status launch_rglru_scan(const void *x, const void *gate_x, const void *gate_a, const float *d_a_param,
                             const int32_t *d_position, const int32_t *d_seq_lens, float *d_state, void *y, int B, int T,
                             int W, void *workspace, size_t ws_bytes, cudaStream_t stream)
{
    RglruParams p;
    p.a_param = d_a_param; p.position = d_position; p.seq_lens = d_seq_lens; p.state = d_state;
    p.y = static_cast<__nv_bfloat16 *>(y);
    p.status = static_cast<unsigned *>(workspace);
    p.B = B; p.T = T; p.W = W;
    p.progress = reinterpret_cast<int *>(static_cast<uint8_t *>(workspace) + kStatusBytes);
    if (T <= kTb) {
        const RglruStepParams sp{static_cast<const uint32_t *>(x), static_cast<const uint32_t *>(gate_x), static_cast<const uint32_t *>(gate_a),
                                 d_a_param, d_position, d_seq_lens, d_state, static_cast<uint32_t *>(y), T, W};
        const Launch launch(dim3((W / 2 + 127) / 128, B), 128, 0, stream);
        return cudaLaunchKernelEx(&launch.cfg, T == 1 ? rglru_steps_kernel<1> : rglru_steps_kernel<8>, sp) == cudaSuccess ? L4L_OK : L4L_ERR_CUDA;
    }
    int segs = 1;
    const int split = rglru_shape(B, T, W, d_position != nullptr, ws_bytes, &segs);
    if (segs > 1)
        return split == 4   ? launch_shape<8, 4, true>(x, gate_x, gate_a, p, segs, stream)
               : split == 2 ? launch_shape<8, 2, true>(x, gate_x, gate_a, p, segs, stream)
                            : launch_shape<8, 1, true>(x, gate_x, gate_a, p, segs, stream);
    if (split == 0) return launch_shape<16, 1>(x, gate_x, gate_a, p, 1, stream);
    if (split == 4) return launch_shape<8, 4>(x, gate_x, gate_a, p, 1, stream);
    if (split == 2) return launch_shape<8, 2>(x, gate_x, gate_a, p, 1, stream);
    return launch_shape<8, 1>(x, gate_x, gate_a, p, 1, stream);
}

// 0: 64-channel strips with teams of 16 warps; 1, 2, 4: teams of 8 warps on strips of 64, 32, 16 channels (sequences of at
// most kTb steps have no tiles). *segments (when given): into how many segments the time axis is cut; positions: the launch has reset positions.
static int rglru_strip_split(int B, int T, int W, int *segments, bool positions)
{
    if (segments) *segments = 1;
    if (T <= kTb) return 1;
    const long long sms = sm_count();
    // A strip is a serial chain that keeps an SM's issue slots busy, so a launch takes as long as the most loaded
    // SM. Estimated time of that SM, in units of one 64-channel strip on an SM of its own: k CTAs of 1/s strip each
    // take k / s; a lone team of 8 warps reaches about three quarters of the issue rate that two co-resident teams
    // or one team of 16 warps reach.
    auto strips = [&](int s) { return (long long)((W + kCb / s - 1) / (kCb / s)) * B; };
    auto fullest = [&](int s) { return (strips(s) + sms - 1) / sms; };
    int best = 1;
    double best_time = fullest(1) >= 2 ? (double)fullest(1) : 1.0 / 0.74;
    if (fullest(1) == 1 && T >= 16 * 2 * kTb) {
        best = 0;
        best_time = 1.0;
    }
    // narrower strips have to win by a tenth or more (their warps pay two or four dependent steps in the hand-off
    // instead of one), and the sequence has to be long enough for their wider tiles
    for (int s = 2; s <= 4; s *= 2) {
        const long long k = fullest(s);
        const double time = k >= 2 ? (double)k / s : (1.0 / s) / 0.74;
        if (time < 0.9 * best_time && T >= 8 * kTb * s) {
            best = s;
            best_time = time;
        }
    }
    // Segments: n blocks take n / (2 SMs) rounds of two resident teams each, a last round with a lone team on an SM 0.68 of
    // a full one; every round of a cut launch pays for set-up, first loads and the drain of the ring (about 1.5 us; 3 us on
    // 16-channel strips). A strip is cut only where the strips alone fill the GPU, so that a segment finds its predecessor
    // finished. B = 4 x 8192 x 2560 with positions, us by (channels, segments), thirty launches back to back on one build: (64, 1)
    // 205, (32, 1) 181, (16, 1) 154, which is the choice without segments, (64, 4) 186, (32, 2) 141, (32, 4) 135, (32, 8) 148, (16, 2) 145,
    // (16, 4) 162. (Kept up for a second the launch takes 148 us: the clock falls under the load.) The model is off by up to a
    // fifth where strips are wide or sequences few, but it orders the shapes well enough: over 92 sizes for which it cuts, of
    // 1024 to 5120 channels, cut launches take 0.86 to 1.013 times what the same launches take uncut, 90 of them less.
    if (!segments || best == 0) return best;
    const double us_per_step_channel = 4.54e-4;          // of a resident pair of teams
    auto estimate = [&](int s, int z) {
        const long long n = strips(s) * z, rest = n % (2 * sms);
        const double rounds = (double)(n / (2 * sms)) + (rest == 0 ? 0.0 : rest <= sms ? 0.68 : 1.0);
        return rounds * ((double)T / z * (kCb / s) * us_per_step_channel + (z == 1 ? 0.0 : s < 4 ? 1.5 : 3.0));
    };
    // (positions slow the uncut narrow shapes down most, every strip reads them; without them a cut has to promise more:
    // 3 x 5000 x 4096 111.0 us cut against 114.3 with positions, 107.0 against 104.0 without)
    best_time = (positions ? 0.95 : 0.85) * estimate(best, 1);
    for (int s = 1; s <= 4; s *= 2)
        for (int z = 2; z <= 4; z *= 2)
            if (strips(s) >= 2 * sms && T >= 1024 * z && estimate(s, z) < best_time) {
                best = s;
                best_time = estimate(s, z);
                *segments = z;
            }
    return best;
}

int rglru_shape(int B, int T, int W, bool positions, size_t ws_bytes, int *segments)
{
    const size_t needed = rglru_workspace_bytes(B, T, W);
    const bool with_counters = needed > kStatusBytes && ws_bytes >= needed;
    *segments = 1;
    const int split = rglru_strip_split(B, T, W, with_counters ? segments : nullptr, positions);
    if (*segments > 1) {
        const int tiles = tiles_of(T, split), each = tiles_per_segment(tiles, *segments, 8);
        *segments = (tiles + each - 1) / each;
    }
    return split;
}

}  // namespace l4l
