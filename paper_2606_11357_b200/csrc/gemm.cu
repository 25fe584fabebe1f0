// Prefill-phase fused GEMM (Section 4.3 "GEMM microkernel"), 1 <= M <= 4096 tokens.
//
// Output tile of one CTA: 128 weight columns (n) x bt tokens, computed "swapped": the dequantized
// weights are the 128-row operand of the tensor-core instruction, the activations the bt-column one,
//     D[n, token] = sum_k W[n, k] * A[token, k]          (tcgen05.mma, bf16 x bf16 -> fp32 in TMEM)
// so that each packed weight is unpacked and dequantized exactly once per CTA tile and then reused by
// all bt token rows (the dequantize-once rule of Section 4.1).
//
// The dequantized weights never touch shared memory: the dequant warps write them with tcgen05.st
// straight into tensor memory, from where tcgen05.mma reads its 128-row operand.  Shared memory then
// carries only the packed 4/8-bit tiles and the activations, which is what keeps the tensor pipe fed:
// with the bf16 weights staged in shared memory the kernel was bound by shared-memory bandwidth.
// Tensor memory (512 columns): one accumulator of up to 256 columns or two of up to 128, operand stages [256, 256 + 4 x 64).
//
// Persistent, warp-specialised CTA (640 threads):
//   warp 0      producer A: tiled TMA loads of activations (128B swizzle).
//   warp 1      tcgen05.mma, 8 per k-tile, and tcgen05.commit, by one elected lane of the converged warp.  (From a branch that
//               one lane takes alone an MMA costs 70 cycles to issue, because no operand is then provably uniform; this way
//               11 with 16 token columns and what it executes for, half a cycle per column, from 32 on.)
//   warp 2      allocates / frees tensor memory.
//   warp 3      producer W: bulk (TMA) copies of packed weight tiles (payload = weights + their scales
//               and zeros, Section 4.2).
//   warps 4-19  four groups of four (one warp per lane quarter of tensor memory).  They dequantize: packed words -> (q - z)
//               exact in bf16 -> times the scale, one rounding (split_scale) -> tcgen05.st, the k-tiles going round the groups; and
//               they drain the accumulators: tcgen05.ld -> bf16 -> y.  The packed words are stored in the register order
//               of the 16x256b store, so a word goes from shared memory to the tensor-memory operand without any shuffle.
// Work split: whole tiles, or the sequence of (output tile, k-tile) units cut into equal contiguous ranges, one per CTA
// (split_gemm).  A CTA that computes part of a tile whose last k-tile is another CTA's does that first and writes its fp32 sums
// to the workspace; the owner of the last k-tile adds them to its own in CTA order (deterministic) and stores y.
// What bounds it: with 256 tokens the tensor pipe (inside a tile a k-tile takes 1100 cycles in pairs of CTAs, 1024 of them MMA; between two
// tiles of a CTA the MMAs wait 6400 cycles for the one accumulator), at a clock that the power limit holds down in a loop (1.3 to 1.5 GHz); up
// to 128 tokens the issue slots of the dequant warps, 70 % used by 509 instructions per warp and k-tile (0.4 us), for short calls the 4 to 5 us
// around them.  us per call in a chain: 24x4096x14336 15.3, 77x2944x11016 (group 32) 13.4, 128x8192x8192 21.3, int8 80x4096x14336 19.1.
// Pairs of CTAs (PAIR): two CTAs of a cluster, on neighbouring SMs, share an output tile of 256 columns x bt tokens.  One MMA of 256 rows
// (cta_group::2) works on both halves, so each SM loads and holds only half of the activations.  A CTA on its own is bound by what its SM can
// take from the L2: 64 KB of activations and 8.5 KB of weights per k-tile of 256 tokens, 62 bytes per cycle at 1195 cycles; a pair takes 41 KB and
// 1100 cycles, and moves fewer bytes, which under the power limit is worth as much: us of the kernel as it is, alone -> in pairs, inputs
// changing, 2048x4096x14336 212.9 -> 196.4, 512x32768x4096 125.7 -> 115.4, int8 1024x4096x4096 34.1 -> 33.1; in a chain 1024x4096x8584 56.2 -> 53.1,
// 600x8192x8200 71.0 -> 66.9.  Each CTA unpacks and drains its own 128 columns; CTA 0 issues the MMAs, and the barriers that its MMA
// warp waits on are arrived at by both (choose_gemm_tiling says when).
// Every mbarrier wait is bounded; on a timeout all roles leave, TMEM is freed, the status word is set.
#include <cuda.h>

#include <atomic>
#include <cstddef>

#include "async.cuh"
#include "common.cuh"
#include "kernels.h"
#include "rings.h"
#include "tensormap.h"

namespace tf {

namespace {

constexpr int kGemmThreads = 640;
constexpr int kBN = 128;                  // weight columns per CTA tile (two packed strips)
constexpr int kFirstDequant = 4;
constexpr int kTmemAccCols = 256;
constexpr int kTmemCols = 512;

// workspace: [0,16) status | [kGemmFlagOffset, + 64 * CTAs) "this dequant warp's part of its CTA's slot is filled" | (the GEMV's
// partial-sum slots, not touched here) | one slot of BT tokens x 128 columns of fp32 sums per CTA (the part of a tile it contributes)
constexpr int kGemmFlagOffset = 4096;          // zero between calls
constexpr size_t kGemmPartialOffset = kWorkspaceZeroBytes;      // behind the GEMV's partial-sum slots, which must stay zero
constexpr int kGemmMaxGrid = 160;
static_assert(kGemmFlagOffset >= kGemvStatusBytes && kGemmFlagOffset + 4 * 4 * kGroups * kGemmMaxGrid <= kWorkspaceHeadBytes,
              "workspace layout shared with the GEMV");

// The CTA's unit range [u_begin, u_end) as segments of one output tile each, in processing order: the last tile first.  A tile
// that is cut between CTAs belongs to the CTA that has its last k-tile.  For that CTA it is the first tile of its range and comes
// last ("finish"), for the others the last tile of theirs and comes first ("contribute"), so their fp32 sums are usually
// there when the owner wants them.  An owner waits for CTAs of lower index only: those were started before it, so they run or
// have ended whatever else is on the GPU, and the lowest of them waits for nobody.
struct Segments {
    int ktiles, tile0, T0, units, count;
    __device__ Segments(int u_begin, int u_end, int ktiles_) : ktiles(ktiles_) {
        tile0 = u_begin / ktiles;
        T0 = u_begin - tile0 * ktiles;
        units = u_end - u_begin;
        count = units > 0 ? (T0 + units + ktiles - 1) / ktiles : 0;
    }
    __device__ void get(int i, int& tile, int& kt0, int& len) const {
        const int t = count - 1 - i;
        tile = tile0 + t;
        kt0 = t == 0 ? T0 : 0;
        len = min(ktiles, T0 + units - t * ktiles) - kt0;
    }
};

struct GemmBarriers {
    uint64_t act_full[kMaxActStages];     // activations landed
    uint64_t act_empty[kMaxActStages];    // tcgen05.commit: the MMAs that read them have run
    uint64_t op_full[kGroups];            // operand stage stored (the four warps of the group); tied: and its activations landed
    uint64_t op_done[kGroups];            // tcgen05.commit: the MMAs that read it have run
    uint64_t wp_full[kMaxWpStages];
    uint64_t wp_empty[kMaxWpStages];
    uint64_t acc_full[2];
    uint64_t acc_empty[2];
    uint32_t tmem_base;
    uint32_t abort_flag;        // [0] which wait gave up (0 = none) ...
    uint32_t wait_kcycles;      // ... [1] limit of a wait in units of 1024 cycles (read by mbar_wait through the flag's address)
};
static_assert(sizeof(GemmBarriers) <= kGemmBarrierBytes, "barrier block");

static_assert(offsetof(GemmBarriers, wait_kcycles) == offsetof(GemmBarriers, abort_flag) + 4, "mbar_wait reads the limit behind the flag");

// What a dequant warp does with its share of a segment's accumulator: the chunks `part`, `part + 4`, ... of its lane quarter, of 8 MATS
// tokens each: 16, or 8 where that is what gives every group of warps a chunk (32 tokens).  A chunk is read in the fragment layout of 8 x 8
// matrices (see tmem_ld_16x256b), the next one being on its way out of tensor memory meanwhile.  No MMA runs on a tile of 256 tokens until
// it is empty, so what counts is the chain of latencies of a chunk, and how few chunks there are (with 8 tokens a tile of 256 took 3700
// cycles, with 16 2900, measured with 1 KB per warp, so that its 16 tokens were transposed at once; a part of a cut one is bound by the L2,
// 128 KB of every CTA's in 5000 cycles).
template <int MATS>
struct DrainShare {
    uint32_t tmem;             // accumulator, this lane quarter
    int part, lane, chunks;    // chunks = bt / (8 MATS)
    uint8_t* tbuf;             // kDrainWarpBytes of this warp

    // A chunk rounded: matrix i of its eight columns c in m[c][i].
    __device__ __forceinline__ static void round(const float (&v)[8 * MATS], uint32_t (&m)[MATS][4]) {
#pragma unroll
        for (int c = 0; c < MATS; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) {       // the operand holds weights in 64ths
                const int r = 4 * MATS * (i >> 1) + 4 * c + 2 * (i & 1);
                m[c][i] = pack_bf16(kCodeUnit * v[r], kCodeUnit * v[r + 1]);
            }
    }
    // ... and stored.  y wants a token's columns side by side: the matrices are transposed by stmatrix and stored as 16 bytes per lane,
    // 8 columns of one token, eight tokens after the other through the same 512 bytes (why no more: kDrainWarpBytes).
    __device__ __forceinline__ void store(const uint32_t (&m)[MATS][4], __nv_bfloat16* y, int M, int N, int n0, int token0) const {
        const int n8 = n0 + 8 * (lane & 3), tl = lane >> 2;
        const uint32_t put = smem_u32(tbuf) + (lane & 7) * 64 + (((lane >> 3) ^ ((lane & 7) >> 1)) & 3) * 16;
        const uint4* get = reinterpret_cast<const uint4*>(tbuf + tl * 64 + (((lane & 3) ^ (tl >> 1)) & 3) * 16);
        __nv_bfloat16* to = y + (size_t)(token0 + tl) * N + n8;
#pragma unroll
        for (int c = 0; c < MATS; ++c) {
            stmatrix_x4_trans(put, m[c]);
            __syncwarp();
            const uint4 d = *get;
            if (token0 + tl + 8 * c < M && n8 < N) *reinterpret_cast<uint4*>(to + (size_t)(8 * c) * N) = d;
            __syncwarp();
        }
    }
    // A whole tile.
    __device__ __forceinline__ void whole(__nv_bfloat16* y, int M, int N, int n0, int token0) const {
        float v[8 * MATS];
        uint32_t m[MATS][4];
        if (part < chunks) tmem_ld_16x256b(tmem + 8 * MATS * part, v);
#pragma unroll 1
        for (int c = part; c < chunks; c += kGroups) {
            tmem_ld_wait_for(v);
            round(v, m);
            if (c + kGroups < chunks) tmem_ld_16x256b(tmem + 8 * MATS * (c + kGroups), v);
            store(m, y, M, N, n0, token0 + 8 * MATS * c);
        }
    }
    // Where this lane's sums of chunk c lie in a slot (as 2 MATS float4, 32 apart): a warp moves 512 bytes at a time.
    __device__ __forceinline__ int slot_index(int quarter, int c) const { return (quarter * chunks + c) * 64 * MATS + lane; }
    // A contributed part: the fp32 sums as they are.
    __device__ __forceinline__ void contribute(float4* slot, int quarter) const {
#pragma unroll 1
        for (int c = part; c < chunks; c += kGroups) {
            float v[8 * MATS];
            tmem_ld_16x256b(tmem + 8 * MATS * c, v);
            tmem_ld_wait_for(v);
            float4* p = slot + slot_index(quarter, c);
#pragma unroll
            for (int i = 0; i < 2 * MATS; ++i) __stcg(p + 32 * i, make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
        }
    }
    // The owner of a cut tile: its own sums, then the others' in CTA order (`slots`: the first one's slot, the next ones
    // `stride` float4 further each), rounded once.  The parts come one chunk of two contributors at a time, the next ones being on their way
    // while a chunk is added up, rounded and stored.
    __device__ __forceinline__ void finish(const float4* slots, size_t stride, int others, int quarter, __nv_bfloat16* y, int M, int N, int n0,
                                           int token0) const {
        float4 x[2][2 * MATS];
        auto ask = [&](int c, int o) {
            const float4* p = slots + o * stride + slot_index(quarter, c);
#pragma unroll
            for (int b = 0; b < 2; ++b)
                if (o + b < others)
#pragma unroll
                    for (int i = 0; i < 2 * MATS; ++i) x[b][i] = load_behind_wait(p + b * stride + 32 * i);
        };
        if (part < chunks) ask(part, 0);
#pragma unroll 1
        for (int c = part; c < chunks; c += kGroups) {
            float v[8 * MATS];
            tmem_ld_16x256b(tmem + 8 * MATS * c, v);
            tmem_ld_wait_for(v);
#pragma unroll 1
            for (int o = 0; o < others; o += 2) {
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    if (o + b < others)
#pragma unroll
                        for (int i = 0; i < 2 * MATS; ++i) {
                            v[4 * i] += x[b][i].x; v[4 * i + 1] += x[b][i].y;
                            v[4 * i + 2] += x[b][i].z; v[4 * i + 3] += x[b][i].w;
                        }
                if (o + 2 < others) ask(c, o + 2);
                else if (c + kGroups < chunks) ask(c + kGroups, 0);
            }
            uint32_t m[MATS][4];
            round(v, m);
            store(m, y, M, N, n0, token0 + 8 * MATS * c);
        }
    }
};

// An fp16 scale has 11 significant bits, a bf16 number 8.  Rounding the scale to bf16 would put the same relative
// error (up to 2^-8) on every weight of a group -- an error that does not average out over k.  So the scale is split
// into its upper 8 bits and the (at most 3) bits below, both exact in bf16, and a weight is
// fma(d, hi, d * lo): for 4-bit codes |d| <= 15 and d * lo is exact, so the result is bf16((q - z) * s) with a single
// rounding; for 8-bit codes d * lo is rounded at 2^-9 of a term that is 2^-8 of the weight, which changes nothing.
__device__ __forceinline__ void split_scale(float s, uint32_t& hi2, uint32_t& lo2) {
    const uint32_t bits = __float_as_uint(s);
    const uint32_t hi = bits & 0xFFFF0000u;                          // truncated to bf16
    const uint32_t lo = __float_as_uint(s - __uint_as_float(hi));    // exact, at most 3 significant bits
    hi2 = (hi >> 16) | hi;
    lo2 = (lo >> 16) | (lo & 0xFFFF0000u);
}
__device__ __forceinline__ uint32_t times_scale(uint32_t d, uint32_t hi2, uint32_t lo2) {
    uint32_t t, w;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(t) : "r"(d), "r"(lo2));
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(w) : "r"(d), "r"(hi2), "r"(t));
    return w;
}

}  // namespace

// G = groups per tile: 1 for group sizes that are multiples of 128, 2 / 4 for the 4-bit group sizes 64 / 32.
// BT = the widest token tile of the instantiation (it sizes the rings); bt = the token columns of this call's tiles, a
// multiple of 16.
template <int BITS, int BT, int G, bool PAIR>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_kernel(const __grid_constant__ CUtensorMap act_map, const uint8_t* __restrict__ blob,
            __nv_bfloat16* __restrict__ y, int M, int K, int N, int ktiles, int n_tiles, int m_tiles, int bt, int act_stages,
            int wp_stages, int aligned, const Ranges ranges,
            uint8_t* __restrict__ workspace, uint32_t debug) {
    static_assert(G == 1 || BITS == 4, "several groups per tile: the 4-bit format only");
    constexpr int kTileBytes = tile_bytes(BITS, G);
    constexpr int kWeightBytes = BITS == 4 ? kW4WeightBytes : kW8WeightBytes;
    constexpr int kWpStageBytes = wp_stage_bytes(BITS, BT, G);
    constexpr int kChunk = chunk_tiles(BITS, BT);
    constexpr int kAccs = BT > 128 ? 1 : 2;               // accumulators in tensor memory: where two fit, the next tile's MMAs run under a drain
    constexpr int kActK = act_stage_k(BT);
    constexpr bool kTied = tied(BT);
    static_assert(!PAIR || !kTied, "pairs of CTAs: the widest token tile only");
    // PAIR: this CTA is one of two that share an output tile of 256 columns; each has 128 of them and loads half of the token rows
    const int rank = PAIR ? (int)cta_rank_in_cluster() : 0;
    const int act_rows = PAIR ? bt / 2 : bt;             // token rows of a stage
    const int act_stage = act_rows * kActK * 2;          // bytes, a multiple of 1024 (act_rows is one of 16)
    constexpr size_t kSlotVec = (size_t)kBN * BT / 4;     // float4 of a CTA's slot

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_shared(smem_raw);
    uint8_t* act_ring = smem;                                        // act_stages x act_stage   (1024-aligned)
    uint8_t* wp_ring = act_ring + act_stages * act_stage;            // wp_stages x kWpStageBytes
    uint8_t* drain_buf = wp_ring + wp_stages * kWpStageBytes;        // 4 kGroups x kDrainWarpBytes
    GemmBarriers* bars = reinterpret_cast<GemmBarriers*>(drain_buf + 4 * kGroups * kDrainWarpBytes);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    // (the shuffle tells the compiler that the warp number is uniform in the warp)
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    // unit = (output tile, k-tile of 128); aligned: ranges of whole tiles (no tile is shared between CTAs)
    // Several CTAs per tile: the grid has a row of CTAs per tile, which share its k-tiles.  Otherwise it has one row.
    // (pairs: all of this counts pairs, and a pair's CTAs do the same in step)
    const int gx = blockIdx.x / (PAIR ? 2 : 1), gridx = gridDim.x / (PAIR ? 2 : 1);
    const int cta = blockIdx.y * gridx + gx;
    const int u_begin = ranges.start(gx) * (aligned ? ktiles : 1) + blockIdx.y * ktiles;
    const int u_end = ranges.start(gx + 1) * (aligned ? ktiles : 1) + blockIdx.y * ktiles;
    const Segments segs(u_begin, u_end, ktiles);
    const int strips = (N + kTileN - 1) / kTileN;
    HeaderWords header(blob);
    DeviceStatus* status = reinterpret_cast<DeviceStatus*>(workspace);
    float4* slots = reinterpret_cast<float4*>(workspace + kGemmPartialOffset) + (PAIR ? rank * kSlotVec : 0);
    constexpr size_t kSlotStride = (PAIR ? 2 : 1) * kSlotVec;            // from one CTA's slot to that of the next with the same columns
    const auto first_strip = [&](int tile) { return PAIR ? 4 * (tile / m_tiles) + 2 * rank : 2 * (tile / m_tiles); };

    // Producer W: packed weight tiles (weights + scales + zeros in one payload), the chunks [from, to) of the CTA's range.  The first
    // wp_stages chunks find their stages free.
    auto produce_weights = [&](int from, int to) {
        int s = 0, n = 0;
        uint32_t parity = 1;
        for (int i = 0; i < segs.count; ++i) {
            int tile, kt0, len;
            segs.get(i, tile, kt0, len);
            const int strip0 = first_strip(tile);
            const bool one = !PAIR || strip0 < strips, two = strip0 + 1 < strips;
            const uint8_t* src = blob + kHeaderBytes + ((size_t)strip0 * ktiles + kt0) * kTileBytes;
            for (int T = 0; T < len; T += kChunk, src += kChunk * kTileBytes, ++n) {
                if (n >= to) return;
                if (n >= from) {
                    if (n >= wp_stages && !mbar_wait(smem_u32(&bars->wp_empty[s]), parity, abort_flag, 0x300 + s)) return;
                    const uint32_t bar = smem_u32(&bars->wp_full[s]), dst = smem_u32(wp_ring + s * kWpStageBytes);
                    const uint32_t bytes = min(kChunk, len - T) * kTileBytes;
                    mbar_arrive_expect_tx(bar, two ? 2 * bytes : one ? bytes : 0);
                    if (one) bulk_copy_g2s(dst, src, bytes, bar);
                    if (two) bulk_copy_g2s(dst + kChunk * kTileBytes, src + (size_t)ktiles * kTileBytes, bytes, bar);
                }
                if (++s == wp_stages) { s = 0; parity ^= 1u; }
            }
        }
    };
    const int early_chunks = min(2, wp_stages);               // issued ahead of the CTA's barrier: never more than the ring holds
    const bool drop_weights = (debug & kDebugDropWeights) != 0;       // failure-path test: nothing ever arrives on wp_full

    // The set-up sits between the start of a CTA and its first copy: a thread per stage, and the thread that copies the weights (constants)
    // initialises their barriers itself, while the header of the blob is on its way, and starts before the others are ready (in a
    // chain the last CTAs to find an SM, 3 us behind the others, end the call: 24x4096x4096 9.6 -> 9.2 us, 77x2944x11016, group 32,
    // 15.4 -> 14.8, 128x4096x14336 21.9 -> 21.4).
    if (threadIdx.x < kMaxActStages) {
        mbar_init(smem_u32(&bars->act_full[threadIdx.x]), 1);
        mbar_init(smem_u32(&bars->act_empty[threadIdx.x]), 1);
        mbar_init_fence();
    } else if (threadIdx.x == 96) {
        for (int s = 0; s < wp_stages; ++s) {
            mbar_init(smem_u32(&bars->wp_full[s]), 1);
            mbar_init(smem_u32(&bars->wp_empty[s]), 4 * kChunk);      // the groups of the chunk
        }
        mbar_init_fence();
        if (header.fit(BITS, (uint32_t)K, (uint32_t)N, G) && !drop_weights) produce_weights(0, early_chunks);
    } else if (threadIdx.x >= 32 && threadIdx.x < 32 + kGroups) {
        mbar_init(smem_u32(&bars->op_full[threadIdx.x - 32]), kTied ? 5 : PAIR ? 8 : 4);
        mbar_init(smem_u32(&bars->op_done[threadIdx.x - 32]), 1);
        mbar_init_fence();
    } else if (threadIdx.x >= 128 && threadIdx.x < 128 + kAccs) {
        mbar_init(smem_u32(&bars->acc_full[threadIdx.x - 128]), 1);
        mbar_init(smem_u32(&bars->acc_empty[threadIdx.x - 128]), (PAIR ? 8 : 4) * kGroups);      // every dequant warp has drained its share
        mbar_init_fence();
    } else if (threadIdx.x == 160) {
        bars->abort_flag = 0;
        bars->wait_kcycles = wait_limit_kcycles(debug);
        mbar_init_fence();
    }
    if (warp == 2) {
        if constexpr (PAIR) {
            tmem_alloc_pair(smem_u32(&bars->tmem_base), kTmemCols);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(smem_u32(&bars->tmem_base), kTmemCols);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();             // the barriers of both CTAs are ready
    tc_fence_after();
    const bool header_ok = header.fit(BITS, (uint32_t)K, (uint32_t)N, G);
    // The next kernel of the stream may start as SMs become free: its set-up and its first weights then run under the last
    // CTAs of this one (released at the end of the kernel instead, a short GEMM took 1 to 2 us longer in a chain).
    grid_launch_dependents();
    const uint32_t tmem_base = bars->tmem_base;
    const uint32_t tmem_a = tmem_base + kTmemAccCols;        // weight-operand stages, one of 64 columns per group

    // Programmatic dependent launch: this kernel may have been started while the previous kernel of the stream was
    // still running.  Only the packed weights (constants) are read before grid_dependency_wait(); activations, y and
    // the workspace are touched after it (by the activation producer, and by the dequant warps when they drain).
    if (warp == 0) grid_dependency_wait();

    if (header_ok) {
        if (warp == 0 && lane == 0) {
            // ================= producer A: activations, one TMA load per stage ====================================
            prefetch_tensormap(&act_map);
            int s = 0, s0 = 0;
            uint32_t parity = kTied ? 0xFu : 1u;              // tied: bit s, operand stage s
            bool ok = true;
            for (int i = 0; i < segs.count && ok; ++i) {
                int tile, kt0, len;
                segs.get(i, tile, kt0, len);
                const int token0 = tile % m_tiles * bt + rank * act_rows;
                for (int T = 0; T < len * (kTileK / kActK); ++T) {
                    if (kTied) s = s0 + T % kChunk;
                    ok = mbar_wait(smem_u32(kTied ? &bars->op_done[s] : &bars->act_empty[s]), kTied ? (parity >> s) & 1u : parity, abort_flag, 0x310 + s);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(kTied ? &bars->op_full[s] : &bars->act_full[s]);
                    const int z = (2 * kt0 * kBK + T * kActK) / kBK;
                    if constexpr (PAIR) {               // both halves are counted by the barrier of the CTA that issues the MMAs
                        if (rank == 0) mbar_arrive_expect_tx(bar, 2 * act_stage);
                        tma_load_3d_pair(smem_u32(act_ring + s * act_stage), &act_map, 0, token0, z, map_to_cta(bar, 0));
                    } else {
                        mbar_arrive_expect_tx(bar, act_stage);
                        tma_load_3d(smem_u32(act_ring + s * act_stage), &act_map, 0, token0, z, bar);
                    }
                    if (kTied) {
                        parity ^= 1u << s;
                        if (T % kChunk == kChunk - 1 || T == len - 1) s0 = (s0 + kChunk) % kGroups;
                    } else if (++s == act_stages) { s = 0; parity ^= 1u; }
                }
            }
        } else if (warp == 3 && lane == 0) {
            if (!drop_weights) produce_weights(early_chunks, 1 << 30);
        } else if (warp == 1 && rank == 0) {
            // ================= MMA issuer: one elected lane of the converged warp =================================
            const uint32_t idesc = umma_idesc_bf16(PAIR ? 2 * kBN : kBN, bt);
            const auto commit = [](uint32_t bar) { PAIR ? tc_commit_pair(bar) : tc_commit(bar); };
            const auto wait = [&](uint64_t* bar, uint32_t parity, uint32_t site) {
                return PAIR ? mbar_wait_warp_cluster(smem_u32(bar), parity, abort_flag, site) : mbar_wait_warp(smem_u32(bar), parity, abort_flag, site);
            };
            int s0 = 0, as = 0;                               // the chunk's first operand stage (= group)
            uint32_t parity = 0, aparity = 0;                 // bit s of `parity`: operand stage s
            bool ok = true;
            for (int i = 0; i < segs.count && ok; ++i) {
                int tile, kt0, len;
                segs.get(i, tile, kt0, len);
                const int acc = i % kAccs;
                const uint32_t d = tmem_base + acc * (kTmemAccCols / kAccs);
                ok = wait(&bars->acc_empty[acc], (i / kAccs & 1) ^ 1, 0x400);
                tc_fence_after();
                for (int T = 0; T < len && ok; ++T) {
                    const int s = s0 + T % kChunk;
                    ok = wait(&bars->op_full[s], (parity >> s) & 1u, 0x410 + s);
                    parity ^= 1u << s;
#pragma unroll
                    for (int part = 0; part < kTileK / kActK; ++part) {
                        if (!kTied) ok = ok && wait(&bars->act_full[as], aparity, 0x420 + as);
                        if (!ok) break;
                        tc_fence_after();
                        const uint64_t b_desc = umma_desc_k_sw128(smem_u32(act_ring + (kTied ? s : as) * act_stage));
                        const uint32_t a = tmem_a + 64 * s + kActK / 2 * part;
                        if (elect_one()) {
#pragma unroll
                            for (int j = 0; j < kActK / 16; ++j)   // 16 k per instruction: 8 TMEM columns / 32 smem bytes
                                if constexpr (PAIR) tc_mma_f16_tmem_a_pair(d, a + 8 * j, b_desc + 2 * (j & 3), idesc, (T | part | j) != 0 ? 1u : 0u);
                                else tc_mma_f16_tmem_a(d, a + 8 * j, b_desc + 2 * (j & 3) + (j >> 2) * (bt * kBK * 2 / 16), idesc, (T | part | j) != 0 ? 1u : 0u);
                            if (!kTied) commit(smem_u32(&bars->act_empty[as]));
                            if (part == kTileK / kActK - 1) commit(smem_u32(&bars->op_done[s]));
                        }
                        __syncwarp();
                        if (!kTied && ++as == act_stages) { as = 0; aparity ^= 1u; }
                    }
                    if (T % kChunk == kChunk - 1 || T == len - 1) s0 = (s0 + kChunk) % kGroups;
                }
                if (!ok) break;
                if (elect_one()) commit(smem_u32(&bars->acc_full[acc]));
                __syncwarp();
            }
        } else if (warp >= kFirstDequant) {
            // ================= dequantize: packed tile -> bf16 operand in tensor memory ========================
            // The k-tiles of the CTA's range go round the four groups.  A group works on its k-tile alone, so the groups are at
            // different points of the chain "weights landed -> shared memory -> arithmetic -> tensor memory -> MMA" and
            // hide each other's latencies (with all warps on one k-tile at a time the chain took 1100 cycles per k-tile,
            // against 450 cycles of arithmetic).  Quarter q of tensor memory = 32 weight columns: strip q >> 1,
            // 16-column blocks 2 (q & 1) and the next.  Thread (g, t) owns rows g, g + 8 of both blocks and, per k-block,
            // the four consecutive k its packed word holds.
            const int q = warp & 3, group = (warp - kFirstDequant) >> 2;
            const int strip_sel = q >> 1;
            const int g = lane >> 2;
            const uint32_t quarter = uint32_t(32 * q) << 16;
            const uint32_t operand = tmem_a + 64 * group + quarter;
            // Every kRound-th chunk is this group's.  The loop below steps from one to the next; stepping through all of them and leaving out the
            // others' cost 450 to 750 of the 3900 to 4900 cycles that a group takes for a k-tile (us, 24x4096x14336 16.1 -> 15.5, 64x4096x14336
            // 17.0 -> 16.7, 128x4096x14336 18.9 -> 18.6, 300x4096x11008 36.8 -> 36.0, 2048x4096x14336 211.5 -> 209.0).
            constexpr int kRound = kGroups / kChunk;
            int behind = group / kChunk, ws = group / kChunk; // chunks from the start of the segment to this group's next one
            uint32_t wparity = 0, done_parity = 1;
            bool ok = true, waited = false;
            // Drain duty: these sixteen warps empty the accumulator of every segment (and release it), each a quarter of its lane
            // quarter, as soon as it is full and at a job boundary.  At the latest before a job that waits for the MMAs of a
            // segment (those of the group's job before it, in segment last_seg) that waits for that accumulator.
            uint32_t* flags = reinterpret_cast<uint32_t*>(workspace + kGemmFlagOffset) + (warp - kFirstDequant);
            int duty = 0, last_seg = 0;
            constexpr int kDrainMats = BT > 32 ? 2 : 1;
            DrainShare<kDrainMats> share;
            share.part = group; share.lane = lane; share.chunks = bt / (8 * kDrainMats);
            // arrivals on the barriers of the CTA that issues the MMAs
            const auto arrive_issuer = [&](uint64_t* bar) {
                if constexpr (PAIR) mbar_arrive_cluster(map_to_cta(smem_u32(bar), 0));
                else mbar_arrive(smem_u32(bar));
            };
            share.tbuf = drain_buf + (warp - kFirstDequant) * kDrainWarpBytes;
            auto do_duty = [&](int sidx) -> bool {
                const int acc = sidx % kAccs;
                if (!mbar_wait_warp(smem_u32(&bars->acc_full[acc]), sidx / kAccs & 1, abort_flag, 0x520)) return false;
                tc_fence_after();
                int dtile, dkt0, dlen;
                segs.get(sidx, dtile, dkt0, dlen);
                const int n0 = first_strip(dtile) * kTileN + 32 * q, token0 = dtile % m_tiles * bt;
                share.tmem = tmem_base + acc * (kTmemAccCols / kAccs) + quarter;
                if (!waited) { grid_dependency_wait(); waited = true; }        // y and the workspace belong to earlier kernels until now
                if (dkt0 + dlen != ktiles) {
                    // the owner's warp of the same number takes what this one stores, so each pair has a flag of its own
                    share.contribute(slots + cta * kSlotStride, q);
                    __syncwarp();
                    if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(flags + (PAIR ? 2 * cta + rank : cta) * 4 * kGroups), "r"(1u) : "memory");
                } else if (dkt0 != 0) {
                    const int first = gridDim.y > 1 ? dtile * gridx : ranges.owner(dtile * ktiles), others = cta - first;
                    for (int o = 0; o < others; o += 32) {              // a lane per contributor
                        uint32_t* flag = flags + (PAIR ? 2 * (first + o + lane) + rank : first + o + lane) * 4 * kGroups;
                        const bool mine = o + lane < others;
                        const long long t_begin = clock64();
                        for (;;) {
                            uint32_t f = 1;
                            if (mine) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(f) : "l"(flag) : "memory");
                            if (__all_sync(0xFFFFFFFFu, f != 0)) break;
                            if (wait_given_up(t_begin, abort_flag, 0x610)) return false;
                        }
                        if (mine) *flag = 0;                            // zero for the next call
                    }
                    __syncwarp();
                    share.finish(slots + first * kSlotStride, kSlotStride, others, q, y, M, N, n0, token0);
                } else {
                    share.whole(y, M, N, n0, token0);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) arrive_issuer(&bars->acc_empty[acc]);
                return true;
            };
            for (int i = 0; i < segs.count && ok; ++i) {
                int tile, kt0, len;
                segs.get(i, tile, kt0, len);
                const bool strip_exists = first_strip(tile) + strip_sel < strips;
                int T = behind * kChunk;
                for (; T < len && ok; T += kRound * kChunk) {
                    auto release_stage = [&]() {
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&bars->wp_empty[ws]));
                        ws += kRound;
                        if (ws >= wp_stages) { ws -= wp_stages; wparity ^= 1u; }
                    };
                    ok = mbar_wait_warp(smem_u32(&bars->wp_full[ws]), wparity, abort_flag, 0x500 + ws);
                    if (!ok) break;
                    if (T + group % kChunk >= len) {          // a chunk of one k-tile, and it is the other group's
                        release_stage();
                        continue;
                    }
                    while (ok && duty < last_seg &&
                           (duty + kAccs <= last_seg ||
                            __all_sync(0xFFFFFFFFu, mbar_try_wait(smem_u32(&bars->acc_full[duty % kAccs]), duty / kAccs & 1))))
                        ok = do_duty(duty++);
                    if (!ok) break;
                    last_seg = i;
                    const uint8_t* tile_smem = wp_ring + ws * kWpStageBytes + (strip_sel * kChunk + group % kChunk) * kTileBytes;
                    // scales of rows (w0,g), (w0,g+8), (w0+1,g), (w0+1,g+8), split into two exact bf16 parts
                    uint32_t s_g[2], s_g8[2], l_g[2], l_g8[2], zg[2], zg8[2];
                    auto load_scales = [&](int gr) {
                        const uint2 sc = *(reinterpret_cast<const uint2*>(tile_smem + kWeightBytes + gr * kScaleBytes + g * 16) + (q & 1));
                        const uint32_t sw[2] = {sc.x, sc.y};
#pragma unroll
                        for (int b = 0; b < 2; ++b) {
                            split_scale(fp16_bits_to_float((uint16_t)(sw[b] & 0xFFFFu)), s_g[b], l_g[b]);
                            split_scale(fp16_bits_to_float((uint16_t)(sw[b] >> 16)), s_g8[b], l_g8[b]);
                        }
                        if (BITS == 4) {
                            const uint32_t zword = *(reinterpret_cast<const uint32_t*>(tile_smem + w4_zero_offset(G, gr)) + g);
#pragma unroll
                            for (int b = 0; b < 2; ++b) w4_minus_zero(q & 1 ? zword >> 8 : zword, b, zg[b], zg8[b]);
                        }
                    };
                    // four steps of 32 k (two k-blocks, half of a 32-column quarter of the stage each)
#pragma unroll
                    for (int step = 0; step < 4; ++step) {
                        if (step % (4 / G) == 0) load_scales(step * G / 4);
                        uint32_t op[2][8];                    // [block][register of the 16x256b.x2 store]
#pragma unroll
                        for (int kb = 0; kb < 2; ++kb) {
                            if (BITS == 4) {
                                const uint2 x = *(reinterpret_cast<const uint2*>(tile_smem + ((2 * step + kb) * 32 + lane) * 16) + (q & 1));
                                const uint32_t xs[2] = {x.x, x.y};
#pragma unroll
                                for (int b = 0; b < 2; ++b) {
                                    op[b][4 * kb + 0] = times_scale(w4_reg(xs[b], 0, zg[b]), s_g[b], l_g[b]);     // row g,   k 0,1
                                    op[b][4 * kb + 1] = times_scale(w4_reg(xs[b], 2, zg[b]), s_g[b], l_g[b]);     // row g,   k 2,3
                                    op[b][4 * kb + 2] = times_scale(w4_reg(xs[b], 1, zg8[b]), s_g8[b], l_g8[b]);  // row g+8, k 0,1
                                    op[b][4 * kb + 3] = times_scale(w4_reg(xs[b], 3, zg8[b]), s_g8[b], l_g8[b]);  // row g+8, k 2,3
                                }
                            } else {
                                const uint4 x = *reinterpret_cast<const uint4*>(tile_smem + (((2 * step + kb) * 2 + (q & 1)) * 32 + lane) * 16);
                                const uint32_t xs[2][2] = {{x.x, x.y}, {x.z, x.w}};
#pragma unroll
                                for (int b = 0; b < 2; ++b) {
                                    uint32_t r0, r1, r2, r3;
                                    w8_word_to_regs(xs[b][0], r0, r1);                     // (row g; k 0,1), (row g+8; k 0,1)
                                    w8_word_to_regs(xs[b][1], r2, r3);                     // (row g; k 2,3), (row g+8; k 2,3)
                                    op[b][4 * kb + 0] = times_scale(r0, s_g[b], l_g[b]);
                                    op[b][4 * kb + 1] = times_scale(r2, s_g[b], l_g[b]);
                                    op[b][4 * kb + 2] = times_scale(r1, s_g8[b], l_g8[b]);
                                    op[b][4 * kb + 3] = times_scale(r3, s_g8[b], l_g8[b]);
                                }
                            }
                        }
                        if (step == 3) release_stage();       // the packed stage has been read
                        if (step == 0) {
                            // the MMAs that read this operand stage last have run
                            ok = mbar_wait_warp(smem_u32(&bars->op_done[group]), done_parity, abort_flag, 0x510 + group);
                            if (!ok) break;
                            done_parity ^= 1u;
                            tc_fence_after();
                        }
                        if (strip_exists) {
                            tmem_st_16x256b_x2(operand + 16 * step, op[0]);
                            tmem_st_16x256b_x2(operand + 16 * step + (16u << 16), op[1]);
                        }
                    }
                    if (!ok) break;
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) arrive_issuer(&bars->op_full[group]);
                }
                behind = (T - (len + kChunk - 1) / kChunk * kChunk) / kChunk;
            }
            while (ok && duty < segs.count) ok = do_duty(duty++);
        }
    }

    // ---------------- teardown --------------------------------------------------------------------------------
    grid_dependency_wait();                                   // (returns at once where it has returned before)
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!header_ok) {
            if (cta == 0 && rank == 0) { status->code = TF_ERR_BLOB; status->detail = 1; }
        } else if (bars->abort_flag != 0) {
            status->code = TF_ERR_TIMEOUT;
            status->detail = bars->abort_flag;
            const long long t_begin = clock64();              // let copies / MMAs in flight land before freeing
            while (clock64() - t_begin < 2000000ll) {}
        }
    }
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();             // nobody touches the other CTA's memory any more (every wait above is bounded)
    if (warp == 2) {
        tc_fence_after();
        if constexpr (PAIR) tmem_dealloc_pair(tmem_base, kTmemCols);
        else tmem_dealloc(tmem_base, kTmemCols);
    }
}

// ------------------------------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------------------------------
size_t gemm_workspace_bytes(int M, int K, int N) {
    (void)K; (void)N;
    return (size_t)kGemmPartialOffset + (size_t)kGemmMaxGrid * kBN * gemm_widest_tile(M) * 4;      // one slot per CTA
}

namespace {

template <int BITS, int BT, int G, bool PAIR = false>
cudaError_t launch_bt(const GemmTiling& tiling, const void* blob, const void* a, void* y, int M, int K, int N, void* workspace, cudaStream_t stream) {
    const int m_tiles = tiling.m_tiles, bt = tiling.bt;
    const GemmSplit& split = tiling.split;
    CUtensorMap map;
    // [K / 64][M][64]: a load brings the 64-k blocks of its stage one after the other, each in the 128-byte rows of the swizzle
    const cuuint64_t dims[3] = {kBK, (cuuint64_t)M, (cuuint64_t)K / kBK};
    const cuuint64_t strides[2] = {(cuuint64_t)K * 2, kBK * 2};
    const int act_rows = PAIR ? bt / 2 : bt;
    const cuuint32_t box[3] = {kBK, (cuuint32_t)act_rows, (cuuint32_t)(act_stage_k(BT) / kBK)};
    cudaError_t me = encode_bf16_map(&map, a, 3, dims, strides, box);
    if (me != cudaSuccess) return me;

    const GemmRings rings = gemm_rings(BITS, BT, act_rows, G);
    // function attributes belong to one device: set them once per device and kernel (twice is harmless)
    constexpr int kMaxDevices = 64;
    // (an atomic flag: two host threads may both find it unset and both set the attribute, which is harmless)
    static std::atomic<bool> configured_on[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
    const bool seen = dev >= 0 && dev < kMaxDevices;
    if (!seen || !configured_on[dev].load(std::memory_order_acquire)) {
        cudaError_t e = cudaFuncSetAttribute(gemm_kernel<BITS, BT, G, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kGemmSmemMax);
        if (e != cudaSuccess) return e;
        if (seen) configured_on[dev].store(true, std::memory_order_release);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(split.grid / split.rows * (PAIR ? 2 : 1), split.rows, 1);
    cfg.blockDim = dim3(kGemmThreads, 1, 1);
    cfg.dynamicSmemBytes = rings.smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // see grid_dependency_wait() in the kernel
    const StreamNote note(stream);
    attr[0].val.programmaticStreamSerializationAllowed = note.may_start_early() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = PAIR ? 2 : 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_kernel<BITS, BT, G, PAIR>, map, static_cast<const uint8_t*>(blob), static_cast<__nv_bfloat16*>(y),
                                             M, K, N, K / kTileK, (N + kBN - 1) / kBN, m_tiles, bt, rings.act_stages, rings.wp_stages,
                                             split.whole_tiles ? 1 : 0, split.ranges, static_cast<uint8_t*>(workspace), debug_word());
    if (e == cudaSuccess) note.launched(LaunchKind::kWholeSm);
    return e;
}

template <int BITS, int G = 1>
cudaError_t launch_bits(const void* blob, const void* a, void* y, int M, int K, int N, void* workspace, int sm_count,
                        cudaStream_t stream) {
    if (sm_count > kGemmMaxGrid) sm_count = kGemmMaxGrid;
    const GemmTiling tiling = choose_gemm_tiling(M, (N + kBN - 1) / kBN, K / kTileK, sm_count);
    if (tiling.pair) return launch_bt<BITS, 256, G, true>(tiling, blob, a, y, M, K, N, workspace, stream);
    if (tiling.width == 256) return launch_bt<BITS, 256, G>(tiling, blob, a, y, M, K, N, workspace, stream);
    if (tiling.width == 128) return launch_bt<BITS, 128, G>(tiling, blob, a, y, M, K, N, workspace, stream);
    if (tiling.width == 64) return launch_bt<BITS, 64, G>(tiling, blob, a, y, M, K, N, workspace, stream);
    return launch_bt<BITS, 32, G>(tiling, blob, a, y, M, K, N, workspace, stream);
}

}  // namespace

cudaError_t launch_gemm(int bits, const void* blob, const void* a, void* y, int M, int K, int N, void* workspace,
                        int sm_count, cudaStream_t stream, int groups) {
    if (groups == 2 && bits == 4) return launch_bits<4, 2>(blob, a, y, M, K, N, workspace, sm_count, stream);
    if (groups == 4 && bits == 4) return launch_bits<4, 4>(blob, a, y, M, K, N, workspace, sm_count, stream);
    if (groups != 1) return cudaErrorInvalidValue;
    return bits == 4 ? launch_bits<4>(blob, a, y, M, K, N, workspace, sm_count, stream)
                     : launch_bits<8>(blob, a, y, M, K, N, workspace, sm_count, stream);
}

}  // namespace tf
