// Decode-phase fused GEMV, M = 1..16 tokens (Sections 4.3 "GEMV microkernel" and 4.4).
//
// Persistent streaming kernel.  The packed blob is one long sequence of tiles (128 k x 64 n, each a
// contiguous payload carrying its scales and zeros, strip after strip).  That sequence is cut into
// equal contiguous ranges, one per CTA, so every CTA streams one contiguous byte range of HBM:
//
//   producer warp : one lane issues, per ring stage, one bulk (TMA) copy of several consecutive tiles;
//                   completion on mbarriers.  Weight bytes in flight are bounded by the ring, not by
//                   registers.  One lane with a short loop is enough: a lone lane streams 16 KB copies at
//                   the full HBM rate, while several lanes of one warp only take turns, and every
//                   instruction of this warp competes for issue slots with consumer warps that never idle.
//                   Weights are constants, so the first ring fill does not wait for earlier kernels of the stream.
//                   Floating-point path (3..16 tokens, small groups): a stage also gets the activations of its tiles by a
//                   tensor copy, the first ones behind the dependency wait.
//   consumer warps: take tiles round-robin.  Floating-point path: the activations lie in the ring, brought once per CTA,
//                   as deep ahead as the ring, by no instruction or wait of a consumer warp.  (Loaded by the warps, fragments of
//                   the next tile to registers or, with 9..16 tokens, to a buffer of the warp's own, they took 3 to 5 of a warp's 26
//                   thousand cycles and the room of four ring stages: the change alone took 4096x28672 from 16.3 to 15.7 us at
//                   4 tokens, from 17.6 to 15.9 at 8 and from 23.2 to 20.4 at 16.  It is 14.1, 14.1 and 18.5 now.)
//                   Integer path: a lane reads its 4 k of the tile's 128 per token straight from global memory (they
//                   sit in L2), one tile ahead and never before the kernels ahead of this one on the stream have completed.
//                   128-bit shared loads, codes -> exact small-integer bf16
//                   (q - z), contraction with the activations on the warp-level tensor-core MMA
//                   (weights = the 16x16 operand, up to 8 tokens = the 16x8 operand: the per-weight
//                   cost does not grow with M), fp16 scale applied in fp32 once per group.
//
//   reducer warp  : when the consumers finish the tiles of one strip inside this CTA's range they drop
//                   their fp32 partials into shared memory and move on; the reducer adds them up (fixed
//                   order), rounds to bf16 and stores y, so the consumers never wait at a strip boundary.
//   The last segment of a range is on the way of the whole call, and nobody has tiles left: there the consumer warps add up a
//   slice each (two token rows), and those of the CTA that puts a cut strip together fetch the same slice of the others' sums, asked
//   for before they wait for their own.  From the last consumer to the end of the kernel it took 2.2 us (4 tokens, 14336x4096)
//   when the one reducer warp did it, one contributor after the other, and takes 1.0 now: that change alone, us per call, 16 tokens
//   14336x4096 12.8 -> 11.0, 4096x6144 8.7 -> 7.1, 4 tokens 4096x4096 5.1 -> 4.5, 14336x4096 9.8 -> 9.0, 1 and 16 tokens 32768x1024
//   10.1 -> 7.2 and 14.1 -> 9.3.  The integer path has one slice; its reducer does the same, as it has time to look for the
//   others' sums while the consumers work (by a consumer warp 1 token 14336x4096 took 8.4 us where the reducer took 8.2).
//
// A range may cut a strip (64 output columns) in two.  A CTA that holds a whole strip stores y
// directly.  Otherwise its fp32 partial goes to the workspace, and the CTA that has the strip's first tile
// collects the partials in CTA order (see Gather) and stores y, so results are deterministic.  This keeps the
// paper's rule that partial sums do not travel between workers for everything but the (at most two) cut strips of a CTA.
#include <cuda.h>

#include <atomic>
#include <type_traits>

#include "async.cuh"
#include "common.cuh"
#include "kernels.h"
#include "tensormap.h"

namespace tf {

namespace {

// Integer warp MMA: D(16x8, s32) += A(16x32, s8) . B(32x8, s8).  Thread (g, t): a0 = row g, k 4t..4t+3; a1 = row g+8;
// a2, a3 = the same rows, k + 16; b0 = column g, k 4t..4t+3; b1 = k + 16; d = rows g, g+8 x columns 2t, 2t+1.
__device__ __forceinline__ void mma_s8_16832(int d[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// The same with D = A . B + c in every element (no accumulator to set first).
__device__ __forceinline__ void mma_s8_16832_first(int d[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1, int c) {
    asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(c));
}

// The same shapes with unsigned bytes in the 16-row operand (4-bit codes 0..15 as they come out of a packed word).
__device__ __forceinline__ void mma_u8s8_16832(int d[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_u8s8_16832_first(int d[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1, int c) {
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(c));
}

// int -> float for |v| < 2^22 without the conversion unit: the bits of the integer 0x4B400000 + v are the float
// 1.5 * 2^23 + v, exactly.  A tile's sums get the bias as the start of the MMAs' accumulators or with the zero point, and
// (f - 1.5 * 2^23) * c is one fused multiply-add with -1.5 * 2^23 * c.
constexpr int kIntAsFloatBias = 0x4B400000;
constexpr float kIntAsFloatBiasValue = 12582912.0f;

// Even split of `total` tiles (or strips) over the CTAs of a cluster (or the clusters); the grid's own ranges come with the launch.
// 32-bit: the products stay below 2^26 (at most 256 x 512 tiles, K and N <= 32768, times at most 257), and a 64-bit division is several
// times the instructions.  These sit between the start of a CTA and its first weight copy, in the reducer's bookkeeping and in
// the cluster-mode finish.
__device__ __forceinline__ int range_start(int cta, int total, int grid) {
    return static_cast<int>((static_cast<uint32_t>(cta) * static_cast<uint32_t>(total)) / static_cast<uint32_t>(grid));
}
__device__ __forceinline__ int range_owner(int tile, int total, int grid) {
    return static_cast<int>(((static_cast<uint32_t>(tile) + 1u) * static_cast<uint32_t>(grid) - 1u) / static_cast<uint32_t>(total));
}

// The chunks of a tile range [t0, t0 + ntiles): up to kR consecutive tiles of one strip each.  Tiles are stored
// strip after strip, so the source pointer only ever advances.
struct ChunkWalk {
    int left, seg_left, T, ktiles, tile_bytes;
    const uint8_t* src;
    __device__ ChunkWalk(int t0, int ntiles, int ktiles_, const uint8_t* tiles, int tile_bytes_)
        : left(ntiles), ktiles(ktiles_), tile_bytes(tile_bytes_) {
        const int strip = t0 / ktiles;
        T = t0 - strip * ktiles;
        seg_left = min(ntiles, ktiles - T);
        src = tiles + (size_t)t0 * tile_bytes;
    }
    __device__ bool done() const { return left == 0; }
    __device__ void next(int kR, int& tiles_here, int& T_first, const uint8_t*& src_first) {
        tiles_here = min(kR, seg_left);
        T_first = T;
        src_first = src;
        src += (size_t)tiles_here * tile_bytes;
        T += tiles_here;
        seg_left -= tiles_here;
        left -= tiles_here;
        if (seg_left == 0) { T = 0; seg_left = min(left, ktiles); }
    }
};

// A strip's sums are an fp32 tile [token][64 n]; slice e of it is the token rows 2e and 2e + 1, a float4 per lane (row 2e + lane / 16,
// columns 4 (lane % 16) .. + 3).  A slice rounded to bf16 -> y; rows >= M and columns >= N are not written (N % 8 == 0: a
// group of 4 columns is in or out).
__device__ __forceinline__ void store_slice(__nv_bfloat16* y, float4 v, int e, int strip, int M, int N, int lane) {
    const int m = 2 * e + (lane >> 4), n = strip * kTileN + 4 * (lane & 15);
    if (m < M && n < N) {
        uint2 o;
        o.x = pack_bf16(v.x, v.y);
        o.y = pack_bf16(v.z, v.w);
        *reinterpret_cast<uint2*>(y + (size_t)m * N + n) = o;
    }
}
__device__ __forceinline__ void add_to(float4& a, float4 v) { a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w; }

// Hand-over of a cut strip without a fence or a counter.  The partial-sum slots of a workspace are all +0.0 bits
// between calls.  A contributor stores its sums with every +0.0 replaced by -0.0 (the same number), so a word that is
// not +0.0 has arrived, whatever the order in which the memory system delivers the words.  The finisher reads a slot
// until all of its words have arrived, adds it, and puts +0.0 back for the next call.  It waits for stores that were
// issued at about the time it starts to look (every wait is bounded), and the critical path of a cut strip is one
// trip to the L2 instead of three (stores acknowledged -> arrival counter returned -> partial sums loaded).
__device__ __forceinline__ float4 never_plus_zero(float4 v) {
    const uint32_t x = __float_as_uint(v.x), y = __float_as_uint(v.y), z = __float_as_uint(v.z), w = __float_as_uint(v.w);
    return make_float4(__uint_as_float(x == 0u ? 0x80000000u : x), __uint_as_float(y == 0u ? 0x80000000u : y),
                       __uint_as_float(z == 0u ? 0x80000000u : z), __uint_as_float(w == 0u ? 0x80000000u : w));
}
// This lane's float4 of the other contributors' slots (kGemvSlotBytes apart, in CTA order): asked for four contributors at a time,
// one trip to the L2 for all of them, added up in CTA order when all have arrived, and their slots cleared.
struct Gather {
    static constexpr int kSlotVec = kGemvSlotBytes / 16;
    float4* slot;
    int count;                 // contributors still missing
    float4 sum, v[4];
    __device__ __forceinline__ Gather(float4* slot_, int count_) : slot(slot_), count(count_), sum(make_float4(0.f, 0.f, 0.f, 0.f)) {}
    __device__ __forceinline__ void ask() {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            v[b] = make_float4(-0.f, -0.f, -0.f, -0.f);
            if (b < count)                       // a real load every time, from the L2
                asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                             : "=f"(v[b].x), "=f"(v[b].y), "=f"(v[b].z), "=f"(v[b].w) : "l"(slot + b * kSlotVec) : "memory");
        }
    }
    // What was asked for, if all of it has arrived (whole warp).
    __device__ __forceinline__ bool take() {
        bool here = true;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            here = here && __float_as_uint(v[b].x) != 0u && __float_as_uint(v[b].y) != 0u && __float_as_uint(v[b].z) != 0u &&
                   __float_as_uint(v[b].w) != 0u;
        if (!__all_sync(0xFFFFFFFFu, here)) return false;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            add_to(sum, v[b]);
            if (b < count) __stcg(slot + b * kSlotVec, make_float4(0.f, 0.f, 0.f, 0.f));
        }
        slot += 4 * kSlotVec;
        count -= 4;
        return true;
    }
};

}  // namespace

// Integer path: the activation pieces of one k-tile (up to two tokens), from the raw bf16 of lane L (k = 4L .. 4L+3).
// dst: [column][kGemvPieceColWords] piece words, the word of lane L at (L & 3) * 8 + (L >> 2), so that a thread of the
// MMA phase finds the eight k-blocks of its column and k quarter in two 16-byte loads (columns 36 words apart fall
// into different banks).  unit[m]: 2^(emax - 148), what the integers of token m are multiples of.
// KEEP (pieces that serve several tiles): also meta: [column] {unit 256^j, sum of the piece over the tile} in 8-byte entries, a thread's two
// columns = one 16-byte load (with 4-byte entries and an 8-byte load the same kernel ran 12 % slower: measured, cause not established).
constexpr int kGemvPieceColWords = 36;
template <int BITS, bool KEEP>
__device__ __forceinline__ void make_pieces(const uint2 (&raws)[2], uint32_t* dst, uint2* meta, float (&unit)[2], int M, int lane) {
    constexpr int kColWords = kGemvPieceColWords;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        if (m < M) {
            const uint32_t x0 = raws[m].x, x1 = raws[m].y;
            const uint32_t pair = __vmaxu2(x0 & 0x7FFF7FFFu, x1 & 0x7FFF7FFFu);
            const uint32_t e = max(__reduce_max_sync(0xFFFFFFFFu, max(pair >> 16, pair & 0xFFFFu)) >> 7, 22u);      // at least 22: keeps both powers of two normal numbers
            const float mult = __uint_as_float((275u - e) << 23);          // 2^(148 - emax)
            // rint(a mult) = v in the low bits of 1.5 * 2^23 + a mult (no conversion unit), and on to v + 0x808080, whose bytes are p0 + 128,
            // p1 + 128, p2 + 128 of the balanced split (what is left above them is not used)
            const auto biased = [&](uint32_t bits) { return __float_as_uint(fmaf(__uint_as_float(bits), mult, kIntAsFloatBiasValue)) + (0x808080u - 0x400000u); };
            const uint32_t v[4] = {biased(x0 << 16), biased(x0 & 0xFFFF0000u), biased(x1 << 16), biased(x1 & 0xFFFF0000u)};
            // 4 x 3 byte transpose: one word per piece, bytes in the k order of the weight operand's bytes
            // (int8: k, k+1, k+2, k+3; 4-bit: k, k+2, k+1, k+3, the order of a packed word's nibble pairs)
            const uint32_t ab01 = __byte_perm(v[0], v[1], 0x5140), ab2 = __byte_perm(v[0], v[1], 0x0062);
            const uint32_t cd01 = __byte_perm(v[2], v[3], 0x5140), cd2 = __byte_perm(v[2], v[3], 0x0062);
            uint32_t word[3];
            word[0] = __byte_perm(ab01, cd01, BITS == 8 ? 0x5410 : 0x5140) ^ 0x80808080u;
            word[1] = __byte_perm(ab01, cd01, BITS == 8 ? 0x7632 : 0x7362) ^ 0x80808080u;
            word[2] = __byte_perm(ab2, cd2, BITS == 8 ? 0x5410 : 0x5140) ^ 0x80808080u;
            // an Inf or NaN among the 128 activations makes this token's outputs NaN
            unit[m] = e == 255u ? __uint_as_float(0x7FC00000u) : __uint_as_float((e - 21u) << 23);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int c = 3 * m + j;
                dst[c * kColWords + (lane & 3) * 8 + (lane >> 2)] = word[j];
                if constexpr (KEEP) {
                    const int psum = __reduce_add_sync(0xFFFFFFFFu, __dp4a((int)word[j], 0x01010101, 0));
                    if (lane == 0) meta[c] = make_uint2(__float_as_uint(unit[m] * (j == 0 ? 1.f : j == 1 ? 256.f : 65536.f)), (uint32_t)psum);
                }
            }
        }
    }
    if (KEEP && lane == 0) {                            // columns without a token contribute nothing
#pragma unroll
        for (int c = 3; c < 8; ++c)
            if (c >= 3 * M) meta[c] = make_uint2(0u, 0u);
    }
}
// The same as a call: where pieces are prepared on the first visit of a k-tile only, the code stays out of the tile
// loop's register allocation.
template <int BITS>
__device__ __noinline__ void make_pieces_call(const uint2 (&raws)[2], uint32_t* dst, uint2* meta, int M, int lane) {
    float unit[2];
    make_pieces<BITS, true>(raws, dst, meta, unit, M, lane);
}

// Floating-point path: token g + 8 mt, k = 16 kb + 4t .. +3 of a tile's activations in the ring.  The 16-byte units of a row are
// permuted by the swizzle: two wavefronts for 256 bytes.
template <int MT>
__device__ __forceinline__ uint2 act_fragment(const uint8_t* acts, int g, int t, int kb, int mt) {
    return *reinterpret_cast<const uint2*>(acts + (kb >> 2) * (1024 * MT) + (g + 8 * mt) * 128 + (((2 * (kb & 3) + (t >> 1)) ^ g) << 4) + (t & 1) * 8);
}

// G = groups per tile: 1 for group sizes that are multiples of 128, 2 / 4 for the 4-bit group sizes 64 / 32.
// I8 = 0: floating-point path; 1: integer path, a consumer warp prepares the activation pieces of every tile it works
// on; 2: integer path for ranges that pass over the same k-tiles more than once, with K a multiple of 128 times the
// number of consumer warps: a warp then meets the same k-tiles on every pass, prepares the pieces of a k-tile on its
// first visit and keeps them (piece table, one entry per k-tile, each entry written and read by one warp only).
struct NoActMap {};
template <int I8> using GemvActMap = std::conditional_t<I8 == 0, CUtensorMap, NoActMap>;      // floating-point path: [K / 64][M][64] activations
template <int BITS, int MT, bool FULL, bool CL, int I8, int G = 1>
__global__ void __launch_bounds__(gemv_max_threads(BITS, MT, FULL, I8 != 0), FULL ? 1 : 2)
gemv_stream_kernel(const __grid_constant__ GemvActMap<I8> act_map, const uint8_t* __restrict__ blob, const __nv_bfloat16* a_glob,
                   __nv_bfloat16* __restrict__ y, int M, int K, int N, int ktiles, int total_tiles, int nstages, int stage_bytes,
                   int csize, int nclusters, const Ranges ranges, int xslot_bytes, int nred, int piece_tab,
                   uint8_t* __restrict__ workspace, uint32_t debug) {
    static_assert(G == 1 || (BITS == 4 && !I8 && !CL && FULL), "several groups per tile: 4-bit, floating-point path, whole SM");
    static_assert((FULL || I8) && (!CL || MT == 2) && (I8 != 2 || BITS == 4), "forms that plan_gemv never chooses");
    constexpr int kTileBytes = tile_bytes(BITS, G);
    constexpr int kWeightBytes = BITS == 4 ? kW4WeightBytes : kW8WeightBytes;
    constexpr int kR = gemv_chunk_tiles(BITS);            // tiles per bulk copy / ring stage
    constexpr int kTok = 8 * MT;
    constexpr int kVecPerKb = BITS == 4 ? 1 : 2;
    constexpr int kRedWarp = (I8 ? 2 : kTok) * kTileN;    // floats one consumer warp drops per strip segment (integer path: two token rows)

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_shared(smem_raw);
    // layout: barriers + flags (kGemvBarrierBytes) | red [consumers][kTok][64] fp32 | ring (1024-aligned stages)
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + (2 * kGemvMaxStages + 4) * 8);
    // stage_tag[s] = index of the chunk whose copies were last issued into ring stage s.  A consumer warp does
    // not touch every use of a stage, so the parity of the stage's mbarrier alone could alias (a warp two uses
    // ahead would see "parity differs" and run on old data); it first waits for its own chunk's tag.
    volatile uint32_t* stage_tag = reinterpret_cast<volatile uint32_t*>(smem + 1024);
    const int nconsumers = (blockDim.x >> 5) - 2;
    float* red = reinterpret_cast<float*>(smem + kGemvBarrierBytes);
    // xred [csize][xslot]: in cluster mode, the partials other CTAs of the cluster send to the finisher of a strip
    uint8_t* xred = smem + kGemvBarrierBytes + nred * nconsumers * kRedWarp * 4;
    // pscr: integer path.  [consumers][1 KB], a warp's activation pieces of the tile it works on; or
    // [piece_tab][kGemvPieceEntryBytes per token], the pieces of every k-tile of the CTA's range
    uint32_t* pscr = reinterpret_cast<uint32_t*>(xred + ((CL ? csize * xslot_bytes : 0) + 1023) / 1024 * 1024);
    // abuf [stages][kR][gemv_act_tile_bytes(MT)]: floating-point path, the activations of the tiles in the ring
    uint8_t* abuf = reinterpret_cast<uint8_t*>(pscr) + (I8 == 2 ? (piece_tab * kGemvPieceEntryBytes * M + 1023) / 1024 * 1024 : I8 == 1 ? nconsumers * 1024 : 0);
    constexpr uint32_t kActStageBytes = I8 == 0 ? kR * gemv_act_tile_bytes(MT) : 0;
    uint8_t* ring = abuf + nstages * kActStageBytes;

    // (the shuffle tells the compiler that the warp number is uniform in the warp)
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int cta = blockIdx.x;
    // "Contributor space": the CTAs that split one pool of tiles evenly among themselves.  Global mode: all CTAs
    // of the grid over all tiles.  Cluster mode: the CTAs of one cluster over the whole strips that cluster owns,
    // so that a strip is only ever shared inside a cluster and can be summed through distributed shared memory.
    // In global mode `nclusters` carries the number of CTAs that take part (the first ones of the grid); the rest
    // of the grid has no tiles and only keeps one CTA of this kernel on every SM (see plan_gemv).
    int cn = nclusters, crank = cta, cbase = 0, ctiles = total_tiles;
    if (CL) {
        const int q = cta / csize, strips = total_tiles / ktiles;
        const int s0 = range_start(q, strips, nclusters), s1 = range_start(q + 1, strips, nclusters);
        cn = csize; crank = cta - q * csize; cbase = s0 * ktiles; ctiles = (s1 - s0) * ktiles;
    }
    const bool idle = crank >= cn;
    auto start_of = [&](int c) { return CL ? range_start(c, ctiles, cn) : ranges.start(c); };
    auto owner_of = [&](int tile) { return CL ? range_owner(tile, ctiles, cn) : ranges.owner(tile); };
    const int t0 = idle ? 0 : cbase + start_of(crank);
    const int ntiles = idle ? 0 : cbase + start_of(crank + 1) - t0;

    DeviceStatus* status = reinterpret_cast<DeviceStatus*>(workspace);
    float* partials = reinterpret_cast<float*>(workspace + kGemvPartialOffset);

    HeaderWords header(blob);

    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kGemvMaxStages);
    const uint32_t seg_full0 = smem_u32(bars + 2 * kGemvMaxStages), seg_free0 = seg_full0 + 16;
    // Integer path: the lane that issues the weight copies initialises the barriers of the ring itself, while the header of the blob is on
    // its way, and issues the first chunk ahead of the barrier that the others meet at (packed weights are constants; 1 token 4096x4096
    // 4.24 -> 4.00 us.  On the floating-point path it changed nothing.)
    ChunkWalk early(t0, I8 != 0 ? ntiles : 0, ktiles, blob + kHeaderBytes, kTileBytes);
    int issued = 0;                                     // chunks
    auto issue_weights = [&](ChunkWalk& walk, int c) {
        int tiles_here, T;
        const uint8_t* src;
        walk.next(kR, tiles_here, T, src);
        stage_tag[c] = (uint32_t)c;
        mbar_arrive_expect_tx(full0 + 8 * c, (uint32_t)tiles_here * kTileBytes + kActStageBytes);
        bulk_copy_g2s(smem_u32(ring + (size_t)c * stage_bytes), src, (uint32_t)tiles_here * kTileBytes, full0 + 8 * c);
    };
    if (I8 != 0 && threadIdx.x == 0) {
        for (int s = 0; s < nstages; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, kR);
            stage_tag[s] = 0xFFFFFFFFu;
        }
        mbar_init_fence();
        if (header.fit(BITS, (uint32_t)K, (uint32_t)N, G) && (debug & kDebugDropWeights) == 0 && !early.done()) issue_weights(early, issued++);
    }
    // One thread per ring stage, one more for the rest: the set-up sits between the start of a CTA and its first
    // weight copy (one thread doing all of it in turn cost the decode step 1.7 us).
    if (I8 == 0 && threadIdx.x < (unsigned)nstages) {
        const int s = threadIdx.x;
        mbar_init(full0 + 8 * s, 1);
        mbar_init(empty0 + 8 * s, kR);           // every tile of a chunk is released by its consumer warp
        stage_tag[s] = 0xFFFFFFFFu;
        mbar_init_fence();
    } else if (threadIdx.x == 64) {
        for (int b = 0; b < 2; ++b) {                   // one pair per partial-sum buffer (nred = 1 or 2)
            mbar_init(seg_full0 + 8 * b, nconsumers);   // every consumer warp has dropped its partial
            mbar_init(seg_free0 + 8 * b, 1);            // the reducer has read them
        }
        abort_flag[0] = 0;
        abort_flag[1] = wait_limit_kcycles(debug);
        mbar_init_fence();
    }
    __syncthreads();
    const bool header_ok = header.fit(BITS, (uint32_t)K, (uint32_t)N, G);
    // Programmatic dependent launch: the next kernel on the stream may start as SMs free up.  In this kernel
    // only the packed weights (constants) are read before grid_dependency_wait(): the producer lane waits before it copies activations,
    // every consumer warp waits before its first activation load, the reducer warp before it touches y or the
    // workspace, thread 0 before it writes the status word.  (What keeps two half-SM CTAs of one GEMV off the same
    // SM when they come in behind a whole-SM kernel is decided at launch: see launch_one.)
    grid_launch_dependents();

    // The sums of slice e of a cut strip, to the CTA that puts it together.  Cluster mode: to that CTA's shared memory (`to`; maybe this
    // one's), where it adds the slots up in rank order after the cluster barrier at the end of the kernel.  Global mode: to this
    // CTA's slot of the workspace, with no fence and no counter: the data says by itself that it has arrived.
    constexpr int kVec = (I8 ? 2 : kTok) / 2;             // slices of a strip
    auto hand_over = [&](float4 v, int e, int to) {
        if (CL) {
            const uint32_t slot = map_to_cta(smem_u32(xred + (size_t)crank * xslot_bytes), (uint32_t)to);
            asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(slot + (32 * e + lane) * 16),
                         "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
        } else {
            __stcg(reinterpret_cast<float4*>(partials + (size_t)crank * (kGemvMaxM * kTileN)) + 32 * e + lane, never_plus_zero(v));
        }
    };

    // The last segment of the range: its strip, and who has the strip's first and last tile.  Global mode: the CTA that holds the
    // strip's first tile puts a cut strip together.  Its part of the strip is the tail of its range; for every other contributor
    // the strip is the head of the range, done early, or all of it.
    struct Last { int strip, first, last; bool whole; };
    auto last_segment = [&]() {
        Last l;
        l.strip = (t0 + max(ntiles, 1) - 1) / ktiles;
        l.whole = t0 <= l.strip * ktiles && t0 + ntiles == (l.strip + 1) * ktiles;
        l.first = owner_of(l.strip * ktiles - cbase);
        l.last = owner_of(l.strip * ktiles + ktiles - 1 - cbase);
        return l;
    };
    // Where this lane's float4 of slice e lies among the 32 of the slice: on the floating-point path the four-column units of a token row are
    // permuted by the row's pair, because the four threads of a warp that write one column of eight tokens would otherwise meet in a bank: at
    // the end of a call eight warps write at once, 1024 wavefronts at 16 tokens, 256 this way (16 tokens 4096x1024 4.37 -> 4.00 us,
    // 4096x28672 18.5 -> 17.6, 4 tokens 4096x1024 3.19 -> 3.07, 4096x14336 8.65 -> 8.42).
    auto red_lane = [&](int e) { return I8 ? lane : lane ^ (2 * (e & 3)); };
    // One warp's part in it: slice e, from buffer rb in its use ru.  What other CTAs hold of a cut strip is asked for before the wait
    // for this CTA's own sums, by a warp that has nothing else to do (`poll`) again and again.
    auto finish = [&](const Last& l, int e, int rb, int ru, bool poll) {
        const bool finisher = !CL && !l.whole && l.first == crank;
        Gather others(reinterpret_cast<float4*>(partials + (size_t)(crank + 1) * (kGemvMaxM * kTileN)) + 32 * e + lane, finisher ? l.last - crank : 0);
        const uint32_t bar = seg_full0 + 8 * rb;
        if (others.count > 0) others.ask();
        if (poll) {
            const long long t_begin = clock64();
            while (others.count > 0) {
                const bool taken = others.take();
                if (!taken && __all_sync(0xFFFFFFFFu, mbar_test(bar, ru & 1))) break;
                if (!taken && wait_given_up(t_begin, abort_flag, 0x430)) return;
                if (others.count > 0) others.ask();
            }
        }
        if (!mbar_wait_warp(bar, ru & 1, abort_flag, 0x410)) return;
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4* src = reinterpret_cast<const float4*>(red + (size_t)rb * nconsumers * kRedWarp) + 32 * e + red_lane(e);
#pragma unroll 4
        for (int w = 0; w < nconsumers; ++w) add_to(sum, src[w * (kRedWarp / 4)]);         // fixed order: warp 0 + warp 1 + ...
        if (!l.whole && !finisher) {
            hand_over(sum, e, l.last);
            return;
        }
        const long long t_begin = clock64();
        while (others.count > 0)
            if (!others.take() && wait_given_up(t_begin, abort_flag, 0x440)) return;
            else if (others.count > 0) others.ask();
        add_to(sum, others.sum);                            // fixed order: the other contributors in CTA order, then this CTA
        store_slice(y, sum, e, l.strip, M, N, lane);
    };

    if (warp == 0) {
        // ---------------- producer: stream this CTA's contiguous tile range through the ring --------------
        // One lane issues, per chunk, one bulk copy of up to kR contiguous tiles of one strip.  Chunks never straddle
        // a strip boundary.  The loop is kept to a few dozen instructions per chunk: this warp shares its scheduler
        // with consumer warps that never idle.  The packed weights are constants: the first ring fill of them does not
        // wait for the kernels before this one and is on its way while they finish.
        if (lane == 0 && header_ok && (debug & kDebugDropWeights) == 0) {
            ChunkWalk walk = I8 != 0 ? early : ChunkWalk(t0, ntiles, ktiles, blob + kHeaderBytes, kTileBytes);
            // first ring fill, weights only: they are constants, so they may be fetched before the dependency wait
            if constexpr (I8 == 0) prefetch_tensormap(&act_map);
            int cg = issued;
            for (; cg < nstages && !walk.done(); ++cg) issue_weights(walk, cg);
            if constexpr (I8 == 0) {                             // the activations of that first fill
                grid_dependency_wait();
                ChunkWalk first(t0, ntiles, ktiles, blob, kTileBytes);
                for (int c = 0; c < cg; ++c) {
                    int tiles_here, T;
                    const uint8_t* src;
                    first.next(kR, tiles_here, T, src);
                    tma_load_3d(smem_u32(abuf + c * kActStageBytes), &act_map, 0, 0, 2 * T, full0 + 8 * c);
                }
            }
            // everything else in ring order
            int s = 0;
            uint32_t parity = 0;
            for (; !walk.done(); ++cg) {
                if (!mbar_wait(empty0 + 8 * s, parity, abort_flag, 0x100 + s)) break;
                int tiles_here, T;
                const uint8_t* src;
                walk.next(kR, tiles_here, T, src);
                const uint32_t dst = smem_u32(ring + (size_t)s * stage_bytes);
                stage_tag[s] = (uint32_t)cg;                 // the stage's previous use is fully consumed by now
                mbar_arrive_expect_tx(full0 + 8 * s, (uint32_t)tiles_here * kTileBytes + kActStageBytes);
                bulk_copy_g2s(dst, src, (uint32_t)tiles_here * kTileBytes, full0 + 8 * s);
                if constexpr (I8 == 0) tma_load_3d(smem_u32(abuf + s * kActStageBytes), &act_map, 0, 0, 2 * T, full0 + 8 * s);
                if (++s == nstages) { s = 0; parity ^= 1u; }
            }
        }
    } else if (warp == 1) {
        // ---------------- reducer: one strip segment at a time, behind the consumers, but for the last one ------------------
        // (The consumer warps put the last segment of the range together themselves: they have nothing else to do then.)
        if (header_ok) {
            int sidx = 0, i = 0;
            const Last last = I8 ? last_segment() : Last();
            grid_dependency_wait();                    // y and the partial sums belong to earlier kernels until now
            while (i + ktiles - (t0 + i) % ktiles < ntiles) {
                const int strip = (t0 + i) / ktiles, seg_len = ktiles - (t0 + i) % ktiles;
                // segment sidx goes through buffer sidx % nred, in that buffer's use number sidx / nred
                const int rb = nred == 2 ? (sidx & 1) : 0, ru = nred == 2 ? (sidx >> 1) : sidx;
                if (!mbar_wait_warp(seg_full0 + 8 * rb, ru & 1, abort_flag, 0x400)) break;
                float4 sum[kVec];
#pragma unroll
                for (int e = 0; e < kVec; ++e) sum[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                // partial of warp 0 + warp 1 + ... (fixed order); rows of tokens >= M hold zeros.  (A run-time bound on the row pairs made
                // this slower: 36.7 against 35.7 us over four shapes at 4 tokens.)
#pragma unroll 4
                for (int w = 0; w < nconsumers; ++w) {
                    const float4* src = reinterpret_cast<const float4*>(red + (size_t)(rb * nconsumers + w) * kRedWarp);
#pragma unroll
                    for (int e = 0; e < kVec; ++e) add_to(sum[e], src[32 * e + red_lane(e)]);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(seg_free0 + 8 * rb);         // consumers may reuse the buffer

                // A segment that ends its strip is the whole strip or, for the first one, its end: then the sums go to the CTA that
                // puts the strip together.
                if (seg_len == ktiles) {
#pragma unroll
                    for (int e = 0; e < kVec; ++e) store_slice(y, sum[e], e, strip, M, N, lane);
                } else {
#pragma unroll
                    for (int e = 0; e < kVec; ++e)
                        if (2 * e < M) hand_over(sum[e], e, crank);
                }
                i += seg_len;
                ++sidx;
            }
            if (I8 && i < ntiles) finish(last, 0, nred == 2 ? (sidx & 1) : 0, nred == 2 ? (sidx >> 1) : sidx, true);
        }
    } else if (header_ok) {
        // ---------------- consumers ---------------------------------------------------------------------------
        const int cw = warp - 2;
        const int g = lane >> 2, t = lane & 3;
        bool aborted = false;

        int i = 0, sidx = 0, chunk_base = 0;
        int cg_cur = 0, s_cur = 0, use_cur = 0;         // this warp's position in the ring (chunks only move forward)
        // This warp's tiles are the local indices cw, cw + nconsumers, ... of the CTA's range, whatever strip they
        // fall into.  Integer path: this lane's four k per token of the warp's NEXT tile are requested from global memory
        // while it works on the current one.  They are written by earlier kernels of the stream, so nothing is read
        // before the dependency wait.
        uint2 araw[2];                                  // integer path: token m, k = 128 T + 4 lane .. +3
        int T_act = (t0 + cw) % ktiles;                 // k-tile index of this warp's current tile (one division per kernel)
        auto load_araw = [&](const __nv_bfloat16* base) {
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                araw[m] = make_uint2(0u, 0u);
                if (m < M) araw[m] = load_behind_wait(reinterpret_cast<const uint2*>(base + (size_t)m * K + 4 * lane));
            }
        };
        constexpr int kColWords = kGemvPieceColWords;
        // Piece table (I8 == 2): local tile j of the range finds its pieces in entry j mod piece_n, piece_n =
        // min(ntiles, ktiles); j < piece_n is the first visit of that k-tile.  ktiles is a multiple of the number of
        // consumer warps, so tiles j and j + ktiles belong to the same warp: no warp reads another warp's entry.
        const int piece_entry_words = (kGemvPieceEntryBytes / 4) * M;
        const int piece_n = min(ntiles, ktiles);
        const int T_first = t0 % ktiles;                // k-tile index of the range's first tile
        int piece_e = cw;                               // entry of this warp's next tile (cw < piece_n whenever it has one)
        // (worked out here, ahead of the wait, or at the end where that costs the tile loop registers: 16 tokens 14336x4096 11.04 us at the
        // end, 11.22 here; 10 tokens, group 64, 7424x18440 21.6 and 21.0; 4 tokens 4096x4096 4.57 and 4.50)
        constexpr bool kLastAtEnd = MT == 2 && G == 1;
        Last last;
        if (!I8 && !kLastAtEnd) last = last_segment();
        // Everything above touches registers and this CTA's shared memory only; from here on the warp reads activations, or
        // waits for them in the ring (the limit of that wait must not run while earlier kernels do).
        grid_dependency_wait();                         // the activations belong to earlier kernels until now
        if (I8 != 0 && cw < ntiles) load_araw(a_glob + (size_t)T_act * kTileK);
        // powers of 256 by which the pieces of this thread's columns 2t and 2t + 1 count (0: a column without a token)
        const float pow_x = t == 0 ? 1.f : t == 1 ? 65536.f : t == 2 && M == 2 ? 256.f : 0.f;
        const float pow_y = t == 0 ? 256.f : M == 1 ? 0.f : t == 1 ? 1.f : t == 2 ? 65536.f : 0.f;
        int T0 = T_first;                               // k-tile index at which the current segment starts (0 after the first)
        int j = cw;                                     // this warp's next tile, as a local index of the CTA's range
        while (i < ntiles && !aborted) {
            const int seg_len = min(ntiles - i, ktiles - T0);
            T0 = 0;

            float acc[4][MT][4];
#pragma unroll
            for (int w = 0; w < 4; ++w)
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[w][mt][e] = 0.f;

            // the warp's tiles come every nconsumers-th tile of the range, whatever segment they fall into
            // Find a tile of this segment in the ring, wait until it has landed and fetch the metadata of its first
            // group.  Called once per tile, in order (the ring position only moves forward).  (Calling it for the next
            // tile already before the current tile's scales are applied, so that the wait would run under the tail of
            // the current tile, was measured slower: 36.9 against 35.8 us over the four shapes at 4 tokens, 53.4 against
            // 52.3 at 16.)
            const uint8_t* nx_tile = nullptr;
            int nx_s = 0, nx_slot = 0, nx_cl = 0;
            uint4 nx_sc = make_uint4(0u, 0u, 0u, 0u);
            uint32_t nx_zw = 0u;
            auto locate_and_wait = [&](int jj) -> bool {
                const int lj = jj - i, cl = lj / kR, slot = lj - cl * kR;
                const int cg = chunk_base + cl;
                s_cur += cg - cg_cur;
                cg_cur = cg;
                while (s_cur >= nstages) { s_cur -= nstages; ++use_cur; }
                const int s = s_cur;
                // (the tag and then the barrier, both asked for before either answer is looked at: what is seen of the barrier
                // is later than the tag, so it is about this chunk if the tag is this chunk's.  One vote and one trip to shared memory
                // per tile instead of two: a pass over four layer shapes at 1 / 4 / 16 tokens 31.2 / 34.3 / 44.1 -> 30.9 / 34.1 / 43.8 us)
                const bool tagged = stage_tag[s] == (uint32_t)cg, landed = mbar_try_wait(full0 + 8 * s, use_cur & 1);
                if (!__all_sync(0xFFFFFFFFu, tagged && landed)) {
                    const long long t_begin = clock64();
                    while (!__all_sync(0xFFFFFFFFu, stage_tag[s] == (uint32_t)cg))      // the producer has not reached this chunk yet
                        if (wait_given_up(t_begin, abort_flag, 0x280 + s)) return false;
                    if (!mbar_wait_warp(full0 + 8 * s, use_cur & 1, abort_flag, 0x200 + s)) return false;
                }
                nx_tile = ring + (size_t)s * stage_bytes + (size_t)slot * kTileBytes;
                nx_s = s; nx_slot = slot; nx_cl = cl;
                if constexpr (!I8) {
                    nx_sc = *(reinterpret_cast<const uint4*>(nx_tile + kWeightBytes) + g);
                    if (BITS == 4) nx_zw = *(reinterpret_cast<const uint32_t*>(nx_tile + w4_zero_offset(G, 0)) + g);
                }
                return true;
            };
            for (; j < i + seg_len; j += nconsumers) {
                if (!locate_and_wait(j)) { aborted = true; break; }
                const uint8_t* tile = nx_tile;
                const int s = nx_s, slot = nx_slot, cl = nx_cl;
                const uint4 sc_first = nx_sc;
                const uint32_t zw_first = nx_zw;
                const bool has_next = j + nconsumers < ntiles;
                int T_nx = T_act + nconsumers;                  // the warp's next tile is nconsumers tiles further along K
                while (T_nx >= ktiles) T_nx -= ktiles;
                T_act = T_nx;
                const __nv_bfloat16* next_base = a_glob + (size_t)T_nx * kTileK;
                if constexpr (I8) {
                    const uint4 sc = *(reinterpret_cast<const uint4*>(tile + kWeightBytes) + g);
                    // ---- integer path (1 or 2 tokens): codes x activation pieces on the integer warp MMA ----
                    // The 128 activations of a (token, k-tile) are scaled by 2^(148 - emax) (emax = largest biased
                    // exponent among them), rounded to integers |v| < 2^22 and split into signed bytes
                    // v = p0 + 256 p1 + 65536 p2: values within 2^14 of the largest are exact, smaller ones are rounded
                    // at 2^-22 of it.  Piece j of token m is column 3m + j of the MMA's 8-column operand; the codes are
                    // the other operand as they are (int8), or after two ANDs per packed word (4-bit: the low nibbles of a
                    // word are this lane's row g, the high nibbles, left in place as 16 q, its row g + 8, as unsigned bytes),
                    // so no weight is ever converted to floating point:
                    //     D[n][3m+j] = sum_k q[k][n] p_j[m][k]            (exact, 32-bit integers)
                    //     4-bit: D[n][3m+j] -= z[n] sum_k p_j[m][k]       (the zero point of Eq. 2, still exact)
                    //     y[m][n] += s[n] 2^(emax-148) sum_j 256^j D[n][3m+j]
                    static_assert(!I8 || MT == 1, "the integer path is built for up to 2 tokens");
                    const uint32_t* scr;                                // this tile's piece words and column metadata
                    float2 col_scale;
                    int p0 = 0, p1 = 0;                                 // sums of the pieces of this thread's columns over the tile's 128 k
                    if constexpr (I8 == 2) {
                        uint32_t* ent = pscr + piece_e * piece_entry_words;
                        uint2* ent_meta = reinterpret_cast<uint2*>(ent + 3 * kColWords * M);
                        piece_e += nconsumers;                          // the warp's next tile is nconsumers k-tiles further
                        while (piece_e >= piece_n) piece_e -= piece_n;
                        if (j < piece_n) {                              // first visit of this k-tile
                            // (as a call in the whole-SM form with its 96 registers: inlined it spilled inside the tile loop,
                            // 17.8 against 17.1 us on 1x4096x32768; inlined in the half-SM form, where the call was the
                            // slower one, 12.0 against 10.9 us on 1x4096x14336)
                            float unit[2];
                            if constexpr (FULL) make_pieces_call<BITS>(araw, ent, ent_meta, M, lane);
                            else make_pieces<BITS, true>(araw, ent, ent_meta, unit, M, lane);
                            if (j + nconsumers < piece_n) load_araw(next_base);    // later visits need no activations
                            __syncwarp();
                        }
                        scr = ent;
                        const uint4 cm = *reinterpret_cast<const uint4*>(ent_meta + 2 * t);
                        col_scale = make_float2(__uint_as_float(cm.x), __uint_as_float(cm.z));
                        p0 = (int)cm.y; p1 = (int)cm.w;
                    } else {
                        uint32_t* mine_scr = pscr + cw * 256;
                        float unit[2] = {0.f, 0.f};
                        make_pieces<BITS, false>(araw, mine_scr, nullptr, unit, M, lane);
                        scr = mine_scr;
                        col_scale = make_float2((t >= 2 ? unit[1] : unit[0]) * pow_x, (t >= 1 ? unit[1] : unit[0]) * pow_y);
                        if (has_next) load_araw(next_base);             // the next tile's activations, under this tile's MMAs
                        __syncwarp();
                    }
                    uint32_t bw[8];                                     // column g: the words of k-blocks 0..7 for this t
#pragma unroll
                    for (int i = 0; i < 8; ++i) bw[i] = 0u;
                    if (g < 3 * M) {
                        const uint4 lo = *reinterpret_cast<const uint4*>(scr + g * kColWords + t * 8);
                        const uint4 hi = *reinterpret_cast<const uint4*>(scr + g * kColWords + t * 8 + 4);
                        bw[0] = lo.x; bw[1] = lo.y; bw[2] = lo.z; bw[3] = lo.w;
                        bw[4] = hi.x; bw[5] = hi.y; bw[6] = hi.z; bw[7] = hi.w;
                    }
                    if constexpr (I8 == 1) __syncwarp();                // the scratch is rewritten for the next tile
                    // 4-bit: one AND per packed word instead of two, no accumulator to set first, one addition per sum more, and a byte times a
                    // piece summed over 128 k still stays below 2^22.  1 token 14336x4096 8.04 -> 7.85 us, 2 tokens 4096x4096 4.42 -> 4.01
                    // (both with the piece sums by MMA, below).  Not in the half-SM form with kept pieces, whose 96 registers it overflows:
                    // 4096x28672 12.85 us without, 13.1 with it.
                    constexpr bool kWholeBytes = FULL || I8 == 1;
                    int d[4][4];
                    if constexpr (BITS == 4) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {                   // 32 k per MMA: k-blocks 2i and 2i+1, one packed word each
                            const uint4 v0 = *reinterpret_cast<const uint4*>(tile + ((size_t)(2 * i) * 32 + lane) * 16);
                            const uint4 v1 = *reinterpret_cast<const uint4*>(tile + ((size_t)(2 * i + 1) * 32 + lane) * 16);
#pragma unroll
                            for (int w = 0; w < 4; ++w) {
                                const uint32_t x0 = w == 0 ? v0.x : w == 1 ? v0.y : w == 2 ? v0.z : v0.w;
                                const uint32_t x1 = w == 0 ? v1.x : w == 1 ? v1.y : w == 2 ? v1.z : v1.w;
                                // Row g: the low nibbles.  Row g + 8: the high nibbles, left in place: the row carries 16 q, its sums come
                                // out 16 times too large and its scale is taken 16 times smaller below (all exact).  With kWholeBytes
                                // the whole bytes, 16 q + row g's code, and row g's sum is taken off again below.
                                const uint32_t a0 = x0 & 0x0F0F0F0Fu, a1 = kWholeBytes ? x0 : x0 & 0xF0F0F0F0u;            // k-block 2i
                                const uint32_t a2 = x1 & 0x0F0F0F0Fu, a3 = kWholeBytes ? x1 : x1 & 0xF0F0F0F0u;            // k-block 2i + 1
                                if (i == 0) mma_u8s8_16832_first(d[w], a0, a1, a2, a3, bw[0], bw[1], kWholeBytes ? 0 : kIntAsFloatBias);
                                else mma_u8s8_16832(d[w], a0, a1, a2, a3, bw[2 * i], bw[2 * i + 1]);
                            }
                        }
                    } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {                       // 32 k per MMA: k-blocks 2i and 2i+1
                        uint4 wv[2][2];
#pragma unroll
                        for (int hb = 0; hb < 2; ++hb)
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                wv[hb][h] = *reinterpret_cast<const uint4*>(tile + ((size_t)((2 * i + hb) * 2 + h) * 32 + lane) * 16);
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            uint32_t a[4];
#pragma unroll
                            for (int hb = 0; hb < 2; ++hb) {
                                const uint4 v = wv[hb][w >> 1];
                                const uint32_t w0 = (w & 1) ? v.z : v.x, w1 = (w & 1) ? v.w : v.y;
                                a[2 * hb] = __byte_perm(w0, w1, 0x5410);         // row g,   k 0..3 of this thread
                                a[2 * hb + 1] = __byte_perm(w0, w1, 0x7632);     // row g+8
                            }
                            if (i == 0) mma_s8_16832_first(d[w], a[0], a[1], a[2], a[3], bw[0], bw[1], kIntAsFloatBias);
                            else mma_s8_16832(d[w], a[0], a[1], a[2], a[3], bw[2 * i], bw[2 * i + 1]);
                        }
                    }
                    }
                    if constexpr (BITS == 4) {
                        if constexpr (I8 == 1) {                        // a row of ones times the same operand (four MMAs instead of three reductions over the warp)
                            int ones[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                if (i == 0) mma_u8s8_16832_first(ones, 0x01010101u, 0u, 0x01010101u, 0u, bw[0], bw[1], 0);
                                else mma_u8s8_16832(ones, 0x01010101u, 0u, 0x01010101u, 0u, bw[2 * i], bw[2 * i + 1]);
                            }
                            p0 = ones[0]; p1 = ones[1];
                        }
                        // zero point: every code of row n stands for q - z[n], so the row's sum loses z[n] times the column's piece sum
                        const uint32_t zword = *(reinterpret_cast<const uint32_t*>(tile + kWeightBytes + kScaleBytes) + g);
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            const int zr = (int)((zword >> (4 * w)) & 15u), zr8 = (int)((zword >> (4 * w + 12)) & 0xF0u);     // z, 16 z
                            if constexpr (kWholeBytes) {
                                d[w][2] += (kIntAsFloatBias - zr8 * p0) - d[w][0]; d[w][3] += (kIntAsFloatBias - zr8 * p1) - d[w][1];
                                d[w][0] += kIntAsFloatBias - zr * p0; d[w][1] += kIntAsFloatBias - zr * p1;
                            } else {
                                d[w][0] -= zr * p0; d[w][1] -= zr * p1;
                                d[w][2] -= zr8 * p0; d[w][3] -= zr8 * p1;
                            }
                        }
                    }
                    __syncwarp();
                    if (lane == 0) {
                        const int tiles_here = min(kR, seg_len - cl * kR);
                        mbar_arrive_n(empty0 + 8 * s, slot == tiles_here - 1 ? (uint32_t)(kR - tiles_here + 1) : 1u);
                    }
                    const uint32_t sw[4] = {sc.x, sc.y, sc.z, sc.w};
                    // d holds the bits of 1.5 * 2^23 + D: (that - 1.5 * 2^23) * column scale is one exact fused multiply-add
                    const float off_x = -kIntAsFloatBiasValue * col_scale.x, off_y = -kIntAsFloatBiasValue * col_scale.y;
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        const float s_g = fp16_bits_to_float((uint16_t)(sw[w] & 0xFFFFu));
                        const float s_g8 = fp16_bits_to_float((uint16_t)(sw[w] >> 16)) * (BITS == 4 ? 0.0625f : 1.f);     // 4-bit: row g + 8 holds 16 (q - z)
                        acc[w][0][0] = fmaf(fmaf(__int_as_float(d[w][0]), col_scale.x, off_x), s_g, acc[w][0][0]);
                        acc[w][0][1] = fmaf(fmaf(__int_as_float(d[w][1]), col_scale.y, off_y), s_g, acc[w][0][1]);
                        acc[w][0][2] = fmaf(fmaf(__int_as_float(d[w][2]), col_scale.x, off_x), s_g8, acc[w][0][2]);
                        acc[w][0][3] = fmaf(fmaf(__int_as_float(d[w][3]), col_scale.y, off_y), s_g8, acc[w][0][3]);
                    }
                } else {
                // ---- floating-point path: group after group (one group per tile unless the group size is 64 or 32) ----
                const uint8_t* acts = abuf + s * kActStageBytes + slot * gemv_act_tile_bytes(MT);
#pragma unroll
                for (int gr = 0; gr < G; ++gr) {
                    uint4 sc = sc_first;
                    uint32_t zword = zw_first;
                    if (gr > 0) {
                        sc = *(reinterpret_cast<const uint4*>(tile + kWeightBytes + gr * kScaleBytes) + g);
                        if (BITS == 4) zword = *(reinterpret_cast<const uint32_t*>(tile + w4_zero_offset(G, gr)) + g);
                    }
                    uint32_t zg[4], zg8[4];
                    if (BITS == 4)
#pragma unroll
                        for (int w = 0; w < 4; ++w) w4_minus_zero(zword, w, zg[w], zg8[w]);
                    float gacc[4][MT][4];
#pragma unroll
                    for (int w = 0; w < 4; ++w)
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                            for (int e = 0; e < 4; ++e) gacc[w][mt][e] = 0.f;

#pragma unroll
                    for (int kb = gr * (8 / G); kb < (gr + 1) * (8 / G); ++kb) {
                        uint2 av[MT];
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt) av[mt] = act_fragment<MT>(acts, g, t, kb, mt);
                        uint4 wv[kVecPerKb];
#pragma unroll
                        for (int h = 0; h < kVecPerKb; ++h)
                            wv[h] = *reinterpret_cast<const uint4*>(tile + ((size_t)(kb * kVecPerKb + h) * 32 + lane) * 16);
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            uint32_t r0, r1, r2, r3;
                            if (BITS == 4) {
                                const uint4 v = wv[0];
                                const uint32_t x = w == 0 ? v.x : w == 1 ? v.y : w == 2 ? v.z : v.w;
                                r0 = w4_reg(x, 0, zg[w]);
                                r1 = w4_reg(x, 1, zg8[w]);
                                r2 = w4_reg(x, 2, zg[w]);
                                r3 = w4_reg(x, 3, zg8[w]);
                            } else {
                                const uint4 v = wv[(w >> 1) % kVecPerKb];
                                w8_word_to_regs((w & 1) ? v.z : v.x, r0, r1);
                                w8_word_to_regs((w & 1) ? v.w : v.y, r2, r3);
                            }
#pragma unroll
                            for (int mt = 0; mt < MT; ++mt)
                                mma_bf16_16816(gacc[w][mt], r0, r1, r2, r3, av[mt].x, av[mt].y);
                        }
                    }
                    if (gr == G - 1) {
                        // all shared-memory reads of this tile are done: hand its share of the stage back to the
                        // producer (the last tile of a short chunk also returns the shares of the missing tiles)
                        __syncwarp();
                        if (lane == 0) {
                            const int tiles_here = min(kR, seg_len - cl * kR);
                            mbar_arrive_n(empty0 + 8 * s, slot == tiles_here - 1 ? (uint32_t)(kR - tiles_here + 1) : 1u);
                        }

                    }

                    // the group's scales, in fp32 (Eq. 1 / Eq. 2 factored per group)
                    const uint32_t sw[4] = {sc.x, sc.y, sc.z, sc.w};
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        const float s_g = fp16_bits_to_float((uint16_t)(sw[w] & 0xFFFFu));
                        const float s_g8 = fp16_bits_to_float((uint16_t)(sw[w] >> 16));
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt) {
                            acc[w][mt][0] = fmaf(s_g, gacc[w][mt][0], acc[w][mt][0]);
                            acc[w][mt][1] = fmaf(s_g, gacc[w][mt][1], acc[w][mt][1]);
                            acc[w][mt][2] = fmaf(s_g8, gacc[w][mt][2], acc[w][mt][2]);
                            acc[w][mt][3] = fmaf(s_g8, gacc[w][mt][3], acc[w][mt][3]);
                        }
                    }
                }
                if (aborted) break;
                }
            }
            if (aborted) break;

            // ---- drop this warp's partial of the segment for the reducer and move on ---------------------------
            // With two buffers a warp that is a segment ahead of the slowest warp does not wait for it: a segment's
            // partials go to buffer sidx % nred, which the reducer must have read nred segments ago.
            const int rb = nred == 2 ? (sidx & 1) : 0, ru = nred == 2 ? (sidx >> 1) : sidx;
            if (!mbar_wait_warp(seg_free0 + 8 * rb, (ru & 1) ^ 1, abort_flag, 0x300)) { aborted = true; break; }
            float* mine = red + (size_t)(rb * nconsumers + cw) * kRedWarp;      // [token][n]
            if constexpr (I8) {
                // columns 3m .. 3m+2 are the pieces of token m, already on a common scale: token 0 is columns 0 and 1 of thread
                // t = 0 and column 2 of t = 1, token 1 column 3 of t = 1 and columns 4 and 5 of t = 2.  Both end where the
                // floating-point path has them (t = 0); what the other threads add up is not used.  (No choice by t: written as
                // nested conditions the compiler made divergent branches of them or not, depending on unrelated code around, and
                // the branches cost 1.1 us per segment: 1x4096x1024 4.7 against 3.6 us, x28672 16.6 against 13.8; this form
                // 3.60 and 13.52.)
#pragma unroll
                for (int w = 0; w < 4; ++w)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const float c0 = acc[w][0][2 * r], c1 = acc[w][0][2 * r + 1], both = c0 + c1;
                        acc[w][0][2 * r] = both + __shfl_down_sync(0xFFFFFFFFu, c0, 1);
                        acc[w][0][2 * r + 1] = __shfl_down_sync(0xFFFFFFFFu, c1, 1) + __shfl_down_sync(0xFFFFFFFFu, both, 2);
                    }
            }
#pragma unroll
            for (int w = 0; w < 4; ++w)
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    const int tok = 8 * mt + 2 * t;
                    if (I8 && t != 0) continue;                 // integer path: tokens 0 and 1 sit in the t = 0 threads, the buffer has two rows
                    // (the floating-point path multiplies with codes in 64ths)
                    constexpr float kUnit = I8 ? 1.f : kCodeUnit;
                    // rows g and g + 8 of the block; floating-point path: in the order of red_lane
                    const int lo = I8 ? 16 * w + g : 4 * (4 * w ^ 2 * t) + g, hi = I8 ? lo + 8 : lo ^ 8;
                    mine[tok * kTileN + lo] = kUnit * acc[w][mt][0];
                    mine[(tok + 1) * kTileN + lo] = kUnit * acc[w][mt][1];
                    mine[tok * kTileN + hi] = kUnit * acc[w][mt][2];
                    mine[(tok + 1) * kTileN + hi] = kUnit * acc[w][mt][3];
                }
            __syncwarp();
            if (lane == 0) mbar_arrive(seg_full0 + 8 * rb);
            chunk_base += (seg_len + kR - 1) / kR;
            i += seg_len;
            if (i < ntiles) { ++sidx; continue; }

            // ---- the last segment: put together by these warps, a slice each, on the integer path (one slice) by the reducer ----
            if (kLastAtEnd) last = last_segment();
            if (!I8)
                for (int e = cw; e < kVec && 2 * e < M; e += nconsumers) finish(last, e, rb, ru, false);
        }
    }

    // ---------------- cluster mode: put together the strip whose last tile this CTA holds ------------------------
    __syncthreads();
    if (CL) {
        // Every CTA of the cluster gets here (all waits above are bounded).  After the barrier the partials the
        // other CTAs stored into this CTA's slots are visible, and nobody touches another CTA's memory again.
        const int strip = t0 / ktiles, head = t0 - strip * ktiles;              // cut before this CTA, ended by it
        const bool mine = ntiles > 0 && head > 0 && head + ntiles >= ktiles;
        const int first = range_owner(strip * ktiles - cbase, ctiles, cn);
        const bool some_empty = ctiles < cn;            // a range can be empty only where the cluster has fewer tiles than CTAs
        cluster_sync_all();
        if (mine && warp >= 2 && header_ok && *abort_flag == 0)
        for (int e = warp - 2; e < kVec && 2 * e < M; e += nconsumers) {
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
            for (int c = first; c <= crank; ++c) {                             // rank order, as in global mode
                if (some_empty && range_start(c + 1, ctiles, cn) == range_start(c, ctiles, cn)) continue;   // empty range: no partial
                add_to(sum, reinterpret_cast<const float4*>(xred + (size_t)c * xslot_bytes)[32 * e + lane]);
            }
            store_slice(y, sum, e, strip, M, N, lane);
        }
    }

    // A CTA without tiles leaves about a microsecond after the dependency is met, not at once.  Measured: when the
    // surplus CTAs of a short GEMV all exit in the instant the previous kernel completes, the kernels behind it
    // on the stream are placed unevenly and a pass over four layer shapes takes 46 us instead of 37; any delay
    // between 1 and 4 us gives the 37 (the CTAs with tiles need 3 us or more from that instant anyway).
    if (idle && threadIdx.x == 0) {
        const long long t_begin = clock64();
        while (clock64() - t_begin < 2000ll) {}
    }

    // ---------------- teardown: report, and never leave with copies in flight ------------------------------
    if (threadIdx.x == 0 && (!header_ok || *abort_flag != 0)) {
        grid_dependency_wait();
        if (!header_ok) {
            if (cta == 0) { status->code = TF_ERR_BLOB; status->detail = 1; }
        } else if (*abort_flag != 0) {
            status->code = TF_ERR_TIMEOUT;
            status->detail = *abort_flag;
            // copies still in flight land within microseconds; give them a bounded moment before the
            // shared memory of this CTA is released
            const long long t_begin = clock64();
            while (clock64() - t_begin < 2000000ll) {}
        }
    }
}

// Function attributes belong to one device: set once per device and kernel instantiation.  The flag is atomic: two
// host threads may both find it unset and both set the attributes, which is harmless.
template <int BITS, int MT, bool FULL, bool CL, int I8, int G = 1>
static cudaError_t configure_one() {
    static std::atomic<bool> configured_on[kGemvMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
    const bool seen = dev >= 0 && dev < kGemvMaxDevices;
    if (seen && configured_on[dev].load(std::memory_order_acquire)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(gemv_stream_kernel<BITS, MT, FULL, CL, I8, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         FULL ? gemv_smem_budget(MT, FULL) : kGemvSoloSmemBytes);
    if (e != cudaSuccess) return e;
    // Always the largest shared-memory carve-out: a GEMV whose ring happens to be a little smaller would
    // otherwise ask for a smaller split of the SM's memory, and an SM changes its split only when idle, so
    // consecutive GEMVs of different shapes could not share an SM.
    e = cudaFuncSetAttribute(gemv_stream_kernel<BITS, MT, FULL, CL, I8, G>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    if (seen) configured_on[dev].store(true, std::memory_order_release);
    return cudaSuccess;
}

// How many clusters of `csize` CTAs the device can hold at once: of the kernel that is launched as clusters, at its block size
// and at the most shared memory that it may ask for (asked once per device).  0 if the question fails: cluster mode is then
// not used.
template <int BITS>
static int max_resident_clusters(int csize) {
    static std::atomic<int> cached[kGemvMaxDevices][4];      // [device][log2 csize], 0 = not asked yet, -1 = failed
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kGemvMaxDevices) return 0;
    const int slot = csize == 2 ? 1 : csize == 4 ? 2 : 3;
    int entry = cached[dev][slot].load(std::memory_order_relaxed);
    if (entry == 0) {                           // two host threads may both ask: same answer, harmless
        int n = 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(csize * 64, 1, 1);
        cfg.blockDim = dim3(gemv_max_threads(BITS, 2, true, false), 1, 1);
        cfg.dynamicSmemBytes = gemv_smem_budget(2, true);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = csize; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaError_t e = configure_one<BITS, 2, true, true, 0>();
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, gemv_stream_kernel<BITS, 2, true, true, 0>, &cfg);
        if (e != cudaSuccess) { cudaGetLastError(); n = 0; }
        entry = n > 0 ? n : -1;
        cached[dev][slot].store(entry, std::memory_order_relaxed);
    }
    return entry > 0 ? entry : 0;
}

// The part of a plan that follows from its form (whole SM or half): consumer warps, ring, piece table, shared memory.
static void lay_out_gemv(GemvPlan& p, int bits, int M, int tiles_per_cta, bool full) {
    const int mt = M <= 8 ? 1 : 2;
    p.full = full;
    // whole-SM integer path: about 66 KB of tiles in the consumer warps' hands (16 warps on 4-bit tiles, 8 on int8 tiles) and the rest
    // of the ring in flight (when it was chosen, one token, 8 / 12 / 16 warps: 4096x32768 4-bit 20.7 / 18.8 / 18.1 us, 4096x14336 int8
    // 12.7 / 13.3 / 14.6).
    p.consumers = p.i8 && p.full ? gemv_i8_full_consumers(bits) : gemv_max_consumers(mt, p.full);
    // Floating-point path up to 8 tokens: 12 warps only for long ranges of 4-bit tiles.  Eight have fewer partial sums to add up
    // at the end of a strip and less of the ring in their hands: us with 8 / 12, 4 tokens 14336x4096 (49 tiles) 8.35 / 8.53, a decoder layer
    // 33.7 / 34.0; 4096x28672 (97 tiles), when it was chosen, 16.4 / 15.8 and int8 at 8 tokens 22.1 / 23.1.  With four groups per tile,
    // whose scales are more work, 5 tokens 4096x14336 9.85 / 9.62.  A multiple of the tiles of a chunk, so that a warp always works on
    // the same place of a stage and a stage is freed by warps that are about equally far (10, 11 and 14 warps are slower than 8, 12, 16).
    const int twelve_from = p.groups == 1 ? kGemvFpTwelveWarpsFromTiles : kGemvFpTwelveWarpsFromTilesGrouped;
    if (mt == 1 && !p.i8 && (bits == 8 || tiles_per_cta < twelve_from)) p.consumers = 8;
    if (tiles_per_cta < p.consumers) p.consumers = tiles_per_cta < 4 ? 4 : tiles_per_cta;
    p.threads = 32 * (p.consumers + 2);          // + producer warp + reducer warp
    const int kr = gemv_chunk_tiles(bits);
    // a stage: one bulk copy of kR packed tiles, padded, and on the floating-point path their activations
    p.stage_bytes = p.i8 ? kGemvStageBytes : (kr * tile_bytes(bits, p.groups) + 127) / 128 * 128;
    const int act_stage_bytes = p.i8 ? 0 : kr * gemv_act_tile_bytes(mt);
    // cluster mode: one slot per CTA of the cluster for the rows of real tokens (two token rows = 512 bytes)
    p.xslot_bytes = p.cluster > 1 ? ((M + 1) / 2) * 512 : 0;
    // two buffers for the consumer warps' partial sums where the whole SM is taken (a boundary between strips then
    // costs a fast warp nothing; measured below), one in the half-SM form, where the second would cost a ring stage
    p.nred = p.full ? 2 : 1;
    const int base = 1024 /*alignment slack*/ + kGemvBarrierBytes + p.nred * p.consumers * (p.i8 ? 2 : 8 * mt) * kTileN * 4 +
                     (p.cluster * p.xslot_bytes + 1023) / 1024 * 1024;
    int fixed = base + (p.i8 ? p.consumers * 1024 : 0);
    int stages = (gemv_smem_budget(mt, p.full) - fixed) / (p.stage_bytes + act_stage_bytes);
    if (stages > kGemvMaxStages) stages = kGemvMaxStages;
    // no more stages than the range has chunks
    const int chunks = (tiles_per_cta + kr - 1) / kr + 2;
    if (stages > chunks) stages = chunks;
    // whole-SM integer path: a ring deeper than eight stages was slower (when it was chosen, 1x4096x32768 4-bit 17.0 / 16.9 / 17.5 us
    // with 6 / 8 / 10 stages, int8 1x4096x14336 12.8 / 12.5 / 12.7 with 6 / 8 / 11)
    if (p.i8 && p.full && stages > kGemvI8FullMaxStages) stages = kGemvI8FullMaxStages;
    // floating-point path up to 8 tokens on 4-bit tiles: five stages with 8 consumer warps (two in their hands), six with 12 (three).
    // us with 5 / 6 / 7 stages: 8 warps, 4 tokens 4096x6144 5.57 / 5.71 / 5.71, 14336x4096 8.35 / - / 9.01; 12 warps 4096x28672 14.25 /
    // 14.07 / 14.07, four groups per tile 5 tokens 4096x14336 9.58 / 9.77.  (Why a deeper ring is slower on 4-bit tiles was not
    // established.)  int8 tiles (four or six stages in the warps' hands) want the deep ring: when it was chosen, 4096x14336 at 4 tokens
    // 19.6 / 18.4 / 17.4 / 16.6 / 16.0 us with 4 / 5 / 6 / 7 / 9 (11.8 now).
    const int most = p.consumers > 8 && p.groups < 4 ? kGemvFpW4MaxStages12 : kGemvFpW4MaxStages8;
    if (!p.i8 && mt == 1 && bits == 4 && stages > most) stages = most;
    // Integer path: where a range passes over the same k-tiles more than once and K is a multiple of 128 x consumer
    // warps, every warp meets the same k-tiles on each pass and keeps the activation pieces it has prepared (one table
    // entry per k-tile instead of one scratch entry per warp), if that costs the ring no stage.
    p.piece_tab = 0;
    // (4-bit weights only: on int8 tiles, whole SM, the table was the slower form, 13.1 against 12.5 us on 1x4096x14336 then)
    if (p.i8 && bits == 4 && tiles_per_cta >= p.ktiles + p.consumers && p.ktiles % p.consumers == 0) {
        const int table = (p.ktiles * kGemvPieceEntryBytes * M + 1023) / 1024 * 1024;
        int with = (gemv_smem_budget(mt, p.full) - (base + table)) / p.stage_bytes;
        if (with > kGemvMaxStages) with = kGemvMaxStages;
        if (with > chunks) with = chunks;
        if (with >= stages) {
            p.piece_tab = p.ktiles;
            fixed = base + table;
        }
    }
    p.stages = stages;
    p.smem_bytes = fixed + p.stages * (p.stage_bytes + act_stage_bytes);
}

// Launch geometry.  Global mode: one persistent CTA per SM (fewer when there are fewer tiles than SMs), all tiles
// cut into equal ranges; a strip cut between CTAs is summed through the workspace.  Cluster mode: clusters of 2, 4
// or 8 CTAs, each cluster owning whole strips and cutting its tiles into equal ranges among its CTAs; a cut strip
// is summed through distributed shared memory, which is several microseconds shorter than the workspace hand-over
// (partial to L2, atomic, loads by the last arriver).  A kernel that contains cluster instructions starts about
// 0.7 us later than one that does not, even when launched without clusters, and a cluster launch overlaps less
// with its neighbours on the stream, so cluster mode has instantiations of its own and is taken only for short
// ranges, where the hand-over dominates the call.
GemvPlan plan_gemv(int bits, int M, int K, int N, int sm_count, int groups) {
    GemvPlan p;
    p.groups = groups;
    p.strips = (N + kTileN - 1) / kTileN;
    p.ktiles = K / kTileK;
    p.total_tiles = p.strips * p.ktiles;
    p.grid = p.total_tiles < sm_count ? p.total_tiles : sm_count;
    const int mt = M <= 8 ? 1 : 2;
    int tiles_per_cta = (p.total_tiles + p.grid - 1) / p.grid;
    // CTAs that get tiles.  The grid of a half-SM launch stays at one CTA per SM even when fewer take part: the
    // block scheduler puts the next GEMV's CTAs wherever a half SM is free, and an SM without a CTA of this
    // kernel would get two of them, which then share one SM for their whole range (measured: 2.5 us per call).
    int active = p.grid;
    // Short ranges (at most two rounds of a half-SM CTA's consumer warps): the hand-over of cut strips is most of the
    // call, so pick ranges that line up with the strips.  (a) Few tiles: no more CTAs than give every consumer warp
    // one tile; the call lasts one tile-time either way, and a strip is shared by fewer CTAs.  (b) Otherwise a
    // range length that divides a strip (or is a multiple of it) and needs no more rounds: every CTA then has one
    // cut instead of two.
    if (mt == 1) {
        const int nc = gemv_max_consumers(1, false);
        int want = 0;
        if (tiles_per_cta < nc) {
            // (A strip of fewer k-tiles is one CTA's.  With eight tiles per CTA all the same, its strips came one after the
            // other, 1 us each: 1x512x4096 took 3.4 us, now 2.0; 4x128x4096 10.5, now 2.0.)
            want = p.ktiles < nc ? p.ktiles * ((p.strips + p.grid - 1) / p.grid) : nc;
        } else if (tiles_per_cta <= 2 * nc) {
            const int rounds = (tiles_per_cta + nc - 1) / nc;
            for (int t = tiles_per_cta; t <= rounds * nc; ++t)
                if ((p.ktiles % t == 0 || t % p.ktiles == 0) && p.total_tiles % t == 0) { want = t; break; }
        }
        if (want > 0) {
            int g = (p.total_tiles + want - 1) / want;
            if (g >= 1 && g < p.grid) { active = g; tiles_per_cta = (p.total_tiles + active - 1) / active; }
        }
    }
    p.cluster = 1;
    p.nclusters = active;
    // Cluster mode, for 9..16 tokens only: the half-SM form of 1 and 2 tokens overlaps its start with the previous kernel's end, a
    // cluster launch next to a plain one does not (about 2.7 us per transition, measured), and in a pass over layers of
    // different sizes that loss is larger than what the short hand-over wins for up to 8 tokens.
    if (mt == 2 && groups == 1 && tiles_per_cta <= 16) {
        int best_c = 1, best_n = 0, best_t = 0;
        for (int c = 2; c <= 8; c *= 2) {
            // one CTA per SM
            int maxc = bits == 4 ? max_resident_clusters<4>(c) : max_resident_clusters<8>(c);
            if (maxc > sm_count / c) maxc = sm_count / c;
            if (maxc < 1) continue;
            const int j = (p.strips + maxc - 1) / maxc;                 // whole strips per cluster, at most
            const int t = (j * p.ktiles + c - 1) / c;                   // longest range of a CTA
            if (best_c == 1 || t < best_t) { best_c = c; best_n = (p.strips + j - 1) / j; best_t = t; }
        }
        // Worth it for short ranges only (there the hand-over dominates the call), and only if the longest range stays
        // within one round of the consumer warps or close to the evenly split one.
        if (best_c > 1 && (best_t <= gemv_max_consumers(mt, true) || best_t * 10 <= tiles_per_cta * 11 + 20)) {
            p.cluster = best_c;
            p.nclusters = best_n;
            p.grid = best_n * best_c;
            tiles_per_cta = best_t;
        }
    }
    if (mt == 1 && p.grid < sm_count) p.grid = sm_count;
    p.i8 = M <= kGemvI8MaxM && groups == 1 && p.cluster == 1;     // several groups per tile: floating-point path only
    // The floating-point path and 9..16 tokens take the whole SM: they are bound by what their consumer warps do, and only one
    // kernel's consumers work at a time.  The integer path of 1 and 2 tokens needs a fraction of the instructions; its short
    // ranges gain more from the next GEMV's CTAs sitting beside this one's with their rings already full, long ones amortise
    // the start of the kernel and take the whole SM too.  Where the line lies depends on whether the half-SM form keeps its
    // activation pieces, so that form is laid out first.
    lay_out_gemv(p, bits, M, tiles_per_cta, !p.i8);
    if (!p.full) {
        const int whole_from = bits == 8 ? kGemvFullFromBytesI8W8 : p.piece_tab > 0 ? kGemvFullFromBytesI8W4Kept : kGemvFullFromBytesI8W4;
        if (tiles_per_cta * tile_bytes(bits, groups) >= whole_from) lay_out_gemv(p, bits, M, tiles_per_cta, true);
    }
    // Late CTAs get shorter ranges in the whole-SM integer form (int8 1x4096x14336 11.07 -> 10.90 us; on the floating-point path it
    // changed little either way: 4 tokens 4096x28672 14.36 -> 14.48, 6 tokens, group 64, 7424x18440 16.5 -> 16.4).
    constexpr int kLate = 10, kLateTiles = 6;
    const bool some_late = p.full && p.i8 && p.nclusters == sm_count && sm_count >= 8 * kLate && p.total_tiles >= 24 * sm_count;
    p.ranges = Ranges::make(p.total_tiles, p.nclusters, some_late ? kLate : 0, kLateTiles);
    return p;
}

static LaunchNotes g_notes;

// The runtime's number of a stream may not be asked for while the stream is capturing (it ends the capture with an error); there the handle names
// it, but for cudaStreamPerThread, which is one handle for many.  The stream's place in the graph has to be a single node as well: with
// several, some are other streams' work.  (Both questions and the notes' lock are 0.11 us of host time per call.)
StreamNote::StreamNote(cudaStream_t stream) : name{0, 0, false}, seen{LaunchKind::kNone, 0} {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    unsigned long long capture = 0;
    const cudaGraphNode_t* nodes = nullptr;
    const cudaGraphEdgeData* edges = nullptr;
    cudaGraph_t graph = nullptr;
    size_t count = 0;
    cudaError_t e = cudaStreamGetCaptureInfo_v3(stream, &status, &capture, &graph, &nodes, &edges, &count);
    if (e == cudaSuccess && status == cudaStreamCaptureStatusNone) {
        e = cudaStreamGetId(stream, &name.stream);
        name.known = e == cudaSuccess;
    } else if (e == cudaSuccess && status == cudaStreamCaptureStatusActive) {
        name = {reinterpret_cast<uintptr_t>(stream), capture, stream != cudaStreamPerThread};
    }
    if (e != cudaSuccess) cudaGetLastError();       // (the launch itself reports what is wrong)
    seen = g_notes.look(name);
    if (name.capture != 0 && count != 1) seen.kind = LaunchKind::kNone;
}
void StreamNote::launched(LaunchKind kind) const { g_notes.launched(name, seen, kind); }
void StreamNote::packed() const { g_notes.packed(name); }

template <int BITS>
static cudaError_t configure_bits() {
    cudaError_t e = cudaSuccess;
    auto all = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    all(configure_one<BITS, 1, true, false, 0>());
    all(configure_one<BITS, 1, false, false, 1>()); all(configure_one<BITS, 1, true, false, 1>());
    all(configure_one<BITS, 2, true, false, 0>());  all(configure_one<BITS, 2, true, true, 0>());
    if constexpr (BITS == 4) {
        all(configure_one<4, 1, false, false, 2>()); all(configure_one<4, 1, true, false, 2>());
        all(configure_one<4, 1, true, false, 0, 2>()); all(configure_one<4, 2, true, false, 0, 2>());
        all(configure_one<4, 1, true, false, 0, 4>()); all(configure_one<4, 2, true, false, 0, 4>());
    }
    return e;
}

// Every one-time step a later launch on the current device could need (function attributes of every instantiation,
// the cluster-occupancy answers), for callers that must not meet them inside a stream capture.
cudaError_t configure_gemv_kernels() {
    cudaError_t e = configure_bits<4>();
    if (e == cudaSuccess) e = configure_bits<8>();
    for (int c = 2; c <= 8; c *= 2) { max_resident_clusters<4>(c); max_resident_clusters<8>(c); }
    return e;
}

template <int BITS, int MT, bool FULL, bool CL, int I8, int G = 1>
static cudaError_t launch_one(const GemvPlan& p, const void* blob, const void* a, void* y, int M, int K,
                              int N, void* workspace, cudaStream_t stream) {
    cudaError_t ce = configure_one<BITS, MT, FULL, CL, I8, G>();
    if (ce != cudaSuccess) return ce;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.grid, 1, 1);
    cfg.blockDim = dim3(p.threads, 1, 1);
    cfg.dynamicSmemBytes = p.smem_bytes;
    cfg.stream = stream;
    // A whole-SM kernel lets its dependents start as its CTAs leave, one by one.  Every SM freed that way is empty and
    // takes two half-SM CTAs of the next GEMV while other SMs get none: that kernel then runs on half of the SMs, and
    // so does every half-SM GEMV behind it, each on the half the one before left free (measured with %smid: 74 SMs
    // with two CTAs each, 11 us lost per transition, until the next whole-SM kernel).  So a half-SM GEMV that does not
    // follow another half-SM GEMV of this library on its stream asks for a little more than half of an SM's shared
    // memory: two of its CTAs no longer fit on one SM, a CTA of the next (plain) half-SM GEMV still fits beside it.
    const StreamNote note(stream);
    if (!FULL && !note.follows_half_sm() && cfg.dynamicSmemBytes < (size_t)kGemvSoloSmemBytes)
        cfg.dynamicSmemBytes = kGemvSoloSmemBytes;
    // Programmatic dependent launch: a CTA uses less than half of an SM (shared memory, registers), so the
    // CTAs of the next GEMV on the stream become resident while this one still runs, fill their rings with
    // weights and then wait for this kernel to finish before they touch activations, y or the workspace.
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = note.may_start_early() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (p.cluster > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = p.cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    GemvActMap<I8> act_map;
    if constexpr (I8 == 0) {
        constexpr int kBlock = 64;                  // k of one 128-byte swizzled row; rows of tokens >= M are read as zeros
        const cuuint64_t dims[3] = {kBlock, (cuuint64_t)M, (cuuint64_t)K / kBlock}, strides[2] = {(cuuint64_t)K * 2, kBlock * 2};
        const cuuint32_t box[3] = {kBlock, 8 * MT, (cuuint32_t)(gemv_chunk_tiles(BITS) * kTileK / kBlock)};
        ce = encode_bf16_map(&act_map, a, 3, dims, strides, box);
        if (ce != cudaSuccess) return ce;
    }
    ce = cudaLaunchKernelEx(&cfg, gemv_stream_kernel<BITS, MT, FULL, CL, I8, G>, act_map, static_cast<const uint8_t*>(blob),
                            static_cast<const __nv_bfloat16*>(a), static_cast<__nv_bfloat16*>(y), M, K, N, p.ktiles, p.total_tiles, p.stages, p.stage_bytes,
                            p.cluster, p.nclusters, p.ranges, p.xslot_bytes, p.nred, p.piece_tab, static_cast<uint8_t*>(workspace), debug_word());
    if (ce == cudaSuccess) note.launched(FULL ? LaunchKind::kWholeSm : LaunchKind::kHalfSm);
    return ce;
}

template <int BITS>
static cudaError_t launch_bits(const GemvPlan& p, const void* blob, const void* a, void* y, int M, int K, int N,
                               void* workspace, cudaStream_t stream) {
    if constexpr (BITS == 4) {
        // group sizes 64 and 32: the whole-SM floating-point kernel with two or four groups per tile
        if (p.groups == 2)
            return M > 8 ? launch_one<4, 2, true, false, 0, 2>(p, blob, a, y, M, K, N, workspace, stream)
                         : launch_one<4, 1, true, false, 0, 2>(p, blob, a, y, M, K, N, workspace, stream);
        if (p.groups == 4)
            return M > 8 ? launch_one<4, 2, true, false, 0, 4>(p, blob, a, y, M, K, N, workspace, stream)
                         : launch_one<4, 1, true, false, 0, 4>(p, blob, a, y, M, K, N, workspace, stream);
    }
    if (p.groups != 1) return cudaErrorInvalidValue;
    if (M > 8)                                  // the cluster instructions are compiled only into what is launched as clusters
        return p.cluster > 1 ? launch_one<BITS, 2, true, true, 0>(p, blob, a, y, M, K, N, workspace, stream)
                             : launch_one<BITS, 2, true, false, 0>(p, blob, a, y, M, K, N, workspace, stream);
    if (!p.i8) return launch_one<BITS, 1, true, false, 0>(p, blob, a, y, M, K, N, workspace, stream);
    if constexpr (BITS == 4) {
        if (p.piece_tab > 0)
            return p.full ? launch_one<4, 1, true, false, 2>(p, blob, a, y, M, K, N, workspace, stream)
                          : launch_one<4, 1, false, false, 2>(p, blob, a, y, M, K, N, workspace, stream);
    }
    return p.full ? launch_one<BITS, 1, true, false, 1>(p, blob, a, y, M, K, N, workspace, stream)
                  : launch_one<BITS, 1, false, false, 1>(p, blob, a, y, M, K, N, workspace, stream);
}

cudaError_t launch_gemv(int bits, const GemvPlan& p, const void* blob, const void* a, void* y, int M, int K,
                        int N, void* workspace, cudaStream_t stream) {
    return bits == 4 ? launch_bits<4>(p, blob, a, y, M, K, N, workspace, stream)
                     : launch_bits<8>(p, blob, a, y, M, K, N, workspace, stream);
}

}  // namespace tf
