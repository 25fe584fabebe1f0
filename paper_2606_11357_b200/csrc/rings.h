// The shared memory of a GEMM CTA: how many stages its rings have.  No CUDA in it, so that a host program can ask.
#pragma once
#include "layout.h"

namespace tf {

constexpr int kGroups = 4;                // dequantization groups of four warps
constexpr int kBK = 64;                   // k of one 128-byte swizzled activation row
constexpr int kMaxActStages = 8;
constexpr int kMaxWpStages = 8;

// Packed-weight ring: one stage = a chunk of one or two k-tiles of the two strips.  A chunk goes to one group per k-tile, and
// the ring is a whole number of rounds of the groups, so a stage always meets the same groups and the parity of its barrier
// cannot alias.  Narrow token tiles consume weights fast and want 66 to 140 KB of them in flight (with 26 KB a 32-token tile
// could not take a k-tile faster than one per 0.34 us: the latency of HBM), 4-bit ones in chunks of two: the thread that
// issues the copies pays about 100 cycles for each.
TF_HD constexpr int chunk_tiles(int bits, int bt) { return bt > 128 || bits == 8 ? 1 : 2; }
TF_HD constexpr int wp_stage_bytes(int bits, int bt, int G) { return 2 * chunk_tiles(bits, bt) * tile_bytes(bits, G); }
// Activations.  Up to 128 tokens a k-tile of them is one stage that goes with an operand stage: one barrier says that both
// are there and one that both are free, so the warp that issues the MMAs, whose waits and issue set the pace of narrow tiles,
// pays for one of each per k-tile.  A k-tile of 256 tokens is 64 KB; there the ring is of half k-tiles, with barriers of its own.
TF_HD constexpr bool tied(int bt) { return bt <= 128; }
TF_HD constexpr int act_stage_k(int bt) { return tied(bt) ? kTileK : kBK; }
constexpr int kGemmSmemMax = 227 * 1024;  // dynamic shared memory one CTA may ask for
// Per dequant warp, for the drain of an accumulator: 8 tokens x 32 columns of bf16.  Rings are whole rounds of the groups, so a few KB here
// can cost a round: with 1024 bytes int8 tiles of 80 tokens have four stages instead of eight, 4-bit ones of 80 and 112 six and four instead of
// eight and six, tiles of 176, 208 and 240 tokens one stage of activations less (us in a chain, 1024 / 512 bytes: int8 80x4096x14336 20.1 / 19.1,
// 144x4096x4096 13.1 / 12.8; 4-bit 80, 112 and 256 tokens within 0.5 %).
constexpr int kDrainWarpBytes = 512;
constexpr int kGemmBarrierBytes = 1024;
constexpr int kGemmSmemFixed = 1024 /*alignment slack*/ + 4 * kGroups * kDrainWarpBytes + kGemmBarrierBytes;
// The rings share what the fixed part leaves: the activations (of the call's own bt columns) come first where they are tied;
// otherwise the weights take one round of the groups and the activations the rest.
struct GemmRings {
    int act_stage_bytes, act_stages, wp_stages, smem_bytes;
};
inline GemmRings gemm_rings(int bits, int BT, int act_rows, int G) {
    GemmRings r;
    const int left = kGemmSmemMax - kGemmSmemFixed, wp = wp_stage_bytes(bits, BT, G), round = kGroups / chunk_tiles(bits, BT);
    r.act_stage_bytes = act_rows * act_stage_k(BT) * 2;
    if (tied(BT)) {
        r.act_stages = kGroups;
        r.wp_stages = (left - r.act_stages * r.act_stage_bytes) / wp / round * round;
        if (r.wp_stages > kMaxWpStages) r.wp_stages = kMaxWpStages;
    } else {
        r.wp_stages = round;
        r.act_stages = (left - r.wp_stages * wp) / r.act_stage_bytes;
        if (r.act_stages > kMaxActStages) r.act_stages = kMaxActStages;
    }
    r.smem_bytes = kGemmSmemFixed + r.act_stages * r.act_stage_bytes + r.wp_stages * wp;
    return r;
}

}  // namespace tf
