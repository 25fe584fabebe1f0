// Device helpers shared by the kernels: unpack (Section 4.3 "unpacking"), exact de-bias,
// warp-level MMA, header check.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "../../include/tilefuse.h"
#include "layout.h"

namespace tf {

// Device status word layout at the start of a workspace.
struct DeviceStatus {
    uint32_t code;      // tf_status
    uint32_t detail;    // where a bounded wait gave up / which header field mismatched
    uint32_t pad[2];
};

// ---- codes -> bf16 ------------------------------------------------------------------------
// A bf16 whose upper eight bits are zero is its lower eight bits times 2^-133 (subnormal up to 127, and the first normal binade
// continues the line to 255), so a masked code already is a number and one fused multiply-add by a power of two takes it to
// its place and subtracts the zero point: exactly (q - z) / 64, the 64 being what the largest power of two that bf16 holds,
// 2^127, leaves over (kCodeUnit; whoever adds the products up multiplies by it, exactly).  Register i of a packed word sits in
// nibbles i and i + 4; registers 1 and 3 stay sixteen times too large under their mask and get a smaller power of two.
// Nine instructions per packed word, five of them on the integer pipe, which takes two cycles for each and bounds every loop that
// unpacks.  (With the code OR-ed into the bf16 128.0 and a subtraction it was eleven and seven: GEMV 4 tokens 4096x28672 15.8 us,
// now 14.9; 16 tokens 20.2 and 19.4; 6 tokens, group 64, 7424x18440 18.3 and 17.4; int8, 8 tokens, 4096x14336 13.4 and 12.5; GEMM
// 77x2944x11016, group 32, 16.0 and 15.4, int8 1024x4096x4096 29.6 and 28.9.)  Results do not change: everything is scaled by a
// power of two, which shows only where sums come within 2^-110 of zero or 2^118 of infinity.
constexpr float kCodeUnit = 64.f;
__device__ __forceinline__ uint32_t bf16x2_fma(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
constexpr uint32_t kCodeScale = 0x7F007F00u, kCodeScale16 = 0x7D007D00u;       // 2^127, 2^123
constexpr uint32_t kMinusCodeScale = 0xFF00FF00u, kMinusCodeScale16 = 0xFD00FD00u;
__device__ __forceinline__ uint32_t w4_masked(uint32_t word, int i) { return (i & 2 ? word >> 8 : word) & (i & 1 ? 0x00F000F0u : 0x000F000Fu); }
// Register i of a packed word: (q + minus_zero * 64) / 64 in both halves.
__device__ __forceinline__ uint32_t w4_reg(uint32_t word, int i, uint32_t minus_zero) {
    return bf16x2_fma(w4_masked(word, i), i & 1 ? kCodeScale16 : kCodeScale, minus_zero);
}
// The zero points of a lane's rows 16 i + g and 16 i + g + 8: -z / 64, each in both halves of a register.
__device__ __forceinline__ void w4_minus_zero(uint32_t zword, int i, uint32_t& row_g, uint32_t& row_g8) {
    const uint32_t pair = bf16x2_fma(w4_masked(zword, i), i & 1 ? kMinusCodeScale16 : kMinusCodeScale, 0x80008000u);
    row_g = __byte_perm(pair, 0, 0x1010);
    row_g8 = __byte_perm(pair, 0, 0x3232);
}
// Four int8 in a word -> two bf16x2 registers (bytes 0, 1 and bytes 2, 3), exactly a byte / 64: the byte plus 128, without a
// sign, then the same multiply-add with -128.  Five instructions per word (through the fraction of 128.0 it took eight).
__device__ __forceinline__ void w8_word_to_regs(uint32_t word, uint32_t& lo, uint32_t& hi) {
    const uint32_t u = word ^ 0x80808080u;
    lo = bf16x2_fma(__byte_perm(u, 0, 0x4140), kCodeScale, 0xC000C000u);       // -2
    hi = bf16x2_fma(__byte_perm(u, 0, 0x4342), kCodeScale, 0xC000C000u);
}

// ---- warp MMA: D(16x8, fp32) += A(16x16, bf16) . B(16x8, bf16) ---------------------------
__device__ __forceinline__ void mma_bf16_16816(float d[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                               uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Two floats rounded to bf16, the first one in the low half.
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// Header fields that kernels compare with its arguments (first 24 bytes of the blob).
__device__ __forceinline__ bool header_matches(const void* blob, uint32_t bits, uint32_t K, uint32_t N) {
    const uint4 h = __ldg(reinterpret_cast<const uint4*>(blob));            // magic, version, bits, K
    const uint2 h2 = __ldg(reinterpret_cast<const uint2*>(blob) + 2);       // N, group_size
    return h.x == kMagic && h.y == kBlobVersion && h.z == bits && h.w == K && h2.x == N;
}

// The group size recorded in the header.
__device__ __forceinline__ uint32_t header_group_size(const void* blob) {
    return __ldg(reinterpret_cast<const uint32_t*>(blob) + 5);
}
// The same in two steps, for a kernel that has something to do while the header is on its way: the words are asked for at its start
// and judged where the answer is needed (GEMV, floating-point path, a chain of whole-SM kernels, where the set-up of the last CTAs is on
// the call's way: 4 tokens 4096x6144 5.76 -> 5.56 us, 14336x4096 8.77 -> 8.56, 16 tokens 4096x28672 18.7 -> 18.5).  With the group
// size, which has to fit a kernel built for G groups per tile (G = 1: any multiple of the tile's k-extent; G = 2, 4: exactly 128 / G).
struct HeaderWords {
    uint4 a;            // magic, version, bits, K
    uint2 b;            // N, group size
    __device__ __forceinline__ explicit HeaderWords(const void* blob)
        : a(__ldg(reinterpret_cast<const uint4*>(blob))), b(__ldg(reinterpret_cast<const uint2*>(blob) + 2)) {}
    // (the empty statement keeps the compiler from judging once, ahead of everything: the wait for the words would be there too)
    __device__ __forceinline__ bool fit(uint32_t bits, uint32_t K, uint32_t N, int G) {
        asm volatile("" : "+r"(a.x), "+r"(a.y), "+r"(a.z), "+r"(a.w), "+r"(b.x), "+r"(b.y));
        return a.x == kMagic && a.y == kBlobVersion && a.z == bits && a.w == K && b.x == N &&
               (G == 1 ? (b.y >= (uint32_t)kTileK && b.y % kTileK == 0) : b.y == (uint32_t)(kTileK / G));
    }
};

__device__ __forceinline__ float fp16_bits_to_float(uint16_t h) {
    return __half2float(__ushort_as_half(h));
}

}  // namespace tf
