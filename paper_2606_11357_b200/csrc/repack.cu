// Pre-tiling on the GPU (Section 4.2 done at run time instead of offline), and the GEMM arm of the layout ablation
// (Section 5.5): the fused GEMM computed from the AWQ arrays as the quantizer wrote them, i.e. re-tiled on the fly
// into scratch memory by the kernel below and then multiplied by the pre-tiled GEMM.  What the paper's offline
// pre-tiling saves is exactly this pass per call.  The device packer writes, byte for byte, what tf_pack_awq writes.
#include <cuda_runtime.h>

#include "../../include/tilefuse.h"
#include "async.cuh"
#include "kernels.h"
#include "layout.h"

namespace tf {

namespace {

// Columns of a word by nibble position: 0,2,4,6,1,3,5,7.
__device__ __forceinline__ uint32_t awq_code_dev(uint32_t word, int c) { return (word >> (4 * (((c & 1) << 2) | (c >> 1)))) & 0xFu; }

// Bits of `a` where mask is set, of `b` elsewhere.
__device__ __forceinline__ uint32_t select_bits(uint32_t a, uint32_t b, uint32_t mask) { return (a & mask) | (b & ~mask); }

// Words `out[c]`, c = 0..3, made of byte c of r0, r1, r2, r3 in this order.
__device__ __forceinline__ void transpose_bytes(uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3, uint32_t (&out)[4]) {
    const uint32_t a = __byte_perm(r0, r1, 0x5140), b = __byte_perm(r2, r3, 0x5140);      // bytes 0 and 1 of a row pair
    const uint32_t c = __byte_perm(r0, r1, 0x7362), d = __byte_perm(r2, r3, 0x7362);      // bytes 2 and 3
    out[0] = __byte_perm(a, b, 0x5410);
    out[1] = __byte_perm(a, b, 0x7632);
    out[2] = __byte_perm(c, d, 0x5410);
    out[3] = __byte_perm(c, d, 0x7632);
}

// A CTA re-tiles four neighbouring tiles (128 k x 256 n).  A thread moves two 8 x 8 nibble blocks, of rows 16 kb + 4t .. +3 (t and t + 2)
// and words 2w, 2w + 1 of its strip: it reads 8 x 8 bytes, transposes them in registers and writes one word of each of the
// eight lanes (g, t).  A warp reads 128-byte row segments, so every sector is moved once.  Bound by DRAM: 4096 x 14336 takes 11.4 us
// in a chain (5.3 TB/s).  Launched as a programmatic dependent, whose CTAs wait for the kernels before it themselves: with a plain
// launch it was 13.8 us, 1024 x 4096 4.1 (now 2.1 from a graph).  (Two tiles per CTA: 1 % slower.  One thread per output word, eight 4-byte loads
// for each: 65.6 us.)  It releases its own dependents only by ending: the GEMV and the GEMM read packed weights before they wait for
// the kernels ahead of them.
constexpr int kRepackThreads = 256, kRepackStrips = 4;
template <bool kPairs, int G>      // G: groups per tile; kPairs: rows are a whole number of word pairs, so a thread's two words are one 8-byte load
__global__ void __launch_bounds__(kRepackThreads) repack_awq_kernel(const uint32_t* qweight, const uint16_t* scales,
                                                                    const uint32_t* qzeros, uint8_t* __restrict__ out, int K, int N,
                                                                    int group_size, int ktiles, int strips) {
    constexpr int tile_bytes_here = w4_tile_bytes(G);
    const int T = blockIdx.y, S0 = kRepackStrips * blockIdx.x;
    const int row_words = N >> 3;
    grid_dependency_wait();                  // the arrays may come from earlier kernels, and those may still read what `out` held
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        tf_blob_header h = {};
        h.magic = kMagic; h.version = kBlobVersion; h.bits = 4; h.K = (uint32_t)K; h.N = (uint32_t)N;
        h.group_size = (uint32_t)group_size; h.n_padded = (uint32_t)(strips * kTileN); h.strips = (uint32_t)strips;
        h.ktiles = (uint32_t)ktiles; h.tile_bytes = (uint32_t)tile_bytes_here; h.tiles_offset = kHeaderBytes;
        h.total_bytes = (uint64_t)kHeaderBytes + (uint64_t)strips * ktiles * tile_bytes_here;
        *reinterpret_cast<tf_blob_header*>(out) = h;
    }
    auto tile_of = [&](int S) { return out + kHeaderBytes + ((size_t)S * ktiles + T) * tile_bytes_here; };

    // ---- metadata: per strip and group 32 words of scale pairs and 8 of zero points ----------------------------------
    // The loads first, so that they are on their way together with those of the weights; the words are put together and
    // stored at the end.  A scale word takes two values, a zero word eight.
    constexpr int kMetaWords = G * (kScaleBytes + kZeroBytes) / 4, kItems = (kRepackStrips * kMetaWords + kRepackThreads - 1) / kRepackThreads;
    uint32_t meta[kItems][8];
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        const int i = threadIdx.x + it * kRepackThreads;
        const int S = S0 + i / kMetaWords, wi = i % kMetaWords;
        if (i >= kRepackStrips * kMetaWords || S >= strips) continue;
        const int n0 = S * kTileN;
        if (wi < G * (kScaleBytes / 4)) {                             // [group][g][w] -> (2w, 2w + 1) = columns +0, +8
            const int gr = wi / (kScaleBytes / 4), rest = wi % (kScaleBytes / 4);
            const int n = n0 + 16 * (rest & 3) + (rest >> 2);
            const int grp = G > 1 ? T * G + gr : T * kTileK / group_size;
            meta[it][0] = n < N ? load_behind_wait(scales + (size_t)grp * N + n) : 0u;
            meta[it][1] = n + 8 < N ? load_behind_wait(scales + (size_t)grp * N + n + 8) : 0u;
        } else {                                                      // [group][g]
            const int gr = (wi - G * (kScaleBytes / 4)) / (kZeroBytes / 4);
            const int grp = G > 1 ? T * G + gr : T * kTileK / group_size;
#pragma unroll
            for (int j = 0; j < 8; ++j) {                             // nibble j: column 16 (j & 3) + 8 (j >> 2) + g
                const int zw = n0 / 8 + 2 * (j & 3) + (j >> 2);
                meta[it][j] = zw < row_words ? load_behind_wait(qzeros + (size_t)grp * row_words + zw) : 0u;
            }
        }
    }
    // ---- weights -----------------------------------------------------------------------------------------------
    {
        const int w = threadIdx.x & 3, S = S0 + ((threadIdx.x >> 2) & 3), kb = threadIdx.x >> 5;
        if (S < strips) {
            const int word0 = S * (kTileN / 8) + 2 * w;
            uint32_t even[2][4], odd[2][4];                              // padded columns: q = z = 0, s = 0
#pragma unroll
            for (int it = 0; it < 2; ++it) {
                const int t = ((threadIdx.x >> 4) & 1) + 2 * it;
                const uint32_t* src = qweight + (size_t)(T * kTileK + 16 * kb + 4 * t) * row_words + word0;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    even[it][r] = odd[it][r] = 0u;
                    if (kPairs) {
                        if (word0 < row_words) {
                            const uint2 v = load_once_behind_wait(reinterpret_cast<const uint2*>(src + (size_t)r * row_words));
                            even[it][r] = v.x; odd[it][r] = v.y;
                        }
                    } else {
                        if (word0 < row_words) even[it][r] = load_behind_wait(src + (size_t)r * row_words);
                        if (word0 + 1 < row_words) odd[it][r] = load_behind_wait(src + (size_t)r * row_words + 1);
                    }
                }
            }
            // low and high nibbles of byte b: columns {0, 4, 1, 5}[b] and {2, 6, 3, 7}[b]; a lane's word takes rows
            // 0, 2, 1, 3 in its bytes, the even word's code in the low nibble, the odd word's in the high one
#pragma unroll
            for (int it = 0; it < 2; ++it) {
                const int t = ((threadIdx.x >> 4) & 1) + 2 * it;
                uint32_t lo[4], hi[4], a[4], b[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    lo[r] = select_bits(even[it][r], odd[it][r] << 4, 0x0F0F0F0Fu);
                    hi[r] = select_bits(even[it][r] >> 4, odd[it][r], 0x0F0F0F0Fu);
                }
                transpose_bytes(lo[0], lo[2], lo[1], lo[3], a);
                transpose_bytes(hi[0], hi[2], hi[1], hi[3], b);
                uint32_t* dst = reinterpret_cast<uint32_t*>(tile_of(S)) + (kb * 32 + t) * 4 + w;      // lane (g, t): 16 g words further
                dst[0] = a[0]; dst[4 * 16] = a[1]; dst[16] = a[2]; dst[5 * 16] = a[3];
                dst[2 * 16] = b[0]; dst[6 * 16] = b[1]; dst[3 * 16] = b[2]; dst[7 * 16] = b[3];
            }
        }
    }
    // ---- metadata, stored --------------------------------------------------------------------------------------------
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        const int i = threadIdx.x + it * kRepackThreads;
        const int S = S0 + i / kMetaWords, wi = i % kMetaWords;
        if (i >= kRepackStrips * kMetaWords || S >= strips) continue;
        uint32_t word = 0;
        if (wi < G * (kScaleBytes / 4)) {
            word = meta[it][0] | (meta[it][1] << 16);
        } else {
            const int g = (wi - G * (kScaleBytes / 4)) % (kZeroBytes / 4);
#pragma unroll
            for (int j = 0; j < 8; ++j) word |= awq_code_dev(meta[it][j], g) << (4 * j);
        }
        reinterpret_cast<uint32_t*>(tile_of(S) + kW4WeightBytes)[wi] = word;
    }
}

}  // namespace

cudaError_t launch_repack_awq(const uint32_t* qweight, const uint16_t* scales, const uint32_t* qzeros, void* out, int K, int N,
                              int group_size, cudaStream_t stream) {
    const int strips = (N + kTileN - 1) / kTileN, ktiles = K / kTileK;
    const dim3 grid((strips + kRepackStrips - 1) / kRepackStrips, ktiles);
    const int G = groups_per_tile(group_size);
    auto* kernel = (N / 8) % 2 == 0 ? (G == 1 ? repack_awq_kernel<true, 1> : G == 2 ? repack_awq_kernel<true, 2> : repack_awq_kernel<true, 4>)
                                    : (G == 1 ? repack_awq_kernel<false, 1> : G == 2 ? repack_awq_kernel<false, 2> : repack_awq_kernel<false, 4>);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kRepackThreads, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const StreamNote note(stream);           // (a packing goes by nothing; it is noted whatever became of the launch)
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, qweight, scales, qzeros, static_cast<uint8_t*>(out), K, N, group_size, ktiles, strips);
    note.packed();
    return e;
}

}  // namespace tf
