// Host-side offline pre-tiling (Section 4.2 of the paper): AWQ / int8 weights -> packed blob.
// Pure byte shuffling; scales are copied bit for bit.
//
// What bounds it: memory.  The matrix is read and written once, and the shuffle between is a transposition of nibbles
// (4-bit) or bytes (int8) inside small blocks that 16-byte vectors do in a few operations per block.  Done code by code
// (the first form of this file) 4096 x 14336 4-bit weights took 59 ms, bound by about 15 scalar operations per code;
// now 0.6 to 0.7 ms with 16 cores (90 to 100 GB/s read and written).
#include <string.h>

#include <thread>
#ifdef __SSE2__
#include <emmintrin.h>
#endif
#ifdef __linux__
#include <sched.h>
#endif

#include "../../include/tilefuse.h"
#include "layout.h"

namespace {

constexpr int kAwqPosOfColumn[8] = {0, 4, 1, 5, 2, 6, 3, 7};   // nibble position of column c%8

bool legal_shape(int bits, int K, int N, int g) {
    if (bits != 4 && bits != 8) return false;
    if (K < tf::kTileK || K > TF_MAX_DIM || N < 8 || N > TF_MAX_DIM) return false;
    if (N % 8 != 0) return false;
    if (K % tf::kTileK != 0) return false;         // also for group sizes below the tile: rows behind the last whole tile would be in none
    if (g <= 0 || K % g != 0) return false;
    if (g % tf::kTileK == 0) return true;
    return bits == 4 && (g == 64 || g == 32);      // several groups inside a tile: the 4-bit format only
}

void write_header(void* out, int bits, int K, int N, int g, size_t total) {
    tf_blob_header h;
    memset(&h, 0, sizeof(h));
    h.magic = tf::kMagic;
    h.version = tf::kBlobVersion;
    h.bits = (uint32_t)bits;
    h.K = (uint32_t)K;
    h.N = (uint32_t)N;
    h.group_size = (uint32_t)g;
    h.n_padded = (uint32_t)((N + tf::kTileN - 1) / tf::kTileN * tf::kTileN);
    h.strips = h.n_padded / tf::kTileN;
    h.ktiles = (uint32_t)(K / tf::kTileK);
    h.tile_bytes = (uint32_t)tf::tile_bytes(bits, tf::groups_per_tile(g));
    h.tiles_offset = tf::kHeaderBytes;
    h.total_bytes = total;
    memcpy(out, &h, sizeof(h));
}

constexpr int kW4RowBytes = tf::kTileN / 2;          // one k of a 4-bit tile: eight words
// The next strip's part of a row is asked for while this one's is worked on: a tile reads 128 rows that are kilobytes apart, more than the
// processor follows by itself, and waited for each of them (4096x14336 4-bit, buffers that are in no cache, 16 cores: 1350 us without, 1110
// with; two lines ahead is no better).  The last strip asks for nothing: what lies behind it is another row, or behind the matrix.
// int8 only for large blobs: smaller ones mostly lie in caches, where 128 requests per tile only cost (us of one core, buffers reused, asked
// ahead / not: 512x512 15.5 / 14.1, 640x2128 87.9 / 86.7; buffers that are in no cache, 4096x11008: 3085 / 3320 with 8 cores, 977 / 997 on a
// machine with more).
constexpr size_t kLine = 64;
constexpr size_t kLargeBlob = 8 << 20;       // of a size that no cache holds until it is read

// Sixteen bytes in the compiler's portable vector form (SSE2, which every x86-64 has, or NEON).
typedef uint8_t v16u8 __attribute__((vector_size(16)));
typedef uint16_t v8u16 __attribute__((vector_size(16)));
typedef uint32_t v4u32 __attribute__((vector_size(16)));

inline v16u8 load16(const void* p) { v16u8 v; memcpy(&v, p, 16); return v; }
inline void store16(void* p, v4u32 v) { memcpy(p, &v, 16); }
inline v16u8 zip8_lo(v16u8 a, v16u8 b) { return __builtin_shuffle(a, b, (v16u8){0, 16, 1, 17, 2, 18, 3, 19, 4, 20, 5, 21, 6, 22, 7, 23}); }
inline v16u8 zip8_hi(v16u8 a, v16u8 b) { return __builtin_shuffle(a, b, (v16u8){8, 24, 9, 25, 10, 26, 11, 27, 12, 28, 13, 29, 14, 30, 15, 31}); }
inline v4u32 zip16_lo(v16u8 a, v16u8 b) { return (v4u32)__builtin_shuffle((v8u16)a, (v8u16)b, (v8u16){0, 8, 1, 9, 2, 10, 3, 11}); }
inline v4u32 zip16_hi(v16u8 a, v16u8 b) { return (v4u32)__builtin_shuffle((v8u16)a, (v8u16)b, (v8u16){4, 12, 5, 13, 6, 14, 7, 15}); }
inline v4u32 even32(v16u8 a, v16u8 b) { return __builtin_shuffle((v4u32)a, (v4u32)b, (v4u32){0, 2, 4, 6}); }
inline v4u32 odd32(v16u8 a, v16u8 b) { return __builtin_shuffle((v4u32)a, (v4u32)b, (v4u32){1, 3, 5, 7}); }

// Rows a, b, c, d of a 4 x 4 block of 32-bit words -> its columns.
inline void store_columns(v4u32 a, v4u32 b, v4u32 c, v4u32 d, uint8_t* col0, uint8_t* col1, uint8_t* col2, uint8_t* col3) {
    const v4u32 lo = {0, 4, 1, 5}, hi = {2, 6, 3, 7};
    const v4u32 ac0 = __builtin_shuffle(a, c, lo), bd0 = __builtin_shuffle(b, d, lo);
    const v4u32 ac1 = __builtin_shuffle(a, c, hi), bd1 = __builtin_shuffle(b, d, hi);
    store16(col0, __builtin_shuffle(ac0, bd0, lo));
    store16(col1, __builtin_shuffle(ac0, bd0, hi));
    store16(col2, __builtin_shuffle(ac1, bd1, lo));
    store16(col3, __builtin_shuffle(ac1, bd1, hi));
}

// The weights of one 4-bit tile.  `src` points at its first row and column, all 32 bytes of every row readable.
// Lane (g, t) of k-block kb takes, for n-block w, nibble p of its word from row 4t + {0, 0, 2, 2, 1, 1, 3, 3}[p], word
// 2w + (p & 1), column g of that word: the eight words of eight g are the 8 x 8 nibble transpose of four rows x two
// words.  Nibbles first (the even word's into the low half of a byte, the odd word's into the high half: the low
// and high nibbles of byte b are columns {0, 4, 1, 5}[b] and {2, 6, 3, 7}[b]), then bytes across the four rows, then
// 32-bit words so that the four w of a lane lie together; one vector holds the four w throughout.
inline void weights_w4(const uint8_t* src, size_t row_bytes, uint8_t* tile, bool ask_ahead) {
    const v4u32 low = {0x0F0F0F0Fu, 0x0F0F0F0Fu, 0x0F0F0F0Fu, 0x0F0F0F0Fu};
    for (int kb = 0; kb < 8; ++kb)
        for (int t = 0; t < 4; ++t) {
            v16u8 first[4], second[4];               // [row] columns 0, 4, 1, 5 and columns 2, 6, 3, 7 of the word pairs
            for (int r = 0; r < 4; ++r) {
                const uint8_t* row = src + (size_t)(16 * kb + 4 * t + r) * row_bytes;
                if (ask_ahead) __builtin_prefetch(row + kLine);
                const v16u8 x = load16(row), y = load16(row + 16);
                const v4u32 even = even32(x, y), odd = odd32(x, y);
                first[r] = (v16u8)((even & low) | ((odd & low) << 4));
                second[r] = (v16u8)(((even >> 4) & low) | (odd & ~low));
            }
            uint8_t* dst = tile + (kb * 32 + t) * 16;            // lane (g, t) lies 64 g bytes further
            // `first` and `second` are [w][b]: the bytes of the four rows side by side make the word of column b of block w
            v16u8 x = zip8_lo(first[0], first[2]), y = zip8_lo(first[1], first[3]);
            v16u8 z = zip8_hi(first[0], first[2]), u = zip8_hi(first[1], first[3]);
            store_columns(zip16_lo(x, y), zip16_hi(x, y), zip16_lo(z, u), zip16_hi(z, u), dst, dst + 4 * 64, dst + 64, dst + 5 * 64);
            x = zip8_lo(second[0], second[2]), y = zip8_lo(second[1], second[3]);
            z = zip8_hi(second[0], second[2]), u = zip8_hi(second[1], second[3]);
            store_columns(zip16_lo(x, y), zip16_hi(x, y), zip16_lo(z, u), zip16_hi(z, u), dst + 2 * 64, dst + 6 * 64, dst + 3 * 64, dst + 7 * 64);
        }
}

// The weights of one int8 tile, all 64 bytes of every row readable.  Lane (g, t) of k-block kb takes, for n-block w and
// r = 0, 1, the bytes (row 4t + 2r, column g), (row + 1, g), (row, g + 8), (row + 1, g + 8) of that block.
template <bool kAskAhead>
inline void weights_w8(const uint8_t* src, size_t row_bytes, uint8_t* tile) {
    for (int kb = 0; kb < 8; ++kb)
        for (int t = 0; t < 4; ++t) {
            if (kAskAhead)
                for (int r = 0; r < 4; ++r) __builtin_prefetch(src + (size_t)(16 * kb + 4 * t + r) * row_bytes + kLine);
            for (int h = 0; h < 2; ++h) {                        // n-blocks 2h and 2h + 1 share a 16-byte vector
                v4u32 g03[4], g47[4];                            // [2 (w & 1) + r] words of g = 0..3 and of g = 4..7
                for (int i = 0; i < 4; ++i) {
                    const uint8_t* row = src + (size_t)(16 * kb + 4 * t + 2 * (i & 1)) * row_bytes + 32 * h + 16 * (i >> 1);
                    const v16u8 a = load16(row), b = load16(row + row_bytes);
                    const v16u8 lo = zip8_lo(a, b), hi = zip8_hi(a, b);
                    g03[i] = zip16_lo(lo, hi);
                    g47[i] = zip16_hi(lo, hi);
                }
                uint8_t* dst = tile + ((kb * 2 + h) * 32 + t) * 16;
                store_columns(g03[0], g03[1], g03[2], g03[3], dst, dst + 64, dst + 2 * 64, dst + 3 * 64);
                store_columns(g47[0], g47[1], g47[2], g47[3], dst + 4 * 64, dst + 5 * 64, dst + 6 * 64, dst + 7 * 64);
            }
        }
}

// A finished tile -> the blob, past the caches: a store that goes through them first fetches the line that it overwrites.  For large blobs,
// which no cache holds until they are read: 4096x14336 4-bit 1110 -> 1060 us with buffers that are in no cache, 930 to 1390 -> 590 to 710 where two
// pairs of buffers take turns; one pair alone, packed again and again, is slower (0.6 -> 0.8 ms).
inline void put_tile(uint8_t* dst, const uint8_t* tile, size_t bytes) {
#ifdef __SSE2__
    for (size_t i = 0; i < bytes; i += 16)
        _mm_stream_si128(reinterpret_cast<__m128i*>(dst + i), _mm_load_si128(reinterpret_cast<const __m128i*>(tile + i)));
#else
    memcpy(dst, tile, bytes);
#endif
}
// Whether tiles go that way: large blobs, 16-byte aligned (the vector store wants it).
inline bool streamed(const uint8_t* tiles, size_t total) {
#ifdef __SSE2__
    return total >= kLargeBlob && reinterpret_cast<uintptr_t>(tiles) % 16 == 0;
#else
    (void)tiles; (void)total;
    return false;
#endif
}
// Behind a thread's last tile: its streaming stores are ordered before whatever it does next.
inline void put_fence() {
#ifdef __SSE2__
    _mm_sfence();
#endif
}

// `valid` bytes of each of a tile's rows, the rest zero: the last strip of an N that is not a multiple of the strip.
inline void copy_padded(uint8_t* dst, size_t dst_row, const uint8_t* src, size_t src_row, size_t valid) {
    for (int k = 0; k < tf::kTileK; ++k) {
        memcpy(dst + k * dst_row, src + k * src_row, valid);
        memset(dst + k * dst_row + valid, 0, dst_row - valid);
    }
}

void write_scales(uint8_t* tile_scales, const uint16_t* scales, int N, int grp, int n0) {
    uint16_t s[64], out[64];
    const int valid = N - n0 < tf::kTileN ? N - n0 : tf::kTileN;
    memcpy(s, scales + (size_t)grp * N + n0, 2 * (size_t)valid);
    memset(s + valid, 0, 2 * (size_t)(tf::kTileN - valid));
    for (int g = 0; g < 8; ++g)
        for (int i = 0; i < 8; ++i) out[g * 8 + i] = s[8 * i + g];          // i = 2w + h: column 16w + 8h + g
    memcpy(tile_scales, out, sizeof(out));
}

void write_zeros(uint8_t* tile_zeros, const uint32_t* qzeros, int N, int grp, int n0) {
    uint32_t z[8] = {0, 0, 0, 0, 0, 0, 0, 0}, out[8];
    const int valid = N - n0 < tf::kTileN ? (N - n0) / 8 : 8;
    memcpy(z, qzeros + (size_t)grp * (N / 8) + n0 / 8, 4 * (size_t)valid);
    for (int g = 0; g < 8; ++g) {
        uint32_t word = 0;                                                  // nibble i: column 16 (i & 3) + 8 (i >> 2) + g
        for (int i = 0; i < 8; ++i) word |= ((z[2 * (i & 3) + (i >> 2)] >> (4 * kAwqPosOfColumn[g])) & 0xFu) << (4 * i);
        out[g] = word;
    }
    memcpy(tile_zeros, out, sizeof(out));
}

// Cores this process may run on.
int usable_cores() {
#ifdef __linux__
    cpu_set_t set;
    if (sched_getaffinity(0, sizeof(set), &set) == 0) return CPU_COUNT(&set);
#endif
    const unsigned n = std::thread::hardware_concurrency();
    return n > 0 ? (int)n : 1;
}

// Calls tile(S, T) for every strip S and k-tile T.  The k-tiles of a strip are written one after the other, the strips
// of a k-tile read one after the other; the inner loop runs over the strips, because 128 source rows are then read
// front to back (a 4-bit strip uses half a cache line of a row, and the other half is still in the L1 for the next).
// The tiles are independent, so the list of them is cut into equal parts, one per core; `bytes` (of the blob) bounds the
// number of threads: below kBytesPerThread each, starting a thread (10 to 20 us) costs what it saves.
constexpr size_t kBytesPerThread = 512 * 1024;
constexpr int kMaxThreads = 16;          // the memory of one socket is busy well before that
template <typename Tile>
void for_each_tile(int strips, int ktiles, size_t bytes, const Tile& tile) {
    const long long tiles = (long long)strips * ktiles;
    auto part = [&tile, strips](long long begin, long long end) {
        int T = (int)(begin / strips), S = (int)(begin % strips);
        for (long long i = begin; i < end; ++i) {
            tile(S, T);
            if (++S == strips) { S = 0; ++T; }
        }
        put_fence();
    };
    long long threads = (long long)(bytes / kBytesPerThread);
    if (threads > 1) {
        const int cores = usable_cores();
        if (threads > cores) threads = cores;
        if (threads > kMaxThreads) threads = kMaxThreads;
        if (threads > tiles) threads = tiles;
    }
    if (threads <= 1) { part(0, tiles); return; }
    std::thread pool[kMaxThreads];
    int started = 0;
    try {                                    // a thread that the system refuses is work for this one
        for (; started < (int)threads - 1; ++started)
            pool[started] = std::thread(part, tiles * started / threads, tiles * (started + 1) / threads);
    } catch (...) {
    }
    part(tiles * started / threads, tiles);
    for (int i = 0; i < started; ++i) pool[i].join();
}

}  // namespace

static_assert(sizeof(tf_blob_header) == tf::kHeaderBytes, "header must be 256 bytes");

extern "C" __attribute__((visibility("default"))) size_t tf_packed_size(int bits, int K, int N, int group_size) {
    if (!legal_shape(bits, K, N, group_size)) return 0;
    size_t strips = (size_t)(N + tf::kTileN - 1) / tf::kTileN;
    size_t ktiles = (size_t)K / tf::kTileK;
    size_t tile = (size_t)tf::tile_bytes(bits, tf::groups_per_tile(group_size));
    return tf::kHeaderBytes + strips * ktiles * tile;
}

extern "C" __attribute__((visibility("default"))) tf_status tf_pack_awq(const uint32_t* qweight, const uint16_t* scales_fp16,
                                 const uint32_t* qzeros, int K, int N, int group_size,
                                 void* out, size_t out_bytes) {
    if (!qweight || !scales_fp16 || !qzeros || !out) return TF_ERR_NULL;
    size_t total = tf_packed_size(4, K, N, group_size);
    if (total == 0) return TF_ERR_SHAPE;
    if (out_bytes < total) return TF_ERR_WORKSPACE;
    write_header(out, 4, K, N, group_size, total);
    const size_t row_bytes = (size_t)N / 2;
    const int strips = (N + tf::kTileN - 1) / tf::kTileN, ktiles = K / tf::kTileK;
    uint8_t* base = static_cast<uint8_t*>(out) + tf::kHeaderBytes;
    const int G = tf::groups_per_tile(group_size), tile_bytes = tf::w4_tile_bytes(G);
    const uint8_t* q = reinterpret_cast<const uint8_t*>(qweight);
    const bool stream = streamed(base, total);
    for_each_tile(strips, ktiles, total, [=](int S, int T) {
        const int k0 = T * tf::kTileK, n0 = S * tf::kTileN;
        uint8_t* dst = base + ((size_t)S * ktiles + T) * tile_bytes;
        alignas(64) uint8_t buffer[tf::w4_tile_bytes(4)];
        uint8_t* tile = stream ? buffer : dst;
        const uint8_t* src = q + (size_t)k0 * row_bytes + n0 / 2;
        if (n0 + tf::kTileN <= N) {
            weights_w4(src, row_bytes, tile, S % 2 == 0 && S + 2 < strips);       // two strips' parts of a row make a line (of rows that begin with one)
        } else {
            // padded columns: q = z = 0, s = 0  ->  dequantizes to exactly 0
            uint8_t part[tf::kTileK * kW4RowBytes];
            copy_padded(part, kW4RowBytes, src, row_bytes, (size_t)(N - n0) / 2);
            weights_w4(part, kW4RowBytes, tile, false);
        }
        for (int gr = 0; gr < G; ++gr) {                 // the groups that meet this tile, along k
            const int grp = (k0 + gr * (tf::kTileK / G)) / group_size;
            write_scales(tile + tf::w4_scale_offset(gr), scales_fp16, N, grp, n0);
            write_zeros(tile + tf::w4_zero_offset(G, gr), qzeros, N, grp, n0);
        }
        if (stream) put_tile(dst, buffer, (size_t)tile_bytes);
    });
    return TF_OK;
}

extern "C" __attribute__((visibility("default"))) tf_status tf_pack_w8(const int8_t* w8, const uint16_t* scales_fp16, int K, int N,
                                int group_size, void* out, size_t out_bytes) {
    if (!w8 || !scales_fp16 || !out) return TF_ERR_NULL;
    size_t total = tf_packed_size(8, K, N, group_size);
    if (total == 0) return TF_ERR_SHAPE;
    if (out_bytes < total) return TF_ERR_WORKSPACE;
    write_header(out, 8, K, N, group_size, total);
    const int strips = (N + tf::kTileN - 1) / tf::kTileN, ktiles = K / tf::kTileK;
    uint8_t* base = static_cast<uint8_t*>(out) + tf::kHeaderBytes;
    const uint8_t* q = reinterpret_cast<const uint8_t*>(w8);
    const bool stream = streamed(base, total), large = total >= kLargeBlob;
    for_each_tile(strips, ktiles, total, [=](int S, int T) {
        const int k0 = T * tf::kTileK, n0 = S * tf::kTileN;
        uint8_t* dst = base + ((size_t)S * ktiles + T) * tf::kW8TileBytes;
        alignas(64) uint8_t buffer[tf::kW8TileBytes];
        uint8_t* tile = stream ? buffer : dst;
        const uint8_t* src = q + (size_t)k0 * N + n0;
        if (n0 + tf::kTileN <= N) {
            if (large && S + 1 < strips) weights_w8<true>(src, (size_t)N, tile);
            else weights_w8<false>(src, (size_t)N, tile);
        } else {
            uint8_t part[tf::kTileK * tf::kTileN];
            copy_padded(part, tf::kTileN, src, (size_t)N, (size_t)(N - n0));
            weights_w8<false>(part, tf::kTileN, tile);
        }
        write_scales(tile + tf::kW8WeightBytes, scales_fp16, N, k0 / group_size, n0);
        if (stream) put_tile(dst, buffer, tf::kW8TileBytes);
    });
    return TF_OK;
}

// Concatenation along N of blobs that share bits, K and group size (fused QKV, fused gate + up).  Section 4.5
// names the cost of dispatching many short GEMV operators per token; fewer, wider operators is the remedy at pack time.  Tiles are stored strip after strip, so the tiles
// of a part whose N is a multiple of the strip width are moved as they are; only the header changes.
extern "C" __attribute__((visibility("default"))) tf_status tf_pack_concat(const void* const* parts, int count, void* out,
                                                                           size_t out_bytes) {
    if (!parts || !out) return TF_ERR_NULL;
    if (count < 1) return TF_ERR_SHAPE;
    tf_blob_header first;
    long long n_total = 0;
    for (int i = 0; i < count; ++i) {
        if (!parts[i]) return TF_ERR_NULL;
        tf_blob_header h;
        memcpy(&h, parts[i], sizeof(h));
        if (h.magic != tf::kMagic || h.version != tf::kBlobVersion) return TF_ERR_BLOB;
        if (h.total_bytes != tf_packed_size((int)h.bits, (int)h.K, (int)h.N, (int)h.group_size) || h.total_bytes == 0)
            return TF_ERR_BLOB;
        if (i == 0) first = h;
        else if (h.bits != first.bits || h.K != first.K || h.group_size != first.group_size) return TF_ERR_SHAPE;
        if (i + 1 < count && h.N % tf::kTileN != 0) return TF_ERR_SHAPE;   // a part that is not last must end on a strip
        n_total += h.N;
    }
    if (n_total > TF_MAX_DIM) return TF_ERR_SHAPE;
    const size_t total = tf_packed_size((int)first.bits, (int)first.K, (int)n_total, (int)first.group_size);
    if (total == 0) return TF_ERR_SHAPE;
    if (out_bytes < total) return TF_ERR_WORKSPACE;
    uint8_t* dst = static_cast<uint8_t*>(out) + tf::kHeaderBytes;
    for (int i = 0; i < count; ++i) {
        tf_blob_header h;
        memcpy(&h, parts[i], sizeof(h));
        const size_t payload = (size_t)h.total_bytes - tf::kHeaderBytes;
        memcpy(dst, static_cast<const uint8_t*>(parts[i]) + tf::kHeaderBytes, payload);
        dst += payload;
    }
    write_header(out, (int)first.bits, (int)first.K, (int)n_total, (int)first.group_size, total);
    return TF_OK;
}

// Column-parallel sharding (Section 4.4: every worker owns distinct output columns, the activation vector is shared,
// no partial sums travel between workers).  Tiles are stored strip after strip, so the blob of a column range that
// starts and ends on strip boundaries is a contiguous byte range of the full blob plus a header of its own.
extern "C" __attribute__((visibility("default"))) tf_status tf_shard_columns(int N, int part, int parts, int* n_begin, int* n_count) {
    if (!n_begin || !n_count) return TF_ERR_NULL;
    if (N < 8 || N > TF_MAX_DIM || N % 8 != 0 || parts < 1 || part < 0 || part >= parts) return TF_ERR_SHAPE;
    const int strips = (N + tf::kTileN - 1) / tf::kTileN;
    if (parts > strips) return TF_ERR_SHAPE;                       // every part must own at least one strip
    const int s0 = (int)(((long long)part * strips) / parts), s1 = (int)(((long long)(part + 1) * strips) / parts);
    const int b = s0 * tf::kTileN, e = s1 * tf::kTileN < N ? s1 * tf::kTileN : N;
    *n_begin = b;
    *n_count = e - b;
    return TF_OK;
}

extern "C" __attribute__((visibility("default"))) tf_status tf_pack_shard(const void* packed, int part, int parts, void* out, size_t out_bytes) {
    if (!packed || !out) return TF_ERR_NULL;
    tf_blob_header h;
    memcpy(&h, packed, sizeof(h));
    if (h.magic != tf::kMagic || h.version != tf::kBlobVersion) return TF_ERR_BLOB;
    if (h.total_bytes == 0 || h.total_bytes != tf_packed_size((int)h.bits, (int)h.K, (int)h.N, (int)h.group_size)) return TF_ERR_BLOB;
    int n0 = 0, nc = 0;
    tf_status st = tf_shard_columns((int)h.N, part, parts, &n0, &nc);
    if (st != TF_OK) return st;
    const size_t total = tf_packed_size((int)h.bits, (int)h.K, nc, (int)h.group_size);
    if (total == 0) return TF_ERR_SHAPE;
    if (out_bytes < total) return TF_ERR_WORKSPACE;
    const size_t strip_bytes = (size_t)h.ktiles * h.tile_bytes;
    memcpy(static_cast<uint8_t*>(out) + tf::kHeaderBytes,
           static_cast<const uint8_t*>(packed) + tf::kHeaderBytes + (size_t)(n0 / tf::kTileN) * strip_bytes, total - tf::kHeaderBytes);
    write_header(out, (int)h.bits, (int)h.K, nc, (int)h.group_size, total);
    return TF_OK;
}
