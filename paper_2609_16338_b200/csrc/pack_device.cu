// Device-side BITCOS packer: dense int8 trits and row-major bf16 scales in device memory -> the
// four packed buffers of the layout in bitcos.h (Section II-A of the paper: presence bitmap,
// compacted sign vector in the same order; entry offsets per tile), byte for byte what the host
// packer writes.  One warp per 32 x 128 tile.
//
// Bound by memory: a byte a weight read, an eighth of one written twice.  Eight lanes take a row's 128 bytes, 16 weights a lane, four rows
// a load: whole lines, where one lane per row (the products' order) touched 32 rows a load at half a sector each.  Those
// 16-weight chunks in the order (load, lane) are the tile's weights in order, and the sign bits of a chunk lie where a
// scan of the chunk counts puts them.
//
// Where a tile's sign bits go is known only when everything before it has been counted.  From kOnceMin tiles on one kernel does all of it
// (pack_once_kernel): a block keeps the compacted sign bits of its tiles in shared memory until the tiles before have been
// counted, so that the trits are read and looked at once.  Smaller matrices, those with more tiles than its ranges hold and calls that
// find no state to share take three kernels: bitmap + scales + per-tile counts (and the sign vector zeroed); an exclusive scan of
// the counts (the entry offsets); the sign vector, from a second reading, mostly from L2.
//
// A C call, three kernels -> one, medians of calls in turn, us: 64 tiles 21.2 -> 19.2, 256 21.7 -> 21.8, 1024 22.4 -> 23.9, 2560 32.6 -> 34.0, 4096 28.9 ->
// 31.0, 6144 33.6 -> 33.5, 8192 38.9 -> 34.9, 10240 (8192x5120) 43.4 -> 38.1, 20480 70.6 -> 51.3, 32000 (25600x5120) 104.7 -> 65.6.  With few tiles the
// look-back's trips to L2 are a larger part than a second reading.  Through the binding 8192x5120 takes 77 (as a cooperative launch of
// one block of 1024 threads per multiprocessor 81), about 40 of them allocations and calls in Python; the trits would pass in 6.4 at
// the memory's rate.  A tile is about 1100 warp instructions (a quarter of them the compress), 0.19 us a tile and multiprocessor, which bounds the
// kernel; behind the tiles come the look-back and the sign words.
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cstdint>

#include "bitcos.h"

namespace bitcos_detail {
void record_cuda_error(int e);      // defined next to bitcos_last_cuda_error
void *mapped_host(const void *p, size_t bytes);
}

namespace {

constexpr int kGroup = BITCOS_GROUP;
constexpr int kRows = BITCOS_TILE_ROWS;
constexpr int kPackWarps = 8;       // tiles per thread block

// words of the caller's scratch
constexpr int kFlagTrit = 0;        // a weight outside {-1, 0, +1}
constexpr int kFlagScale = 1;       // a scale that is negative, NaN or Inf
constexpr int kFlagOverflow = 2;    // more than 2^32 - 1 non-zero weights
constexpr int kFlagWait = 3;        // (one-pass kernel) a wait for the tiles before ran out
constexpr int kNnzLo = 4;           // 64-bit count of non-zero weights (two words, 8-byte aligned)

inline int check_cuda(cudaError_t e) {
    if (e == cudaSuccess) return BITCOS_OK;
    bitcos_detail::record_cuda_error(static_cast<int>(e));
    cudaGetLastError();                 // (or the next call's launch check would find this one's error)
    return BITCOS_ERR_CUDA;
}
inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline int64_t padded_rows(int64_t M) { return (M + kRows - 1) / kRows * kRows; }

// 16 consecutive weights (a 16-byte load) -> presence and negative masks of 16 bits.  A trit's bit 0 says present, its bit 7 negative, and
// a dp4a with the powers of two gathers four of them.  `squares` sums the squares: they are the number of non-zero weights
// unless one is not in {-1, 0, +1} (an even one adds 4 or more to the squares and nothing to the count, an odd one 9 or more and one).
__device__ __forceinline__ void masks16(const uint4 &v, uint32_t &pres, uint32_t &neg, int &squares) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t p[2], n[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        p[i] = __dp4a(w[2 * i + 1] & 0x01010101u, 0x80402010u, __dp4a(w[2 * i] & 0x01010101u, 0x08040201u, 0u));
        n[i] = __dp4a(w[2 * i + 1] & 0x80808080u, 0x80402010u, __dp4a(w[2 * i] & 0x80808080u, 0x08040201u, 0u));      // (times 128)
#pragma unroll
        for (int j = 0; j < 2; ++j) squares = __dp4a(static_cast<int>(w[2 * i + j]), static_cast<int>(w[2 * i + j]), squares);
    }
    pres = p[0] + (p[1] << 8);
    neg = (n[0] + (n[1] << 8)) >> 7;
}

// Chunk i of this lane in the tile (row block rb, group g): weights 16 (lane % 8) .. + 15 of row 4 i + lane / 8; rows
// beyond M read as zero.
__device__ __forceinline__ uint4 load_chunk(const int8_t *__restrict__ trits, int64_t M, int64_t K, int64_t rb, int g, int i, int lane) {
    const int64_t m = rb * kRows + 4 * i + (lane >> 3);
    if (m >= M) return make_uint4(0u, 0u, 0u, 0u);
    return __ldg(reinterpret_cast<const uint4 *>(trits + m * K + static_cast<int64_t>(g) * kGroup) + (lane & 7));
}

// The bits of both halves of `src` at the set positions of the halves of `mask`, packed towards bit 0 of each half (the inverse
// of the deposit of Fig. 4): the parallel-suffix compress of Warren, "Hacker's Delight", 2nd ed., section 7-4, its shifts kept inside the
// halves; in round i every selected bit moves right by 2^i if the number of
// unselected positions below it has bit i set.
__device__ __forceinline__ uint32_t extract_halves(uint32_t src, uint32_t mask) {
    uint32_t x = src & mask, m = mask;
    uint32_t mk = (~m << 1) & 0xFFFEFFFEu;       // the unselected positions, moved up by one: what lies below each bit
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint32_t mp = mk ^ ((mk << 1) & 0xFFFEFFFEu);      // prefix parity of mk, half by half
        mp ^= (mp << 2) & 0xFFFCFFFCu;
        mp ^= (mp << 4) & 0xFFF0FFF0u;
        mp ^= (mp << 8) & 0xFF00FF00u;
        const uint32_t mv = mp & m;              // bits to move in this round (they stay in their half: 2^i positions below are unselected)
        m = (m ^ mv) | (mv >> (1 << i));
        const uint32_t t = x & mv;
        x = (x ^ t) | (t >> (1 << i));
        mk &= ~mp;
    }
    return x;
}

// Kernel 1: bitmap, scales in tile order, number of non-zero weights per tile (into tile_off, with two bits above it for
// what is wrong with the tile); and zeros over the sign vector, into which kernel 3 ORs the words that two tiles share.
constexpr uint32_t kBadTrit = 0x80000000u, kBadScale = 0x40000000u, kCountMask = 0x3FFFFFFFu;
// (A block per eight tiles, no loop: with a grid of eight blocks per multiprocessor most warps had one tile and a few two.)
__global__ void __launch_bounds__(kPackWarps * 32) pack_bitmap_kernel(const int8_t *__restrict__ trits,
                                                                      const uint16_t *__restrict__ scales, int64_t M, int64_t K,
                                                                      uint16_t *__restrict__ bitmap,
                                                                      uint16_t *__restrict__ scales_tiled,
                                                                      uint32_t *__restrict__ tile_off, int64_t n_tiles,
                                                                      uint4 *__restrict__ signs, int64_t sign_quads) {
    const int lane = threadIdx.x & 31;
    const int G = static_cast<int>(K / kGroup);
    int squares = 0;
    const int64_t t = static_cast<int64_t>(blockIdx.x) * kPackWarps + (threadIdx.x >> 5);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (t < n_tiles) {
        const int64_t rb = t / G;
        const int g = static_cast<int>(t - rb * G);
        uint4 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = load_chunk(trits, M, K, rb, g, i, lane);
        const int64_t m = rb * kRows + lane;
        uint16_t s = 0;
        if (m < M) s = __ldg(scales + m * G + g);
        uint32_t c = 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            uint32_t pres, neg;
            masks16(v[i], pres, neg, squares);
            bitmap[t * 256 + 32 * i + lane] = static_cast<uint16_t>(pres);
            c += __popc(pres);
        }
        scales_tiled[t * kRows + lane] = s;
        const bool bad = static_cast<uint32_t>(squares) != c;
        c = __reduce_add_sync(0xFFFFFFFFu, c);
        if (__any_sync(0xFFFFFFFFu, bad)) c |= kBadTrit;
        if (__any_sync(0xFFFFFFFFu, (s & 0x8000u) || (s & 0x7F80u) == 0x7F80u)) c |= kBadScale;
        if (lane == 0) tile_off[t] = c;
    }
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < sign_quads; i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        signs[i] = make_uint4(0u, 0u, 0u, 0u);
}

// Kernel 2: exclusive scan of the per-tile counts in place, one thread block walking the array 8192 tiles at a time
// (eight to a thread); tile_off[n_tiles] and the 64-bit total receive the sum, the words after it up to n_words zero.
// The offsets also go straight to the host's copy where that is mapped (off_host, may be NULL): 41 KB that cross the bus
// while kernel 3 runs, where a copy after it took 11 us.
constexpr int kScanThreads = 1024;
constexpr int kScanQuads = 2;       // 16-byte loads per thread
__global__ void __launch_bounds__(kScanThreads) scan_counts_kernel(uint32_t *__restrict__ tile_off, uint32_t *__restrict__ off_host,
                                                                   int64_t n_tiles, int64_t n_words,
                                                                   unsigned int *__restrict__ flags, volatile unsigned int *report) {
    __shared__ uint32_t warp_sum[kScanThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long carry = 0ull;                 // the same in every thread
    bool over = false;
    uint32_t seen = 0u;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int64_t base = 0; base < n_tiles; base += kScanThreads * kScanQuads * 4) {
        const int64_t i0 = base + static_cast<int64_t>(threadIdx.x) * (kScanQuads * 4);
        uint32_t c[kScanQuads * 4];
        uint32_t mine = 0u;
#pragma unroll
        for (int q = 0; q < kScanQuads; ++q) {
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            const int64_t i = i0 + 4 * q;
            if (i < n_words) v = __ldcg(reinterpret_cast<const uint4 *>(tile_off + i));      // (n_words: a multiple of four)
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t x = i + j < n_tiles ? w[j] : 0u;
                seen |= x;
                c[4 * q + j] = x & kCountMask;
                mine += c[4 * q + j];
            }
        }
        uint32_t upto = mine;                        // (a pass holds at most 8192 x 4096 non-zeros)
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, upto, d);
            if (lane >= d) upto += o;
        }
        if (lane == 31) warp_sum[warp] = upto;
        __syncthreads();
        uint32_t w_upto = warp_sum[lane];            // every warp scans the warps' sums itself
        const uint32_t w_mine = w_upto;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, w_upto, d);
            if (lane >= d) w_upto += o;
        }
        const uint32_t before = __shfl_sync(0xFFFFFFFFu, w_upto - w_mine, warp), pass = __shfl_sync(0xFFFFFFFFu, w_upto, 31);
        unsigned long long at = carry + before + (upto - mine);
#pragma unroll
        for (int q = 0; q < kScanQuads; ++q) {
            const int64_t i = i0 + 4 * q;
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                w[j] = i + j <= n_tiles ? static_cast<uint32_t>(at) : 0u;
                over = over || (i + j <= n_tiles && at > 0xFFFFFFFFull);
                at += c[4 * q + j];
            }
            if (i < n_words) {
                *reinterpret_cast<uint4 *>(tile_off + i) = make_uint4(w[0], w[1], w[2], w[3]);
                if (off_host) *reinterpret_cast<uint4 *>(off_host + i) = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
        carry += pass;
        __syncthreads();
    }
    const int any_over = __syncthreads_or(over || carry > 0xFFFFFFFFull);
    const int any_trit = __syncthreads_or((seen & kBadTrit) != 0u), any_scale = __syncthreads_or((seen & kBadScale) != 0u);
    // the sentinel, where the last pass ended exactly on it
    for (int64_t i = n_tiles + threadIdx.x; i < n_words; i += kScanThreads) {
        tile_off[i] = i == n_tiles ? static_cast<uint32_t>(carry) : 0u;
        if (off_host) off_host[i] = i == n_tiles ? static_cast<uint32_t>(carry) : 0u;
    }
    if (threadIdx.x == 0) {
        flags[kFlagTrit] = any_trit ? 1u : 0u;
        flags[kFlagScale] = any_scale ? 1u : 0u;
        flags[kFlagOverflow] = any_over ? 1u : 0u;
        flags[kNnzLo] = static_cast<unsigned int>(carry);
        flags[kNnzLo + 1] = static_cast<unsigned int>(carry >> 32);
        // what the host wants to know, straight into its memory
        report[kFlagTrit] = any_trit ? 1u : 0u;
        report[kFlagScale] = any_scale ? 1u : 0u;
        report[kFlagOverflow] = any_over ? 1u : 0u;
        report[kNnzLo] = static_cast<unsigned int>(carry);
        report[kNnzLo + 1] = static_cast<unsigned int>(carry >> 32);
    }
    __threadfence_system();
}

// Kernel 3: the sign vector.  Tile t owns the bits tile_off[t] .. tile_off[t + 1] - 1; its chunks' sign bits are gathered in
// shared memory, aligned to the vector's words, and go out as whole words, the first and the last (which the tile may
// share with its neighbours) by an atomic OR.  Two chunks are compacted at a time, in the halves of one word.  Nothing
// is written if the counts found something wrong or the vector does not fit its buffer (the host reports it).
constexpr int kSignWords = kRows * kGroup / 32 + 1;      // 4096 bits starting anywhere in a word
__global__ void __launch_bounds__(kPackWarps * 32) pack_signs_kernel(const int8_t *__restrict__ trits, int64_t M, int64_t K,
                                                                     const uint32_t *__restrict__ tile_off,
                                                                     uint32_t *__restrict__ signs, unsigned long long max_nnz, int64_t n_tiles,
                                                                     const unsigned int *__restrict__ flags) {
    __shared__ uint32_t words[kPackWarps][kSignWords + 3];
    const int lane = threadIdx.x & 31;
    const int G = static_cast<int>(K / kGroup);
    uint32_t *buf = words[threadIdx.x >> 5];
    const int64_t t = static_cast<int64_t>(blockIdx.x) * kPackWarps + (threadIdx.x >> 5);
    if (t < n_tiles) {
        const int64_t rb = t / G;
        const int g = static_cast<int>(t - rb * G);
        uint4 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = load_chunk(trits, M, K, rb, g, i, lane);
        for (uint32_t i = lane; i < kSignWords; i += 32) buf[i] = 0u;
        // the chunks' sign bits and where they lie inside the tile
        uint32_t both[4], cnt[4], at0[4], at1[4], at = 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t p0, n0, p1, n1;
            int unused = 0;                          // (kernel 1 has looked at the values)
            masks16(v[2 * i], p0, n0, unused);
            masks16(v[2 * i + 1], p1, n1, unused);
            both[i] = extract_halves(n0 | (n1 << 16), p0 | (p1 << 16));
            cnt[i] = __popc(p0) | (__popc(p1) << 16);
            uint32_t upto = cnt[i];                  // (at most 512 per load: both scans in one register)
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, upto, d);
                if (lane >= d) upto += o;
            }
            const uint32_t total = __shfl_sync(0xFFFFFFFFu, upto, 31), before = upto - cnt[i];
            at0[i] = at + (before & 0xFFFFu);
            at1[i] = at + (total & 0xFFFFu) + (before >> 16);
            at += (total & 0xFFFFu) + (total >> 16);
        }
        // All of that needed the trits alone; the tile's place needs the scan.
        asm volatile("griddepcontrol.wait;" ::: "memory");
        // (from L2: this kernel may have been resident before those words were written)
        if (__ldcg(flags + kFlagTrit) || __ldcg(flags + kFlagScale) || __ldcg(flags + kFlagOverflow) ||
            (__ldcg(flags + kNnzLo) | (static_cast<unsigned long long>(__ldcg(flags + kNnzLo + 1)) << 32)) > max_nnz)
            return;
        const uint32_t first = __ldcg(tile_off + t);
        const uint32_t sh0 = first & 31u, bits = sh0 + at;      // bits of the buffer in use
        __syncwarp();
        auto put = [&](uint32_t pos, uint32_t b, uint32_t n) {
            if (!b) return;
            atomicOr(buf + (pos >> 5), b << (pos & 31u));
            if ((pos & 31u) + n > 32u) atomicOr(buf + (pos >> 5) + 1, b >> (32u - (pos & 31u)));
        };
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t c0 = cnt[i] & 0xFFFFu;    // (at most 16)
            put(sh0 + at0[i], both[i] & 0xFFFFu, c0);
            put(sh0 + at1[i], both[i] >> 16, cnt[i] >> 16);
        }
        __syncwarp();
        uint32_t *out = signs + (first >> 5);
        const uint32_t full = bits >> 5;             // whole words, the first one among them if sh0 == 0
        for (uint32_t i = lane; i < (bits + 31u) >> 5; i += 32) {
            if ((i == 0 && sh0) || i >= full) {
                if (buf[i]) atomicOr(out + i, buf[i]);
            } else {
                out[i] = buf[i];
            }
        }
    }
}

// Inclusive scan over the lanes of a warp (the shuffle's own in-range predicate guards each addition).
__device__ __forceinline__ uint32_t scan_add(uint32_t v) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
        asm volatile("{\n\t.reg .b32 o;\n\t.reg .pred p;\n\tshfl.sync.up.b32 o|p, %0, %1, 0, 0xFFFFFFFF;\n\t@p add.u32 %0, %0, o;\n\t}" : "+r"(v) : "r"(d));
    return v;
}

// All of it in one pass: a block takes the next range of the tiles (its sign bits are contiguous too).  It counts and
// compacts them, the sign bits into 512 bytes of shared memory a tile, publishes its total, adds up those of the ranges before its
// own, and writes its offsets and sign words.  The sum is a decoupled look-back (Merrill and Garland, "Single-pass Parallel Prefix Scan
// with Decoupled Look-back", 2016): a word per range, first its own total, then the total up to and with it.
// A range is taken by a ticket, and a block waits for lower tickets only: those blocks are running and wait for none above
// them, so the kernel ends whatever else is on the chip, as few of its blocks as may find room at a time (a cooperative launch
// of one block per multiprocessor waited for all of the chip to be free).  The waits are bounded all the same.
constexpr int kOnceThreads = 256;
constexpr int kOnceTiles = 88;                   // per range at most: 516 bytes each, together within the 48 KB that need no attribute
constexpr int kOnceMin = 6144;                   // tiles: from here on one kernel is faster (see above)
constexpr int kOnceBlocks = 4;                   // resident per multiprocessor (64 registers a thread)
constexpr int kOnceRanges = 2048;
constexpr unsigned long long kOnceLimitNs = 500ull * 1000 * 1000;
constexpr int kReportSlots = 64;
// A range's word: its count, what is wrong with it, how far the count reaches, and the number of the call (words of
// earlier calls are thereby void: nothing has to be cleared between calls, whatever became of them).
constexpr int kWordBad = 32, kWordState = 34, kWordTag = 36;
constexpr unsigned int kStateOwn = 1u, kStateUpTo = 2u, kStateGaveUp = 3u;
constexpr unsigned long long kOnceTags = 1ull << (64 - kWordTag);
struct OnceState {                               // one per report slot and device
    unsigned int ticket;                         // 0 between calls: every block takes one, and the last one wraps
    unsigned long long range[kOnceRanges];
};
__device__ OnceState g_once_state[kReportSlots];

__device__ __forceinline__ unsigned long long range_word(uint32_t count, uint32_t bad, unsigned int state, unsigned long long tag) {
    return count | static_cast<unsigned long long>(bad >> 30) << kWordBad | static_cast<unsigned long long>(state) << kWordState | tag << kWordTag;
}
__device__ __forceinline__ void publish(unsigned long long *at, unsigned long long word) {
    __threadfence();
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(at), "l"(word) : "memory");
}

// Total and faults of the ranges before range r (one warp); false if a wait ran out here or there.
__device__ __forceinline__ bool look_back(const OnceState &st, int r, unsigned long long tag, int lane, unsigned long long limit_ns, uint32_t &base,
                                          uint32_t &bad) {
    base = bad = 0u;
    for (int nearest = r - 1;; nearest -= 32) {
        const int j = nearest - lane;
        unsigned long long word, t0 = 0;
        uint32_t use;                                // the lanes up to and with the first whose total reaches back to the beginning
        bool to_the_start;
        for (uint32_t i = 0;; ++i) {
            word = range_word(0u, 0u, kStateUpTo, tag);      // (in front of the first range)
            if (j >= 0) asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(word) : "l"(st.range + j) : "memory");
            const unsigned int state = (word >> kWordTag) == tag ? static_cast<unsigned int>(word >> kWordState) & 3u : 0u;
            const uint32_t ready = __ballot_sync(0xFFFFFFFFu, state != 0u), up_to = __ballot_sync(0xFFFFFFFFu, state == kStateUpTo);
            if (__any_sync(0xFFFFFFFFu, state == kStateGaveUp)) return false;
            to_the_start = up_to != 0u;
            use = 2u * (up_to & (0u - up_to)) - 1u;  // (all lanes if there is none, or only the last)
            if ((ready & use) == use) break;
            if ((i & 15u) == 15u) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now));
                if (!t0) t0 = now;
                if (__any_sync(0xFFFFFFFFu, now - t0 > limit_ns)) return false;
            }
        }
        const bool mine = (use >> lane) & 1u;
        base += __reduce_add_sync(0xFFFFFFFFu, mine ? static_cast<uint32_t>(word) : 0u);
        bad |= __reduce_or_sync(0xFFFFFFFFu, mine ? (static_cast<uint32_t>(word >> kWordBad) & 3u) << 30 : 0u);
        if (to_the_start) return true;
    }
}

__global__ void __launch_bounds__(kOnceThreads, kOnceBlocks) pack_once_kernel(const int8_t *__restrict__ trits, const uint16_t *__restrict__ scales, int64_t M,
                                                                   int64_t K, uint32_t *__restrict__ bitmap, uint16_t *__restrict__ scales_tiled,
                                                                   uint32_t *__restrict__ tile_off, uint32_t *__restrict__ off_host, int n_tiles,
                                                                   int per_range, int n_words, uint32_t *__restrict__ signs, int64_t sign_quads,
                                                                   unsigned long long max_nnz, int slot, unsigned long long tag,
                                                                   unsigned long long limit_ns, volatile unsigned int *report) {
    extern __shared__ __align__(16) uint32_t shared[];
    __shared__ uint32_t s_bad, s_base, s_warp[kOnceThreads / 32];
    __shared__ int s_range, s_ok;
    OnceState &st = g_once_state[slot];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_ranges = static_cast<int>(gridDim.x);
    const int G = static_cast<int>(K / kGroup);
    uint32_t *words = shared, *count = shared + per_range * 128;      // [tile][128], [tile]
    if (threadIdx.x == 0) {
        s_bad = 0u;
        s_range = static_cast<int>(atomicInc(&st.ticket, static_cast<unsigned int>(n_ranges - 1)));
    }
    __syncthreads();
    const int r = s_range, t_lo = r * per_range, mine = n_tiles - t_lo < per_range ? n_tiles - t_lo : per_range;
    // ---- counts, bitmap, scales; sign bits into shared memory
    uint4 v[8];
    uint16_t s_v = 0;
    auto fetch = [&](int lt, uint4 (&o)[8], uint16_t &sc) {
        const int t = t_lo + lt, rb = t / G, g = t - rb * G;
        const int64_t m = static_cast<int64_t>(rb) * kRows, row = m + (lane >> 3);
        const int8_t *from = trits + row * K + g * kGroup + 16 * (lane & 7);
        if (m + kRows <= M) {
#pragma unroll
            for (int i = 0; i < 8; ++i, from += 4 * K) o[i] = __ldg(reinterpret_cast<const uint4 *>(from));
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i, from += 4 * K) o[i] = row + 4 * i < M ? __ldg(reinterpret_cast<const uint4 *>(from)) : make_uint4(0u, 0u, 0u, 0u);
        }
        sc = m + lane < M ? __ldg(scales + (m + lane) * G + g) : static_cast<uint16_t>(0);
    };
    for (int lt = warp; lt < mine; lt += kOnceThreads / 32) {
        fetch(lt, v, s_v);
        const int64_t t = t_lo + lt;
        uint32_t *buf = words + lt * 128;
#pragma unroll
        for (int i = 0; i < 4; ++i) buf[32 * i + lane] = 0u;
        uint32_t both[4], cnt[4], at0[4], at1[4], at = 0u, c = 0u;
        int squares = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t p0, n0, p1, n1;
            masks16(v[2 * i], p0, n0, squares);
            masks16(v[2 * i + 1], p1, n1, squares);
            // presence words: even lanes store those of load 2 i, odd lanes those of load 2 i + 1
            const uint32_t give = (lane & 1) ? p0 : p1, got = __shfl_xor_sync(0xFFFFFFFFu, give, 1);
            const uint32_t word = (lane & 1) ? got | (p1 << 16) : p0 | (got << 16);
            bitmap[t * 128 + 32 * i + 16 * (lane & 1) + (lane >> 1)] = word;
            both[i] = extract_halves(n0 | (n1 << 16), p0 | (p1 << 16));
            cnt[i] = __popc(p0) | (__popc(p1) << 16);
            c += cnt[i];
            const uint32_t upto = scan_add(cnt[i]);  // (at most 512 per load: both scans in one register)
            const uint32_t total = __shfl_sync(0xFFFFFFFFu, upto, 31), before = upto - cnt[i];
            at0[i] = at + (before & 0xFFFFu);
            at1[i] = at + (total & 0xFFFFu) + (before >> 16);
            at += (total & 0xFFFFu) + (total >> 16);
        }
        scales_tiled[t * kRows + lane] = s_v;
        uint32_t flags = 0u;
        if (__any_sync(0xFFFFFFFFu, static_cast<uint32_t>(squares) != (c & 0xFFFFu) + (c >> 16))) flags |= kBadTrit;
        if (__any_sync(0xFFFFFFFFu, (s_v & 0x8000u) || (s_v & 0x7F80u) == 0x7F80u)) flags |= kBadScale;
        if (lane == 0) {
            count[lt] = at;
            if (flags) atomicOr(&s_bad, flags);
        }
        __syncwarp();                                // (the zeros, before the bits)
        const uint32_t buf_at = static_cast<uint32_t>(__cvta_generic_to_shared(buf));
        auto put = [&](uint32_t pos, uint32_t bits) {
            // (without branches: few chunks have no negative weight, and one in four reaches into the next word)
            const uint32_t lo = bits << (pos & 31u), hi = __funnelshift_l(bits, 0u, pos);
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tred.shared.or.b32 [%0], %1;\n\t@p red.shared.or.b32 [%0 + 4], %2;\n\t}" ::"r"(
                             buf_at + ((pos >> 3) & ~3u)),
                         "r"(lo), "r"(hi)
                         : "memory");
        };
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            put(at0[i], both[i] & 0xFFFFu);
            put(at1[i], both[i] >> 16);
        }
    }
    // Zeros over the sign vector: the words that would be this range's if every weight were there, and a share of what lies behind all of
    // those.  Sign bits never lie further back, so a range's zeros are written over by itself and later ranges only, which
    // have waited for its word.  (Behind the reading of the tiles: in front of it 16384x5120 | 25600x5120 took 53.3 | 68.7 us a call, here
    // 51.3 | 65.6.)
    uint4 *const zeros = reinterpret_cast<uint4 *>(signs);
    const uint4 none = make_uint4(0u, 0u, 0u, 0u);
    const int64_t z_lo = static_cast<int64_t>(t_lo) * 32, z_hi = z_lo + mine * 32 < sign_quads ? z_lo + mine * 32 : sign_quads;
    for (int64_t i = z_lo + threadIdx.x; i < z_hi; i += kOnceThreads) zeros[i] = none;
    for (int64_t i = static_cast<int64_t>(n_tiles) * 32 + r * kOnceThreads + threadIdx.x; i < sign_quads; i += static_cast<int64_t>(n_ranges) * kOnceThreads)
        zeros[i] = none;
    __syncthreads();
    // ---- this range's total, and every tile's place behind the range's first sign bit (a tile per thread)
    const uint32_t c = threadIdx.x < static_cast<unsigned>(mine) ? count[threadIdx.x] : 0u;
    const uint32_t upto = scan_add(c);
    if (lane == 31) s_warp[warp] = upto;
    __syncthreads();
    uint32_t before = 0u, total = 0u;
#pragma unroll
    for (int w = 0; w < kOnceThreads / 32; ++w) {
        if (w < warp) before += s_warp[w];
        total += s_warp[w];
    }
    const uint32_t place = before + upto - c;
    if (warp == 0) {
        uint32_t base = 0u, bad = 0u;
        if (r && lane == 0) publish(st.range + r, range_word(total, s_bad, kStateOwn, tag));
        const bool ok = (limit_ns || !r) && look_back(st, r, tag, lane, limit_ns, base, bad);
        __syncwarp();                                // (what the lanes have acquired, before lane 0 passes it on)
        if (lane == 0) {
            bad |= s_bad;
            publish(st.range + r, range_word(base + total, bad, ok ? kStateUpTo : kStateGaveUp, tag));
            s_base = base;
            s_ok = ok;
            if (!ok) {
                report[kFlagWait] = 1u;
            } else if (r == n_ranges - 1) {
                report[kFlagTrit] = (bad & kBadTrit) ? 1u : 0u;
                report[kFlagScale] = (bad & kBadScale) ? 1u : 0u;
                report[kFlagOverflow] = 0u;          // (kOnceTiles x kOnceRanges tiles hold fewer than 2^32 weights)
                report[kNnzLo] = base + total;
                report[kNnzLo + 1] = 0u;
            }
        }
    }
    __syncthreads();
    if (!s_ok) return;
    const uint32_t base = s_base;
    if (threadIdx.x < static_cast<unsigned>(mine)) {
        count[threadIdx.x] = place;
        tile_off[t_lo + threadIdx.x] = base + place;
        if (off_host) off_host[t_lo + threadIdx.x] = base + place;
    }
    if (r == n_ranges - 1) {
        for (int i = n_tiles + static_cast<int>(threadIdx.x); i < n_words; i += kOnceThreads) {
            tile_off[i] = i == n_tiles ? base + total : 0u;
            if (off_host) off_host[i] = i == n_tiles ? base + total : 0u;
        }
    }
    __syncthreads();
    // ---- the sign words; the first and the last of a tile may hold bits of its neighbours.  A vector that is too small gets those
    // that fit (the host reports it).
    for (int lt = warp; lt < mine; lt += kOnceThreads / 32) {
        const uint32_t *buf = words + lt * 128;
        const uint32_t from = count[lt], bits = (lt + 1 < mine ? count[lt + 1] : total) - from;
        const uint32_t first = base + from, sh = first & 31u, full = (sh + bits) >> 5;
        if (static_cast<unsigned long long>(first) + bits > max_nnz) break;
        uint32_t *out = signs + (first >> 5);
        for (uint32_t i = lane; i < (sh + bits + 31u) >> 5; i += 32) {
            const uint32_t w = __funnelshift_l(i ? buf[i - 1] : 0u, i < 128u ? buf[i] : 0u, sh);
            if ((i == 0 && sh) || i >= full) {
                if (w) atomicOr(out + i, w);
            } else {
                out[i] = w;
            }
        }
    }
}

// Non-zero count and validity only (to size the sign vector before packing).
__global__ void __launch_bounds__(256) count_nnz_kernel(const int8_t *__restrict__ trits, int64_t n16,
                                                        unsigned int *__restrict__ flags) {
    unsigned long long c = 0ull;
    bool bad = false;
    const uint4 *src = reinterpret_cast<const uint4 *>(trits);
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n16;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const uint4 v = __ldg(src + i);
        uint32_t pres, neg;
        int squares = 0;
        masks16(v, pres, neg, squares);
        bad = bad || squares != __popc(pres);
        c += __popc(pres);
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, d);
    if (bad) atomicOr(flags + kFlagTrit, 1u);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(reinterpret_cast<unsigned long long *>(flags + kNnzLo), c);
}

int grid_for(int64_t units, int per_block) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 128;
    const int64_t want = (units + per_block - 1) / per_block;
    const int64_t cap = static_cast<int64_t>(sms) * 8;
    return static_cast<int>(want < 1 ? 1 : (want < cap ? want : cap));
}

// As few ranges as the chip holds blocks: all start together and look back once, at their ends (ranges of 8 | 16 | 32 tiles took
// 144 | 144 | 130 us where 55 take 116, 25600x5120, and 96 | 89 | 85 where 18 take 81, 8192x5120).
int tiles_per_range(int64_t n_tiles) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) sms = 128;
    const int64_t at_once = static_cast<int64_t>(sms) * kOnceBlocks;
    const int64_t rounds = (n_tiles + at_once * kOnceTiles - 1) / (at_once * kOnceTiles);
    int64_t per_range = (n_tiles + at_once * rounds - 1) / (at_once * rounds);
    while (per_range * kOnceRanges < n_tiles) ++per_range;
    return static_cast<int>(per_range);
}

// The host's end of scan_counts_kernel's report: 64-byte slots of one pinned page, mapped into every device, taken for the
// time of a call (a copy of 32 bytes to pageable memory costs about 10 us more than this).  A caller that finds no
// free slot gets none and reads the scratch words by a copy.
struct ReportSlot {
    static std::atomic<uint64_t> &taken() {
        static std::atomic<uint64_t> t{0};
        return t;
    }
    static unsigned int *page() {
        static unsigned int *p = [] {
            void *v = nullptr;
            if (cudaHostAlloc(&v, kReportSlots * 64, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
                cudaGetLastError();
                v = nullptr;
            }
            return static_cast<unsigned int *>(v);
        }();
        return p;
    }
    // numbers for the calls that use a slot's device state (by its holder only)
    static unsigned long long next_tag(int slot) {
        static unsigned long long used[kReportSlots];
        return ++used[slot];
    }
    int slot = -1;
    ReportSlot() {
        if (!page()) return;
        uint64_t t = taken().load();
        while (~t) {
            const int i = __builtin_ctzll(~t);
            if (taken().compare_exchange_weak(t, t | (1ull << i))) {
                slot = i;
                return;
            }
        }
    }
    ~ReportSlot() {
        if (slot >= 0) taken().fetch_and(~(1ull << slot));
    }
    ReportSlot(const ReportSlot &) = delete;
    ReportSlot &operator=(const ReportSlot &) = delete;
    unsigned int *host() const { return slot < 0 ? nullptr : page() + slot * 16; }
};

// A launch that may start while the kernel before it is still running (what depends on it waits in the kernel).
template <typename... KArgs, typename... Args>
int launch_behind(void (*kernel)(KArgs...), int64_t grid, int threads, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return check_cuda(cudaLaunchKernelEx(&cfg, kernel, args...));
}

int read_flags(const void *scratch, cudaStream_t stream, unsigned int (&h)[8]) {
    int rc = check_cuda(cudaMemcpyAsync(h, scratch, sizeof h, cudaMemcpyDeviceToHost, stream));
    if (rc) return rc;
    return check_cuda(cudaStreamSynchronize(stream));
}

}  // namespace

extern "C" {

int bitcos_count_nnz_device(const int8_t *trits, int64_t M, int64_t K, uint64_t *nnz, void *scratch, void *cuda_stream) {
    if (!trits || !nnz || !scratch) return BITCOS_ERR_NULL;
    if (M < 1 || K < kGroup || K % kGroup != 0) return BITCOS_ERR_SHAPE;
    if (!aligned16(trits) || !aligned16(scratch)) return BITCOS_ERR_ALIGN;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    int rc = check_cuda(cudaMemsetAsync(scratch, 0, BITCOS_PACK_SCRATCH_BYTES, stream));
    if (rc) return rc;
    const int64_t n16 = M * K / 16;
    count_nnz_kernel<<<grid_for(n16, 256 * 8), 256, 0, stream>>>(trits, n16, static_cast<unsigned int *>(scratch));
    rc = check_cuda(cudaGetLastError());
    if (rc) return rc;
    unsigned int h[8];
    rc = read_flags(scratch, stream, h);
    if (rc) return rc;
    if (h[kFlagTrit]) return BITCOS_ERR_TRIT;
    *nnz = static_cast<uint64_t>(h[kNnzLo]) | (static_cast<uint64_t>(h[kNnzLo + 1]) << 32);
    return BITCOS_OK;
}

int bitcos_pack_device(const int8_t *trits, const uint16_t *scales_bf16, int64_t M, int64_t K, uint32_t *bitmap,
                       uint32_t *signs, size_t sign_capacity_bytes, uint32_t *tile_off, uint16_t *scales_tiled,
                       uint32_t *tile_off_host, uint64_t *nnz_out, void *scratch, void *cuda_stream) {
    return bitcos_pack_device_limited(trits, scales_bf16, M, K, bitmap, signs, sign_capacity_bytes, tile_off, scales_tiled, tile_off_host, nnz_out,
                                      scratch, kOnceLimitNs, nullptr, cuda_stream);
}

int bitcos_pack_device_limited(const int8_t *trits, const uint16_t *scales_bf16, int64_t M, int64_t K, uint32_t *bitmap, uint32_t *signs,
                               size_t sign_capacity_bytes, uint32_t *tile_off, uint16_t *scales_tiled, uint32_t *tile_off_host, uint64_t *nnz_out,
                               void *scratch, uint64_t limit_ns, int *kernels, void *cuda_stream) {
    if (!trits || !scales_bf16 || !bitmap || !signs || !tile_off || !scales_tiled || !scratch) return BITCOS_ERR_NULL;
    if (M < 1 || K < kGroup || K % kGroup != 0) return BITCOS_ERR_SHAPE;
    if (!aligned16(trits) || !aligned16(scales_bf16) || !aligned16(bitmap) || !aligned16(signs) || !aligned16(tile_off) ||
        !aligned16(scales_tiled) || !aligned16(scratch))
        return BITCOS_ERR_ALIGN;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    const int64_t n_tiles = padded_rows(M) / kRows * (K / kGroup);
    size_t off_bytes = 0;
    int rc = bitcos_pack_sizes(M, K, 0, nullptr, nullptr, &off_bytes, nullptr);
    if (rc) return rc;
    // the sign bits the caller's buffer has room for (32 bytes of zero slack behind them; the whole is a multiple of 16)
    const size_t slack = 32;
    unsigned long long max_nnz = 0;
    if (sign_capacity_bytes >= slack) max_nnz = static_cast<unsigned long long>((sign_capacity_bytes - slack) / 16 * 16) * 8;
    unsigned int *flags = static_cast<unsigned int *>(scratch);
    // the host's copy of the offsets, if the device can write there (all of it: else it is copied)
    uint32_t *off_mapped = tile_off_host ? static_cast<uint32_t *>(bitcos_detail::mapped_host(tile_off_host, off_bytes)) : nullptr;
    if (!aligned16(off_mapped)) off_mapped = nullptr;
    const int64_t grid = (n_tiles + kPackWarps - 1) / kPackWarps;
    if (grid > 0x7FFFFFFF) return BITCOS_ERR_SHAPE;
    const ReportSlot report;
    unsigned int *report_dev = flags;                // (no slot: the words report on themselves)
    if (report.host()) {
        rc = check_cuda(cudaHostGetDevicePointer(reinterpret_cast<void **>(&report_dev), report.host(), 0));
        if (rc) return rc;
    }
    bool once = report.host() && n_tiles >= kOnceMin && n_tiles <= static_cast<int64_t>(kOnceTiles) * kOnceRanges;
    unsigned long long tag = 0;
    if (once) {
        tag = ReportSlot::next_tag(report.slot);
        once = tag < kOnceTags;
    }
    auto enqueue = [&]() -> int {
        int e = BITCOS_OK;
        if (once) {
            const int per_range = tiles_per_range(n_tiles);
            report.host()[kFlagWait] = 0u;
            pack_once_kernel<<<static_cast<unsigned>((n_tiles + per_range - 1) / per_range), kOnceThreads, static_cast<size_t>(per_range) * 516, stream>>>(
                trits, scales_bf16, M, K, bitmap, scales_tiled, tile_off, off_mapped, static_cast<int>(n_tiles), per_range,
                static_cast<int>(off_bytes / 4), signs, static_cast<int64_t>(sign_capacity_bytes / 16), max_nnz, report.slot, tag, limit_ns,
                static_cast<volatile unsigned int *>(report_dev));
            e = check_cuda(cudaGetLastError());
            if (!e && tile_off_host && !off_mapped) e = check_cuda(cudaMemcpyAsync(tile_off_host, tile_off, off_bytes, cudaMemcpyDeviceToHost, stream));
            return e;
        }
        pack_bitmap_kernel<<<static_cast<unsigned>(grid), kPackWarps * 32, 0, stream>>>(
            trits, scales_bf16, M, K, reinterpret_cast<uint16_t *>(bitmap), scales_tiled, tile_off, n_tiles, reinterpret_cast<uint4 *>(signs),
            static_cast<int64_t>(sign_capacity_bytes / 16));
        e = check_cuda(cudaGetLastError());
        if (!e)
            e = launch_behind(scan_counts_kernel, 1, kScanThreads, stream, tile_off, off_mapped, n_tiles, static_cast<int64_t>(off_bytes / 4),
                              flags, static_cast<volatile unsigned int *>(report_dev));
        if (!e)
            e = launch_behind(pack_signs_kernel, grid, kPackWarps * 32, stream, trits, M, K, static_cast<const uint32_t *>(tile_off), signs,
                              max_nnz, n_tiles, static_cast<const unsigned int *>(flags));
        if (!e && tile_off_host && !off_mapped)
            e = check_cuda(cudaMemcpyAsync(tile_off_host, tile_off, off_bytes, cudaMemcpyDeviceToHost, stream));
        return e;
    };
    unsigned int h[8];
    for (int launched = 0;;) {
        rc = enqueue();
        if (rc) {
            cudaStreamSynchronize(stream);           // what was enqueued writes the report's slot and the caller's buffers
            return rc;
        }
        launched += once ? 1 : 3;
        if (kernels) *kernels = launched;
        if (report.host()) {
            rc = check_cuda(cudaStreamSynchronize(stream));
            for (int i = 0; i < 8; ++i) h[i] = static_cast<const volatile unsigned int *>(report.host())[i];
        } else {
            rc = read_flags(scratch, stream, h);     // (waits for the stream)
        }
        if (rc) return rc;
        if (!once || !h[kFlagWait]) break;
        // A block in front of another one stood still for longer than the limit.  The three kernels wait for nothing of the kind,
        // and write every output anew.
        once = false;
    }
    if (h[kFlagTrit]) return BITCOS_ERR_TRIT;
    if (h[kFlagScale]) return BITCOS_ERR_SCALE;
    if (h[kFlagOverflow]) return BITCOS_ERR_OVERFLOW;
    const uint64_t nnz = static_cast<uint64_t>(h[kNnzLo]) | (static_cast<uint64_t>(h[kNnzLo + 1]) << 32);
    size_t need = 0;
    rc = bitcos_pack_sizes(M, K, nnz, nullptr, &need, nullptr, nullptr);
    if (rc) return rc;
    if (sign_capacity_bytes < need) return BITCOS_ERR_CAPACITY;
    if (nnz_out) *nnz_out = nnz;
    return BITCOS_OK;
}

}  // extern "C"
