// The products' kernels and their launch functions (plans, layouts, the persistent staged kernel body); the C entry
// points are in gemv.cu, the instantiations in gemv_inst.cu.
//
// Work decomposition (all formats).  Rows are handled 32 at a time (a "row block"), one
// row per lane, so that the activations a warp needs are the same for all of its lanes
// and arrive by broadcast reads; the reduction is cut into groups of 128.  A tile is one
// group of one row block (32 x 128 weights); one warp decodes one tile at a time.  An
// "item" is a run of up to 20 consecutive tiles -- CG groups of one row block, or several
// whole row blocks when a row has few groups -- and is what one thread block processes per
// pipeline stage: because tiles are stored in that order, an item's bitmap words, sign bits,
// scales and entry offsets are four contiguous byte ranges, fetched with four bulk asynchronous
// copies (cp.async.bulk + mbarrier) into a ring of shared-memory stages while earlier stages are
// being decoded.  Thread blocks are persistent and take either a contiguous range of the item
// list or every n-th row-block chunk.  Row sums are formed in a fixed order (a fixed tree over the
// groups inside a block through shared memory; column blocks ascending through a scratch buffer
// and an arrival counter), so results do not depend on scheduling.
//
// Contraction.  One token (the baseline formats: two): dp4a against activations kept in shared memory.  More:
// mma.m16n8k32 (int8 in, int32 out), so that the decode is paid once per call whatever the batch; BITCOS tiles are
// decoded in fragment order (FragmentRows), the rows of the two baseline formats pass through a small shared-memory
// buffer to ldmatrix.
//
// BITCOS decode (paper Section II-D, Eq. 4, adapted): the GPU has no bit-deposit
// instruction, so four weights at a time are rebuilt from a (presence nibble, next four
// sign bits) key through a 256-entry table held in shared memory, replicated once per lane
// so that lookups never conflict.  Entries are the four weights as int8 (w = p - 2n, Eq. 2)
// ready for dp4a or the tensor cores.  A lane's position in the sign vector is the tile's entry offset
// plus a warp prefix sum over the rows' population counts; the four 32-bit presence words of
// a lane's row are decoded as four independent chains, each rotating its own sign window by
// a running position that advances by the sign bits a nibble consumed.
#ifndef BITCOS_GEMV_CUH
#define BITCOS_GEMV_CUH

#include "bitcos.h"
#include "decode.cuh"

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdlib>
#include <algorithm>
#include <cstring>
#include <mutex>
#include <tuple>
#include <type_traits>
#include <utility>
#include <vector>

namespace bitcos_kernels {

using namespace bitcos_dev;

constexpr int kGroup = BITCOS_GROUP;
constexpr int kRows = BITCOS_TILE_ROWS;
constexpr int kMaxWarps = 20;             // warps per thread block = tiles per item
constexpr int kWarps16 = 14;              // the same for more than 8 tokens (16 warps per block: 128 registers per thread)
constexpr int kMaxStages = 8;             // upper bound on the shared-memory ring depth (Plan::stages)
constexpr uint64_t kWaitLimitNs = 500ull * 1000 * 1000;   // an mbarrier wait gives up after half a second
constexpr int64_t kXResidentBytes = 48 * 1024;   // activations up to this size are kept in shared memory
constexpr int kMmaMinBatch = 4;           // from this many tokens on the contraction runs on the tensor cores
constexpr int kScrRowBytes = 48;          // a quarter of a decoded row (32 int8) + 16 bytes of padding against bank conflicts
constexpr int kScrBytes = kRows * kScrRowBytes;   // per decoder warp: the transposition buffer in front of ldmatrix

enum Format { kBitcos = 0, kTrit5 = 1, kBit2 = 2 };

inline thread_local int g_last_cuda_error = 0;

// The replicated lookup tables in their shared-memory form (decode.cuh); each thread block fetches
// its copy from global memory with one bulk asynchronous copy.
__device__ __align__(128) const LutBig g_bitcos_lut = make_bitcos_lut();
__device__ __align__(128) const LutBig g_trit5_lut = make_trit5_big();
__device__ __align__(128) const LutBig g_bitcos_bf16_lut = make_bitcos_bf16_lut();

// ---------------------------------------------------------------------------------------------
// Launch plan and problem description.
// ---------------------------------------------------------------------------------------------
struct Plan {
    int CG;          // groups per column block
    int CS;          // column blocks per row
    int RBC;         // row blocks per item (1 unless CS == 1)
    int NW;          // decoder warps per thread block = ceil(CG * RBC / tpw)
    int tpw;         // tiles of an item per decoder warp: 1, or 2 or 3 on large matrices
    int sub, wsub, wrow;   // make_run_plan: tiles and warps of a column block of the one-tile plan, warps of a row
    int64_t items;   // ceil(RB / RBC) * CS
    int cyclic;      // 1: blocks take whole row-block chunks round robin; 0: contiguous balanced ranges
    int stages;      // depth of the shared-memory ring (2 .. kMaxStages), set at launch
    int x_in_stage;  // 1: every stage also receives the item's activation rows (grouped launch, 1-2 tokens)
    int wq, wrem;    // contiguous walk: blocks 0 .. wrem-1 own wq + 1 items, the others wq (set at launch)
};

struct Problem {
    const uint32_t *payload;   // bitmap / five-trit words / 2-bit words
    const uint32_t *signs;
    const uint32_t *tile_off;
    const uint16_t *scales;    // tile order
    const int8_t *x;
    const float *x_scale;
    const int32_t *xrow;       // NULL: token b reads row b of x
    float *y;
    int32_t *acc_debug;
    float *partial;
    unsigned int *counters;
    unsigned int *status;      // device word set to 1 if an mbarrier wait ran out
    int64_t M, K;
    int G, RB;
    int nb;                    // tokens in this call / group
    int64_t out_row0;          // first output row of y / acc_debug for token 0
};

// Entry offsets of every thread block's first item (sign-vector positions of its first tile and of
// the tile after its last), passed by value when the caller supplied a host copy of tile_off.
constexpr int kMaxGrid = 160;
struct FirstOff {
    uint32_t lo[kMaxGrid];
    uint32_t hi[kMaxGrid];
    int valid;
    // every block's share of the items, worked out on the host (no divisions at kernel start)
    int first[kMaxGrid];
    int count[kMaxGrid];
    int walks;                 // 1: first / count are filled in
};

// Arrays some LATER launch will read (the packed weights of the next products of a layer): every
// thread block asks for its 1 / gridDim.x share of each to be brought into L2 once its own first
// copies are on their way, so that the later launch starts from L2 instead of device memory.
constexpr int kMaxPrefetch = 28;
struct PrefetchList {
    const uint8_t *ptr[kMaxPrefetch];
    uint32_t bytes[kMaxPrefetch];     // multiples of 16
    int n;
#ifdef BITCOS_TIMELINE
    unsigned long long *tl;           // debug build: 16 time stamps per thread block of this launch
#endif
};
#ifdef BITCOS_TIMELINE
#define BITCOS_TLP(src, i)                                                                                              \
    do {                                                                                                                \
        if constexpr (Segs::kHetero)                                                                                    \
            if ((src).pa->tl) (src).pa->tl[static_cast<size_t>(blockIdx.x) * 32 + (src).phase * 6 + (i)] = global_timer_ns(); \
    } while (0)
#else
#define BITCOS_TLP(src, i) \
    do {                   \
    } while (0)
#endif
// What the producer warp needs to send a thread block's first copies on their way, worked out on
// the host for every block of a multi launch: with it the block's first tiles and its lookup table
// are requested a few hundred cycles after the block starts, before any of the block's own address
// arithmetic (arguments, layout, walk, item ranges), which then runs while the data is in flight.
struct FirstCopies {
    const void *src[4];      // entry offsets, bitmap, sign bits, scales of the block's first item
    uint32_t bytes[4];       // (bytes[2] may be 0: an item without a nonzero weight)
    uint32_t dst[4];         // byte offsets inside the block's shared memory
    uint32_t desc[4];        // the item's descriptor for the decoder warps (see issue_item)
    uint32_t desc_off;       // where it goes
    uint32_t bar;            // byte offset of the barrier region
};
struct FirstCopiesTable {
    FirstCopies c[kMaxGrid];
    int valid;
};
// (the table is 14 KB of kernel arguments: free when the launch is recorded into a CUDA graph, whose
// arguments are staged once, but about 4 us of launch latency on a plain stream launch, which therefore
// goes without it)
struct NoFirstCopies {
    int valid;
};
template <typename T>
struct first_copy {
    __device__ static bool sent(const T &, int) { return false; }
};
template <>
struct first_copy<FirstCopiesTable> {
    __device__ static bool sent(const FirstCopiesTable &t, int b) { return t.valid != 0 && t.c[b].bytes[1] != 0; }
};

// Debug build (-DBITCOS_TIMELINE): where a thread block of the multi launch spends its time.
#ifdef BITCOS_TIMELINE
#define BITCOS_TL(i, v)                                                                   \
    do {                                                                                  \
        if (pf && pf->tl) pf->tl[static_cast<size_t>(blockIdx.x) * 32 + (i)] = (v);      \
    } while (0)
#else
#define BITCOS_TL(i, v) \
    do {                \
    } while (0)
#endif

struct GroupedArgs {
    const bitcos_weights *experts;
    const int32_t *group_expert;
    const int32_t *group_begin;
    size_t ws_stride;          // workspace bytes per group
    int n_experts;
    int n_groups;
    int flat;                  // 1: one list of all groups' items, split evenly over the thread blocks
    int n_pairs;               // length of the pair list (outputs, pair_xrow)
    int n_xrows;               // rows of x
    const int32_t *n_groups_dev;   // NULL, or device word holding the number of groups (n_groups is then its upper bound)
};

// A group of a grouped product as its routing lists describe it; ok = false if the lists are
// malformed for it (its pairs outside the pair list, more tokens than the launch was sized for, an
// activation row outside x).  Such a group is skipped -- nothing of it is read or written -- and its
// status word and the launch's (word 0 of the first group's workspace) are set to 2.
struct GroupDesc {
    int e, begin, end;
    bool ok, empty;
};
__device__ __forceinline__ GroupDesc read_group(const GroupedArgs &ga, const int32_t *pair_xrow, unsigned int *status0, int grp,
                                                int nb_max) {
    GroupDesc d;
    d.e = __ldg(ga.group_expert + grp);
    d.begin = __ldg(ga.group_begin + grp);
    d.end = __ldg(ga.group_begin + grp + 1);
    d.empty = d.end <= d.begin;
    d.ok = d.e >= 0 && d.e < ga.n_experts && d.begin >= 0 && d.end <= ga.n_pairs && d.end - d.begin <= nb_max;
    if (d.ok && !d.empty)
        for (int i = d.begin; i < d.end; ++i) {
            const int r = __ldg(pair_xrow + i);
            if (r < 0 || r >= ga.n_xrows) d.ok = false;
        }
    if (!d.ok && !d.empty) {
        *reinterpret_cast<unsigned int *>(reinterpret_cast<uint8_t *>(status0) + static_cast<size_t>(grp) * ga.ws_stride) = 2u;
        *status0 = 2u;
    }
    return d;
}

inline int64_t padded_rows(int64_t M) { return (M + kRows - 1) / kRows * kRows; }

// Decoder warps per thread block: 20, or 14 for more than 8 tokens (the tensor-core path then holds
// 16 accumulators and 16 activation fragments per lane; with 20 warps it spills).
__host__ __device__ constexpr int decoder_warps(int batch) { return batch > 8 ? kWarps16 : kMaxWarps; }
// Threads of the widest block an instantiation for up to nb tokens is launched with.
__host__ __device__ constexpr int max_block_threads(int nb) { return (decoder_warps(nb) + 2) * 32; }

inline Plan make_plan(int64_t M, int64_t K, int max_warps_per_block, int tpw = 1) {
    const int G = static_cast<int>(K / kGroup);
    const int64_t RB = padded_rows(M) / kRows;
    Plan p{};
    p.tpw = tpw;
    const int max_warps = max_warps_per_block * tpw;       // tiles an item may hold
    const int blocks = (G + max_warps - 1) / max_warps;
    p.CG = (G + blocks - 1) / blocks;
    p.CS = (G + p.CG - 1) / p.CG;
    p.RBC = 1;
    if (p.CS == 1) {
        int64_t r = max_warps / p.CG;
        if (r > RB) r = RB;
        if (r < 1) r = 1;
        p.RBC = static_cast<int>(r);
    }
    p.NW = (p.CG * p.RBC + tpw - 1) / tpw;
    p.items = ((RB + p.RBC - 1) / p.RBC) * p.CS;
    return p;
}

// Several tiles per warp (BITCOS, two tokens and more): a warp takes tpw neighbouring groups of one row block and adds
// their sums in registers.
// The bits of a product must not depend on how many tiles its launch gives a warp (a launch of several products has
// more tiles than each of them), so both plans add in one order: runs of tpw groups inside a column block of the one-tile
// plan, the runs of a column block, the column blocks one after the other.  A wide item is therefore as many whole column
// blocks of the one-tile plan (sub groups, wsub warps each) as its warps hold.  At three tiles per warp the one-tile plan's
// column blocks are made a little uneven where that takes a warp less a row and lets an item hold two rows (20 groups: 11 and
// 9, seven warps, for 10 and 10, eight); and rows of more than 40 groups are cut by their own width instead, because fourteen
// warps hold only two such column blocks (200 groups would be eight items instead of five): their last bits may
// differ from the one-tile plan's.  own_order: a product that no launch of several takes (the 16-bit variant).
__host__ __device__ constexpr bool one_order(int G, int tpw) { return tpw == 2 || G <= 40; }
inline int row_warps(int G, int cg, int tpw) { return G / cg * ((cg + tpw - 1) / tpw) + (G % cg + tpw - 1) / tpw; }

// The one-tile plan of a product that other launches run with tpw tiles per warp.
inline Plan make_one_tile_plan(int64_t M, int64_t K, int max_warps, int tpw) {
    Plan p = make_plan(M, K, max_warps);
    const int G = static_cast<int>(K / kGroup), whole = (G + tpw - 1) / tpw;
    if (tpw != 3 || !one_order(G, tpw) || p.CS == 1) return p;
    int cg = p.CG;
    while (cg < max_warps && (row_warps(G, cg, tpw) > max_warps || max_warps / row_warps(G, cg, tpw) < max_warps / whole)) ++cg;
    p.CG = p.NW = cg;
    return p;
}

inline Plan make_run_plan(int64_t M, int64_t K, int max_warps, int tpw, bool own_order) {
    const int G = static_cast<int>(K / kGroup);
    const int64_t RB = padded_rows(M) / kRows;
    Plan p = make_plan(M, K, max_warps, tpw);
    if (own_order || !one_order(G, tpw)) {
        p.sub = p.CG;
        p.wsub = p.wrow = (p.CG + tpw - 1) / tpw;
    } else {
        p.sub = make_one_tile_plan(M, K, max_warps, tpw).CG;
        p.wsub = (p.sub + tpw - 1) / tpw;
        p.wrow = row_warps(G, p.sub, tpw);
    }
    if (p.CS == 1) {
        p.RBC = static_cast<int>(std::min<int64_t>(max_warps / p.wrow, RB));
        p.NW = p.RBC * p.wrow;
    } else if (p.sub < p.CG) {
        const int subs = (G + p.sub - 1) / p.sub, fit = max_warps / p.wsub, items = (subs + fit - 1) / fit, n = (subs + items - 1) / items;
        p.CG = n * p.sub;
        p.CS = (G + p.CG - 1) / p.CG;
        p.NW = p.wrow = n * p.wsub;
    }
    p.items = (RB + p.RBC - 1) / p.RBC * p.CS;
    return p;
}

// workspace: [0, 256) header (word 0 = status), arrival counters, partial sums
constexpr size_t kHeaderBytes = 256;
inline size_t counters_bytes(int64_t RB) { return static_cast<size_t>((RB * 4 + 255) / 256 * 256); }

inline size_t workspace_bytes_for(int64_t M, int64_t K) {
    const Plan p = make_plan(M, K, kWarps16);        // the plan with the most column blocks
    const int64_t RB = padded_rows(M) / kRows;
    size_t b = kHeaderBytes + counters_bytes(RB);
    if (p.CS > 1) b += static_cast<size_t>(RB) * p.CS * BITCOS_MAX_BATCH * kRows * sizeof(float);
    return b;
}

// Shared-memory layout of a thread block (byte offsets).
struct SmemLayout {
    uint32_t lut;        // lookup tables (0 bytes for 2-bit)
    uint32_t stage;      // stage 0
    uint32_t stage_bytes;
    uint32_t payload_cap, sign_cap, scale_cap, off_cap, x_cap;   // per-stage capacities
    uint32_t x;          // activations, [nb][K], if x_bytes != 0
    uint32_t x_bytes;    // 0: the activations do not fit and are read from global memory
    uint32_t red;        // 2 x [NW][NB][32] floats
    uint32_t scr;        // tensor-core path of the baselines: NW transposition buffers of kScrBytes
    uint32_t bar;        // mbarriers, then per-stage sign base words
    uint32_t total;
};

__host__ __device__ inline uint32_t align_up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }

// Partial-sum slots.  Up to two tokens: [warp][token][row] floats.  Tensor-core path:
// [warp][row][token], tokens fastest, so that a decoder lane stores its accumulator pairs (tokens
// 2c, 2c + 1) as one 8-byte word and the epilogue warp reads four tokens per load; token t of row r
// sits at position t ^ red_swizzle(r), which keeps both the stores (lane = row / 4-column pair) and
// the loads (lane = row) free of bank conflicts without padding.
template <int NB>
__host__ __device__ constexpr int red_swizzle(int row) {
    return NB < 8 ? 0 : ((row >> 2) & 1) * 4 + (NB > 8 ? ((row >> 1) & 1) * 8 : 0);
}

// Partial-sum slots between the decoder warps and the epilogue warp (how many items the
// decoders may run ahead of it).
__host__ __device__ constexpr int red_slots(int nbmax) { return nbmax <= 1 ? 8 : nbmax <= 2 ? 4 : 2; }

// Bytes from one token's activations to the next in shared memory (the 16 bytes on top keep two tokens'
// fragment loads off each other's banks).
__host__ __device__ constexpr int64_t x_stride(int64_t K) { return K + 16; }

// Which products decode their tiles in the tensor cores' fragment order (run_segments): BITCOS from two tokens on.
// (clocks per tile and multiprocessor, 18944 -> 56832 x 5120, rows -> fragments: 107 -> 121 with one token, which
// therefore keeps rows and dp4a; 148 -> 121 with two, 170 -> 133 with four, 186 -> 157 with eight, 268 -> 253 with
// sixteen; with two tiles per warp 115, 127, 137 and 206.)
__host__ __device__ constexpr bool fragment_order(int fmt, int nb) { return fmt == kBitcos && nb >= 2; }

// Tiles per warp in large launches (wants_two_tiles): two, or three with the fourteen decoder warps of more than eight tokens, which two
// tiles each would leave four of idle where rows have 20 or 40 groups (25600x5120 at sixteen tokens 27.1 -> 24.7 us).  At
// other lengths three tiles fill fewer warps (28 or 56 groups: 10 of 14, 22 or 43: 8); against one tile per warp they
// are faster at all of them (32000 tiles at sixteen tokens, rows of 14, 22, 28, 43 and 56 groups: 35.3 -> 27.4, 35.8 -> 29.2, 33.2 -> 26.7,
// 42.5 -> 32.9, 30.6 -> 26.9 us), two tiles per warp have not been measured there.
__host__ __device__ constexpr int wide_tiles(int fmt, int nb) { return fragment_order(fmt, nb) && nb > 8 ? 3 : 2; }

// The plan with one tile per warp.
inline Plan one_tile_plan(int fmt, int64_t M, int64_t K, int nb_template) {
    return make_one_tile_plan(M, K, decoder_warps(nb_template), wide_tiles(fmt, nb_template));
}

// scr: the tensor-core path passes its rows through transposition buffers
__host__ __device__ inline SmemLayout smem_layout(int fmt, const Plan &pl, int G, int nbmax, int64_t K, bool scr) {
    SmemLayout L{};
    uint32_t off = 0;
    L.lut = off;
    off += (fmt == kBit2) ? 0 : kLutBytes;
    const uint32_t tiles = static_cast<uint32_t>(pl.NW * pl.tpw);
    if (fmt == kBitcos) {
        L.payload_cap = tiles * 512;
        L.sign_cap = tiles * 512 + 64;
        L.off_cap = pl.tpw > 1 ? 192 : 128;   // the item's slice of tile_off (at most 21 or 43, + 3 + 3 words)
    } else if (fmt == kTrit5) {
        const uint32_t WPR = (26u * static_cast<uint32_t>(G) + 3) / 4;
        // whole rows when CS == 1, else at most CG groups (+1 shared word) of one row block
        L.payload_cap = (pl.CS == 1) ? static_cast<uint32_t>(pl.RBC) * WPR * 128
                                     : ((26u * static_cast<uint32_t>(pl.CG) + 3) / 4 + 1) * 128;
        L.sign_cap = 0;
    } else {
        L.payload_cap = tiles * 1024;
        L.sign_cap = 0;
    }
    L.scale_cap = tiles * 64;
    L.off_cap = align_up(L.off_cap, 16);
    L.x_cap = pl.x_in_stage ? static_cast<uint32_t>(nbmax * x_stride(K)) : 0u;
    L.stage = off;
    L.stage_bytes = align_up(L.payload_cap + L.sign_cap + L.scale_cap + L.off_cap + L.x_cap, 128);
    off += L.stage_bytes * static_cast<uint32_t>(pl.stages);
    L.x = off;
    // (the tensor-core path takes its activation fragments straight from global memory)
    L.x_bytes = (nbmax < kMmaMinBatch && !pl.x_in_stage && static_cast<int64_t>(nbmax) * K <= kXResidentBytes)
                    ? static_cast<uint32_t>(nbmax * x_stride(K)) : 0u;
    // (at least 128 bytes per decoder warp and token: the products that take 16-bit activations
    // quantise each warp's group into its own slice of this area)
    uint32_t x_area = L.x_bytes;
    if (L.x_bytes && x_area < static_cast<uint32_t>(pl.NW * nbmax * kGroup)) x_area = static_cast<uint32_t>(pl.NW * nbmax * kGroup);
    off += align_up(x_area, 128);
    L.red = off;
    // (several tiles per warp leave one partial sum, or with rows and dp4a two in half as many slots)
    off += static_cast<uint32_t>(red_slots(nbmax) * pl.NW * nbmax) * kRows * 4;
    L.scr = off;
    off += scr ? static_cast<uint32_t>(pl.NW) * kScrBytes : 0u;
    L.bar = off;
    off += 512;          // mbarriers, then (16-byte aligned) one 16-byte item descriptor per stage
    L.total = off;
    return L;
}

// ---------------------------------------------------------------------------------------------
// Device helpers.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float bf16_to_float(uint16_t b) { return __uint_as_float(static_cast<uint32_t>(b) << 16); }

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Bulk asynchronous copy global -> shared; size and both addresses are multiples of 16 bytes.
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
// Asks for a range of global memory to be brought into L2 (no destination, nothing to wait for);
// the address and the size are multiples of 16 bytes.
__device__ __forceinline__ void bulk_prefetch_l2(const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint64_t global_timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ uint32_t mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done;
}
// Polls until the phase completes, for at most limit_ns; false if it gave up.
__device__ __forceinline__ bool mbar_wait_limited(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
    uint64_t t0 = 0;
    for (uint32_t i = 0;; ++i) {
        if (mbar_try(bar, parity)) return true;
        if ((i & 15u) == 15u) {
            const uint64_t now = global_timer_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > limit_ns) return false;
        }
    }
}
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity) { return mbar_wait_limited(bar, parity, kWaitLimitNs); }
// Waits for the given phase parity (bounded); the common case, an already completed phase, costs
// one instruction.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try(bar, parity)) return true;
    return mbar_wait_slow(bar, parity);
}

// Four additions, packed in two instructions where that pays (with sixteen tokens pairs, and batches without guards, cost the
// 32B-model layer 103.5 -> 106 us, in the 16-bit variant 8192x5120 at four tokens 11.30 -> 11.40).
template <bool PACKED>
__device__ __forceinline__ float4 add_quads(float4 a, float4 b) {
    if (!PACKED) return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
    float4 c;
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%4, %5};\n\tmov.b64 y, {%8, %9};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t"
        "mov.b64 x, {%6, %7};\n\tmov.b64 y, {%10, %11};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%2, %3}, x;\n\t}"
        : "=f"(c.x), "=f"(c.y), "=f"(c.z), "=f"(c.w)
        : "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w));
    return c;
}

// Four 8x8 matrices of 16-bit elements from shared memory, one row address per lane: as int8 data
// this is exactly the A operand (16 rows x 32 bytes) of mma.m16n8k32.
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&a)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(addr)
                 : "memory");
}
// c[16 x 8] += a[16 x 32] * b[32 x 8], int8 operands, int32 accumulators.
__device__ __forceinline__ void mma_s8(int (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// c[16 x 8] += a[16 x 16] * b[16 x 8], bf16 operands, fp32 accumulators.
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void sts128(uint32_t addr, int a, int b, int c, int d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// ---------------------------------------------------------------------------------------------
// Tile decoders.  For the lane's row they produce the 32 int8x4 words of the row; the contraction
// follows as a separate step (dp4a per token, or the tensor cores from four tokens on).
// ---------------------------------------------------------------------------------------------

// int32 accumulator of one row (lane) and group against token activations xg[0..127] (shared memory).
template <int FMT>
__device__ __forceinline__ int contract(const int (&w)[32], const int4 *xg, int lane) {
    if (FMT == kBit2) {
        int a0 = 0, a1 = 0, a2 = 0, a3 = 0;
        // sum of the group's activations, needed because the stored code is weight + 1
        int sx = __dp4a(0x01010101, reinterpret_cast<const int *>(xg)[lane], 0);
        sx = __reduce_add_sync(0xFFFFFFFFu, sx);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int4 xq = xg[q];
            a0 = dp4a_us(static_cast<uint32_t>(w[4 * q + 0]), xq.x, a0);
            a1 = dp4a_us(static_cast<uint32_t>(w[4 * q + 1]), xq.y, a1);
            a2 = dp4a_us(static_cast<uint32_t>(w[4 * q + 2]), xq.z, a2);
            a3 = dp4a_us(static_cast<uint32_t>(w[4 * q + 3]), xq.w, a3);
        }
        return a0 + (a1 >> 2) + (a2 >> 4) + (a3 >> 6) - sx;
    } else {
        int a0 = 0, a1 = 0, a2 = 0, a3 = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int4 xq = xg[q];
            a0 = __dp4a(w[4 * q + 0], xq.x, a0);
            a1 = __dp4a(w[4 * q + 1], xq.y, a1);
            a2 = __dp4a(w[4 * q + 2], xq.z, a2);
            a3 = __dp4a(w[4 * q + 3], xq.w, a3);
        }
        return (a0 + a1) + (a2 + a3);
    }
}

// Activation quantiser arithmetic (used by the quantiser kernels and by the products that take
// 16-bit activations): a = max(max |x| over the group, 2^-100), scale = a / 127,
// code = rint(x * (127 / a)), IEEE float32 quotient and product, ties to even.
constexpr float kAmaxFloor = 7.888609052210118e-31f;      // 2^-100

__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t quant_code(float x, float inv) {
    int c = __float2int_rn(__fmul_rn(x, inv));
    c = c > 127 ? 127 : (c < -127 ? -127 : c);
    return static_cast<uint32_t>(c) & 0xFFu;
}
// the two values of a 32-bit word -> two codes in the low 16 bits
__device__ __forceinline__ uint32_t quant_pair(uint32_t u, float inv) {
    return quant_code(bf16_lo(u), inv) | (quant_code(bf16_hi(u), inv) << 8);
}

// ---------------------------------------------------------------------------------------------
// The persistent, staged kernel body.
// ---------------------------------------------------------------------------------------------

// Items are numbered row-block chunk major, column block minor: item = c * CS + cs.  A thread
// block owns a CONTIGUOUS range of items (balanced split of all items over the grid), so it
// streams a contiguous piece of the packed matrix and usually sees all column blocks of a row
// block itself; only the row blocks cut by a range boundary need the cross-block protocol.
struct Walk {
    int first, count;   // this block's first item and number of items
    int cstride;        // chunk stride after the last column block of a chunk (1 = contiguous range)
    int q, rem;         // contiguous mode: blocks 0 .. rem-1 own q + 1 items, the others q
};

// Two ways to hand items to thread blocks.  Cyclic: block b takes chunks b, b + n, b + 2n, ...
// with all their column blocks (no row block is ever shared; all blocks read neighbouring
// addresses at any time).  Contiguous: a balanced split of the item list (perfect balance when
// there are few chunks per block, at the price of sharing the row blocks cut by a boundary).
__host__ __device__ __forceinline__ Walk make_walk(const Plan &pl, int block, int n_blocks) {
    Walk w;
    const int items = static_cast<int>(pl.items);
    if (pl.cyclic) {
        const int chunks = items / pl.CS;
        w.first = block * pl.CS;
        w.count = block < chunks ? ((chunks - block + n_blocks - 1) / n_blocks) * pl.CS : 0;
        w.cstride = n_blocks;
        w.q = 1;
        w.rem = 0;
        return w;
    }
    w.q = items / n_blocks;
    w.rem = items - w.q * n_blocks;
    w.first = block * w.q + (block < w.rem ? block : w.rem);
    w.count = w.q + (block < w.rem ? 1 : 0);
    w.cstride = 1;
    return w;
}

// This block's walk: from the launch's table if there is one, else computed here.
__device__ __forceinline__ Walk block_walk(const FirstOff &fo, int index, const Plan &pl, int block, int n_blocks) {
    if (!fo.walks) return make_walk(pl, block, n_blocks);
    Walk w;
    w.first = fo.first[index];
    w.count = fo.count[index];
    w.cstride = pl.cyclic ? n_blocks : 1;
    w.q = pl.wq;
    w.rem = pl.wrem;
    return w;
}

// Which thread block owns an item in contiguous mode (inverse of the split above).
__device__ __forceinline__ int owner_of(const Walk &w, int item) {
    const int big = w.rem * (w.q + 1);
    if (item < big) return item / (w.q + 1);
    return w.rem + (item - big) / w.q;
}

struct ItemRange {
    int rb0;         // first row block
    int cs;          // column block
    int g0;          // first group
    int nt;          // tiles (= busy warps)
    int64_t t0;      // first tile
};

__host__ __device__ __forceinline__ ItemRange item_range(const Problem &pr, const Plan &pl, int c, int cs) {
    ItemRange r;
    r.rb0 = c * pl.RBC;
    r.cs = cs;
    r.g0 = cs * pl.CG;
    if (pl.CS == 1) {
        int nrb = pr.RB - r.rb0;
        if (nrb > pl.RBC) nrb = pl.RBC;
        r.nt = nrb * pr.G;
    } else {
        r.nt = pr.G - r.g0 < pl.CG ? pr.G - r.g0 : pl.CG;
    }
    r.t0 = static_cast<int64_t>(r.rb0) * pr.G + r.g0;
    return r;
}

// (chunk, column block) of an item, and the step to the next item, without divisions in loops
struct ItemIter {
    int c, cs;
    __host__ __device__ __forceinline__ void init(const Plan &pl, int item) {
        if (pl.CS == 1) { c = item; cs = 0; }
        else { c = item / pl.CS; cs = item - c * pl.CS; }
    }
    __host__ __device__ __forceinline__ void next(const Plan &pl, const Walk &w) {
        if (++cs == pl.CS) { cs = 0; c += w.cstride; }
    }
};

// What differs between the segments of one launch (everything else -- shape, activations,
// outputs -- is read from the launch's one Problem), behind accessors: the plain kernels read the
// values from the kernel parameters every time (no registers spent on them), the grouped launch
// holds the current group's values.
struct ParamView {
    __device__ __forceinline__ const uint32_t *payload(const Problem &p) const { return p.payload; }
    __device__ __forceinline__ const uint32_t *signs(const Problem &p) const { return p.signs; }
    __device__ __forceinline__ const uint32_t *tile_off(const Problem &p) const { return p.tile_off; }
    __device__ __forceinline__ const uint16_t *scales(const Problem &p) const { return p.scales; }
    __device__ __forceinline__ const int32_t *xrow(const Problem &p) const { return p.xrow; }       // NULL: token b reads row b
    __device__ __forceinline__ unsigned int *status(const Problem &p) const { return p.status; }
    __device__ __forceinline__ int64_t out_row0(const Problem &p) const { return p.out_row0; }      // first output row of token 0
    __device__ __forceinline__ int nb(const Problem &p) const { return p.nb; }                      // tokens of the segment
};
struct GroupView {
    const uint32_t *payload_, *signs_, *tile_off_;
    const uint16_t *scales_;
    const int32_t *xrow_;
    unsigned int *status_;
    int begin_, nb_;
    __device__ __forceinline__ const uint32_t *payload(const Problem &) const { return payload_; }
    __device__ __forceinline__ const uint32_t *signs(const Problem &) const { return signs_; }
    __device__ __forceinline__ const uint32_t *tile_off(const Problem &) const { return tile_off_; }
    __device__ __forceinline__ const uint16_t *scales(const Problem &) const { return scales_; }
    __device__ __forceinline__ const int32_t *xrow(const Problem &) const { return xrow_; }
    __device__ __forceinline__ unsigned int *status(const Problem &) const { return status_; }
    __device__ __forceinline__ int64_t out_row0(const Problem &) const { return begin_; }
    __device__ __forceinline__ int nb(const Problem &) const { return nb_; }
};

// Issues the bulk copies of one item into stage `s` (one thread) and publishes the item's
// descriptor (sign_base[4s .. 4s+3]; word 3 = index of the first sign bit held in the stage).  o_lo / o_hi: sign-vector
// positions of the item's first tile and of the tile after its last (BITCOS only).
template <int FMT, typename View>
__device__ __forceinline__ void issue_item(const Problem &pb, const View &pr, const Plan &pl, const ItemRange &r,
                                           const SmemLayout &L, uint8_t *smem, int s, uint32_t *sign_base, uint32_t o_lo,
                                           uint32_t o_hi, const int (&xrows)[2], unsigned long long *tl = nullptr) {
#ifdef BITCOS_TIMELINE
#define BITCOS_TLI(i) do { if (tl) tl[i] = clock64(); } while (0)
#else
#define BITCOS_TLI(i) do { } while (0)
#endif
    BITCOS_TLI(21);
    uint8_t *stage = smem + L.stage + static_cast<uint32_t>(s) * L.stage_bytes;
    const uint32_t bar = smem_addr(smem + L.bar) + 8u * static_cast<uint32_t>(s);
    const uint32_t d_payload = smem_addr(stage);
    const uint32_t d_signs = d_payload + L.payload_cap;
    const uint32_t d_scales = d_signs + L.sign_cap;
    const uint32_t scale_bytes = static_cast<uint32_t>(r.nt) * 64u;
    const uint8_t *g_scales = reinterpret_cast<const uint8_t *>(pr.scales(pb)) + r.t0 * 64;
    // what the decoder warps need to know about the item (read by them once the stage is full)
    sign_base[s * 4 + 0] = static_cast<uint32_t>(r.nt) | (static_cast<uint32_t>(r.t0 & 3) << 8);
    sign_base[s * 4 + 1] = static_cast<uint32_t>(r.g0);
    sign_base[s * 4 + 2] = static_cast<uint32_t>(r.rb0);
    const uint32_t x_bytes = pl.x_in_stage ? static_cast<uint32_t>(pr.nb(pb)) * static_cast<uint32_t>(pb.K) : 0u;
    // (issued after the format's expect_tx below; a grouped launch only)
    auto copy_x = [&]() {
        // the activation rows of this group's tokens (from L2): the decoders of a grouped launch
        // find them next to the weights and need no block-wide staging step per group
        if (pl.x_in_stage)
            for (int b = 0; b < pr.nb(pb) && b < 2; ++b)
                bulk_copy(d_scales + L.scale_cap + L.off_cap + static_cast<uint32_t>(b) * static_cast<uint32_t>(x_stride(pb.K)),
                          pb.x + static_cast<int64_t>(xrows[b]) * pb.K, static_cast<uint32_t>(pb.K), bar);
    };
    if (FMT == kBitcos) {
        const uint32_t b_lo = (o_lo >> 7) << 4, b_hi = ((o_hi + 127u) >> 7) << 4;
        const uint32_t sign_bytes = b_hi - b_lo;
        const uint32_t bm_bytes = static_cast<uint32_t>(r.nt) * 512u;
        sign_base[s * 4 + 3] = b_lo * 8u;
        // the tiles' entry offsets: the 16-byte aligned slice of tile_off that covers t0 .. t0 + nt
        const uint32_t o_first = static_cast<uint32_t>(r.t0 & 3);
        const uint32_t off_bytes = ((o_first + static_cast<uint32_t>(r.nt) + 1u + 3u) & ~3u) * 4u;
        BITCOS_TLI(22);
        mbar_expect_tx(bar, bm_bytes + sign_bytes + scale_bytes + off_bytes + x_bytes);
        BITCOS_TLI(23);
        copy_x();
        bulk_copy(d_scales + L.scale_cap, pr.tile_off(pb) + (r.t0 - o_first), off_bytes, bar);
        BITCOS_TLI(24);
        bulk_copy(d_payload, reinterpret_cast<const uint8_t *>(pr.payload(pb)) + r.t0 * 512, bm_bytes, bar);
        BITCOS_TLI(25);
        if (sign_bytes) bulk_copy(d_signs, reinterpret_cast<const uint8_t *>(pr.signs(pb)) + b_lo, sign_bytes, bar);
        BITCOS_TLI(26);
        bulk_copy(d_scales, g_scales, scale_bytes, bar);
        BITCOS_TLI(27);
    } else if (FMT == kTrit5) {
        const int64_t WPR = (26 * static_cast<int64_t>(pb.G) + 3) / 4;
        const int64_t w_lo = r.rb0 * WPR + ((26 * r.g0) >> 2);
        int64_t w_hi;   // exclusive
        if (pl.CS == 1) w_hi = (r.rb0 + r.nt / pb.G) * WPR;
        else w_hi = r.rb0 * WPR + ((26 * (r.g0 + r.nt) - 1) >> 2) + 1;
        const uint32_t bytes = static_cast<uint32_t>(w_hi - w_lo) * 128u;
        mbar_expect_tx(bar, bytes + scale_bytes + x_bytes);
        copy_x();
        bulk_copy(d_payload, reinterpret_cast<const uint8_t *>(pr.payload(pb)) + w_lo * 128, bytes, bar);
        bulk_copy(d_scales, g_scales, scale_bytes, bar);
    } else {
        const uint32_t bytes = static_cast<uint32_t>(r.nt) * 1024u;
        mbar_expect_tx(bar, bytes + scale_bytes + x_bytes);
        copy_x();
        bulk_copy(d_payload, reinterpret_cast<const uint8_t *>(pr.payload(pb)) + r.t0 * 1024, bytes, bar);
        bulk_copy(d_scales, g_scales, scale_bytes, bar);
    }
}

// mbarrier slots inside the `bar` region (8 bytes each)
constexpr int kBarFull = 0;                       // [stages] stage filled by the copy engine
constexpr int kBarEmpty = kMaxStages;             // [stages] stage released (by the epilogue warp, once all decoder warps have posted the item's sums)
constexpr int kBarRedFull = 2 * kMaxStages;       // [slots] partial sums of an item written by all decoder warps
constexpr int kBarRedEmpty = 2 * kMaxStages + 8;  // [slots] partial sums consumed by the epilogue warp
constexpr int kBarLut = 2 * kMaxStages + 16;      // lookup table arrived
constexpr int kBarX = 2 * kMaxStages + 17;        // activations arrived in shared memory (plain kernels, 1-2 tokens)

// Arrival by lane 0 only, as one predicated instruction (no divergent branch around it).
__device__ __forceinline__ void mbar_arrive_lane0(uint32_t bar, int lane) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.eq.s32 p, %1, 0;\n\t"
        "@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(bar), "r"(lane)
        : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// A row block whose column blocks were split over several thread blocks: this block's share.
struct Share {
    int rb;             // row block
    int slot;           // position of this block among the sharers (= order of summation)
    int sharers;        // number of thread blocks holding a piece of the row block
    unsigned int old;   // value of the arrival counter before this block's arrival
};

// If this block's arrival was the last one: add the shares in slot order and write the outputs.
template <int NB, bool XG, bool BL>
__device__ __forceinline__ void finish_share(const Problem &pr, const Plan &pl, const int (&xr)[NB], const Share &sh,
                                             int lane) {
    const unsigned int old = __shfl_sync(0xFFFFFFFFu, sh.old, 0);
    if (old != static_cast<unsigned int>(sh.sharers - 1)) return;
    __threadfence();
    const int64_t m = static_cast<int64_t>(sh.rb) * kRows + lane;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        if (b < pr.nb) {
            float tot = 0.f;
            for (int j = 0; j < sh.sharers; ++j)
                tot += __ldcg(pr.partial + ((static_cast<int64_t>(sh.rb) * pl.CS + j) * pr.nb + b) * kRows + lane);
            if (m < pr.M) pr.y[(pr.out_row0 + b) * pr.M + m] = BL ? kBf16WeightInverse * tot : XG ? tot : __ldg(pr.x_scale + xr[b]) * tot;
        }
    }
    if (lane == 0) pr.counters[sh.rb] = 0u;    // leave the counter ready for the next call
}

// What a thread block runs back to back: one problem and its share of the items (the plain
// kernels), or the pieces of several groups (the grouped launch).  Every warp role walks its own
// copy of the source.
template <bool DEBUG, bool XG = false, bool XQ = false, bool BL = false>
struct OneSegT {
    typedef ParamView View;
    static constexpr bool kSingle = true;      // never more than one segment
    static constexpr bool kHetero = false;     // all segments share one problem shape and one plan
    static constexpr bool kListsLate = false;  // (no routing lists)
    static constexpr bool kDebug = DEBUG;      // false: acc_debug is known to be NULL (no code for it)
    static constexpr bool kGroupScales = XG;   // x_scale holds one scale per token AND group: [nb][G]
    static constexpr bool kQuantize = XQ;      // x holds bf16 activations: quantised per group of 128 by the decoder warps
    static constexpr bool kBlend = BL;         // x holds bf16 activations, used as they are against weights +-s (tensor cores)
    const Problem *pr;
    Walk wk;
    bool used;
    __device__ __forceinline__ const Problem &shape() const { return *pr; }
    __device__ __forceinline__ int block_in_job(int block) const { return block; }
    __device__ __forceinline__ bool next(View &v, Walk &w) {
        if (used) return false;
        used = true;
        (void)v;
        w = wk;
        return true;
    }
};

// This block's share of the arrays a later launch will read, requested into L2: entries first,
// first + step, ...
__device__ __forceinline__ void prefetch_share(const PrefetchList *pf, int first, int step) {
    const uint32_t nblk = gridDim.x, bid = blockIdx.x;
    for (int i = first; i < pf->n; i += step) {
        const uint32_t total = pf->bytes[i];
        const uint32_t chunk = ((total / 16u + nblk - 1u) / nblk) * 16u;
        const uint32_t off = bid * chunk;
        if (off < total) bulk_prefetch_l2(pf->ptr[i] + off, total - off < chunk ? total - off : chunk);
    }
}

// Warp roles: warps 0 .. NW-1 decode one tile per item each; warp NW adds the decoders' partial
// sums in a fixed order and writes the outputs (and runs the cross-block protocol); the block's
// LAST warp (known without reading a kernel argument) feeds the stage ring with bulk copies.  The roles meet only through mbarriers, every
// wait is bounded, and there is no block-wide barrier inside the loop.
// `segs` yields the problems this block works on, one after the other, with its share of each
// one's items; the stage ring, the partial-sum slots and their barriers run on across them.
template <int FMT, int NB, int TPW, typename Segs>
__device__ __forceinline__ void run_segments(const Segs &segs, const Plan &pl_in, uint8_t *smem, int block,
                                             const FirstOff *fo = nullptr, int fo_index = 0, const PrefetchList *pf = nullptr,
                                             bool first_sent = false) {
    // first_sent: the caller has already initialised the barriers of stage 0 and of the lookup table
    // and issued the table's copy and the copies of this block's first item (send_first_copies)
    // (through a shuffle, so that what depends on it is in uniform registers; not with sixteen tokens, 170.5 -> 174 clocks per tile;
    // the 16-bit variant gains nothing)
    const int warp = NB > 8 || Segs::kBlend ? static_cast<int>(threadIdx.x >> 5) : __shfl_sync(0xFFFFFFFFu, static_cast<int>(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int prod_warp = static_cast<int>(blockDim.x >> 5) - 1;      // the producer: always the block's last warp
    if (static_cast<int>(threadIdx.x) == prod_warp * 32) BITCOS_TL(16, clock64());
    // The problem and the plan of the segment a warp role is working on.  The plain and the grouped
    // launches have one shape and one plan for all their segments.  A phased launch (kHetero) moves
    // from job to job: only what the shared-memory layout and the barrier counts need -- the widest
    // plan, the longest row -- is common (pl_in, segs.shape()), and every role re-binds pb / pl to its
    // own copy of the current job's problem and plan.
    const Problem *pbp = &segs.shape();
    const Plan *plp = &pl_in;
#define pb (*pbp)
#define pl (*plp)
    constexpr bool kFrag = fragment_order(FMT, NB);
    const SmemLayout L = smem_layout(FMT, pl, segs.shape().G, NB, segs.shape().K, NB >= kMmaMinBatch && !kFrag);
    typename Segs::View pr{};
    Walk wk{};
    const uint8_t *lut = smem + L.lut;
    float *red = reinterpret_cast<float *>(smem + L.red);
    // per stage: {tiles | (first tile & 3) << 8, first group, first row block, first sign bit held}
    uint32_t *sign_base = reinterpret_cast<uint32_t *>(smem + L.bar + 384);
    const uint32_t bar0 = smem_addr(smem + L.bar);
    static_assert(TPW == 1 || kFrag || (TPW == 2 && NB < kMmaMinBatch), "several tiles per warp: fragment order, or one or two tokens");
    constexpr bool kPairs = kFrag && TPW > 1;                  // one partial sum per warp, not per tile
    // one activation scale per token and group (applied by the decoder warps, tile by tile)
    // instead of one per token (applied by the epilogue warp to the finished sums)
    constexpr bool kXQ = Segs::kQuantize;                      // (one or two tokens only)
    constexpr bool kBlend = Segs::kBlend;                      // (tensor-core path, up to eight tokens)
    static_assert(!kBlend || ((NB == 4 || NB == 8) && FMT == kBitcos), "16-bit weights: the four- and eight-token BITCOS kernels");
    constexpr bool kXG = Segs::kGroupScales || kXQ || kBlend;   // no token scale in the epilogue
    static_assert(!kXQ || NB < kMmaMinBatch, "16-bit activations: one or two tokens only");
    const uint32_t red_slot = static_cast<uint32_t>(kPairs ? pl.NW : pl.NW * TPW) * NB * kRows;     // floats per partial-sum slot
    // partial-sum slots in use: red_slots(NB), half as many (of twice the size) where a warp leaves two tiles' sums
    constexpr int rs_log2 = (red_slots(NB) == 8 ? 3 : red_slots(NB) == 4 ? 2 : 1) - (kPairs ? 0 : TPW - 1);
    constexpr int rs_mask = (1 << rs_log2) - 1;

    // Programmatic dependent launch: the next kernel in the stream may be scheduled as soon as
    // every block of this one got here; whatever it reads from us it reads after its own
    // griddepcontrol.wait.
    // (every thread: a trigger from one warp alone measured 0.02 us per layer pass faster, which is not worth
    // depending on how a block's trigger is counted)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // A block launched wider than this problem needs (several problems in one launch): the spare
    // warps only take part in the one block-wide barrier.
    if (warp > pl.NW && warp < prod_warp) {
        __syncthreads();
        return;
    }

    // ------------------------------------------------------------------ producer warp
    // It also sets the barriers up, so that the first copies are in flight before anything else
    // happens in the block.
    if (warp == prod_warp) {
        if (lane == 0) {
            BITCOS_TL(13, clock64());
            BITCOS_TL(0, global_timer_ns());
            BITCOS_TL(17, clock64());
        }
        // All 33 barrier slots at once, one per lane (slots of unused stages included): slots
        // kBarRedFull .. kBarRedFull + 7 count the decoder warps, the others one arrival.  Every
        // barrier is initialised and fenced before the first asynchronous copy is issued.
        static_assert(kBarFull == 0 && kBarEmpty == 8 && kBarRedFull == 16 && kBarRedEmpty == 24 && kBarLut == 32,
                      "one barrier slot per lane, plus the table's");
        if (!(first_sent && lane == kBarFull))
            mbar_init(bar0 + 8u * static_cast<uint32_t>(lane), (lane >= kBarRedFull && lane < kBarRedEmpty) ? pl.NW : 1);
        if (lane == 0 && !first_sent) mbar_init(bar0 + 8u * kBarLut, 1);
        if (lane == 1) mbar_init(bar0 + 8u * kBarX, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        __syncwarp();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // the other lanes' barriers, seen by this lane's copies
        if (lane == 0) BITCOS_TL(14, clock64());
        // The first copies go out before the block-wide barrier below, while the other warps are
        // still fetching the activations.
        // Entry offsets are requested two items before they are needed (r0 = item k, r1 = item
        // k + 1, r2 = item k + 2), so that the load is never waited for.
        Segs src = segs;
        if constexpr (Segs::kHetero) {
            pbp = src.problem_ptr();
            plp = src.plan_ptr();
        }
        ItemIter it2;
        ItemRange r0{}, r1{}, r2{};
        uint32_t lo0 = 0, hi0 = 0, lo1 = 0, hi1 = 0;
        int k0 = 0, ps = 0;
        int kk = 0;                // items issued so far, over all segments
        int xrows[2] = {0, 0};     // activation rows of the segment's tokens (when they travel with the stage)
        uint32_t pphase = 1;       // parity of the phase before the one the decoders complete next
        bool ok = true;
        auto offsets = [&](const ItemRange &r, uint32_t &lo, uint32_t &hi) {
            if (FMT != kBitcos) return;
            // two independent loads (no reuse of the previous item's upper offset: that would make
            // every request wait for the one before it)
            lo = __ldg(pr.tile_off(pb) + r.t0);
            hi = __ldg(pr.tile_off(pb) + r.t0 + r.nt);
        };
        auto second_item = [&]() {
            if (wk.count > 1) {
                it2.next(pl, wk);
                r1 = item_range(pb, pl, it2.c, it2.cs);
                offsets(r1, lo1, hi1);
            }
        };
        auto issue_loop = [&](int k_end) {
            for (int k = k0; k < k_end; ++k, ++kk) {
                const int s = ps;
                uint32_t lo2 = 0, hi2 = 0;
                // (the block's very first item goes out before anything is worked out for the items after it)
                auto look_ahead = [&]() {
                    if (k + 2 < wk.count) {
                        it2.next(pl, wk);
                        r2 = item_range(pb, pl, it2.c, it2.cs);
                        offsets(r2, lo2, hi2);
                    }
                };
                if (kk != 0) look_ahead();
                if (kk >= pl.stages) {
                    if (!mbar_wait(bar0 + 8u * (kBarEmpty + s), pphase)) {
                        if (pr.status(pb)) *pr.status(pb) = 1u;
                        ok = false;
                        return;
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                }
                if (!(first_sent && kk == 0)) {
#ifdef BITCOS_TIMELINE
                    issue_item<FMT>(pb, pr, pl, r0, L, smem, s, sign_base, lo0, hi0, xrows,
                                    (kk == 0 && pf && pf->tl) ? pf->tl + static_cast<size_t>(blockIdx.x) * 32 : nullptr);
#else
                    issue_item<FMT>(pb, pr, pl, r0, L, smem, s, sign_base, lo0, hi0, xrows);
#endif
                }
                if (kk == 0) {
                    second_item();
                    look_ahead();
                }
                r0 = r1; lo0 = lo1; hi0 = hi1;
                r1 = r2; lo1 = lo2; hi1 = hi2;
                if (++ps == pl.stages) {
                    ps = 0;
                    pphase ^= 1u;
                }
            }
            k0 = k_end;
        };
        // first item(s) of a segment: ranges and entry offsets of items 0 and 1 (the block's first
        // segment: of item 0 only; item 1 follows once item 0 is on its way)
        auto prime = [&](bool first_segment) {
            k0 = 0;
            it2.init(pl, wk.first);
            r0 = item_range(pb, pl, it2.c, it2.cs);
            if (FMT == kBitcos) {
                if (first_segment && fo && fo->valid) {
                    lo0 = fo->lo[fo_index];
                    hi0 = fo->hi[fo_index];
                } else {
                    lo0 = __ldg(pr.tile_off(pb) + r0.t0);
                    hi0 = __ldg(pr.tile_off(pb) + r0.t0 + r0.nt);
                }
            }
            if (!first_segment) second_item();
            if (pl.x_in_stage) {
                xrows[0] = pr.xrow(pb) ? __ldg(pr.xrow(pb)) : 0;
                xrows[1] = pr.nb(pb) > 1 ? (pr.xrow(pb) ? __ldg(pr.xrow(pb) + 1) : 1) : 0;
            }
        };
        // A grouped launch reads its routing lists (which may come from the previous kernel in the
        // stream) to find its first item: the table copy, which depends on nothing, goes out before
        // the wait for that kernel.
        bool lut_issued = first_sent;
        if constexpr (Segs::kListsLate) {
            if (lane == 0 && FMT != kBit2) {
                mbar_expect_tx(bar0 + 8u * kBarLut, kLutBytes);
                bulk_copy(smem_addr(smem + L.lut), Segs::kBlend ? g_bitcos_bf16_lut.v : FMT == kBitcos ? g_bitcos_lut.v : g_trit5_lut.v, kLutBytes,
                          bar0 + 8u * kBarLut);
                lut_issued = true;
            }
            asm volatile("griddepcontrol.wait;" ::: "memory");
        }
        bool have = src.next(pr, wk);
        while (have && wk.count <= 0) have = src.next(pr, wk);
        // The lookup table first: it is the largest transfer of the start-up (64 KB from L2) and
        // needs no address arithmetic.
        if (lane == 0 && have && FMT != kBit2 && !lut_issued) {
            mbar_expect_tx(bar0 + 8u * kBarLut, kLutBytes);
            bulk_copy(smem_addr(smem + L.lut), Segs::kBlend ? g_bitcos_bf16_lut.v : FMT == kBitcos ? g_bitcos_lut.v : g_trit5_lut.v, kLutBytes,
                      bar0 + 8u * kBarLut);
        }
        if (lane == 0) BITCOS_TL(15, clock64());
        // Only the first item goes out before the block-wide barrier: issuing a bulk copy costs this
        // thread on the order of a hundred nanoseconds, and the other warps wait at that barrier.
        // (first item already sent by the kernel's first instructions: its bookkeeping waits until
        // the other warps have been let through the block-wide barrier)
        if (lane == 0 && have && !first_sent) {
            prime(true);
            BITCOS_TL(18, clock64());
            issue_loop(1);
        }
        if (lane == 0) BITCOS_TL(2, clock64());
        __syncthreads();       // pairs with the barrier the other warps reach after staging the activations
        if (lane == 0) BITCOS_TL(12, clock64());
        if (lane == 0 && have && first_sent) {
            prime(true);
            issue_loop(1);
        }
        if (lane == 0 && !have && lut_issued && !first_sent) mbar_wait(bar0 + 8u * kBarLut, 0);      // no copy may outlive the block
        // The hint for a later launch goes out behind this block's own first copies (as many as the
        // ring holds): measured, requests issued before them or from another warp gain less.
        if (pf && lane == 0) {
            if (have && ok) issue_loop(wk.count < pl.stages ? wk.count : pl.stages);
            prefetch_share(pf, 0, 1);
        }
        if (lane != 0 || !have) return;
        if (ok) issue_loop(wk.count);
        while (!Segs::kSingle && ok && src.next(pr, wk)) {
            if (wk.count <= 0) continue;
            prime(false);
            issue_loop(wk.count);
        }
        return;
    }

    // What may depend on the previous kernel in the stream: activations, routing lists, outputs,
    // workspace.  The packed weights do not, so the producer never waits, and in the plain kernels
    // with one or two tokens (kEarly) the decoder warps do not either until they have decoded
    // their first tile: only the contraction needs the activations, which the epilogue warp
    // fetches into shared memory (one bulk copy per token) as soon as the dependency is resolved.
    // With four tokens and more (tensor-core path) the decoders fetch their activation fragments
    // from global memory right after that first decode instead.
    constexpr bool kLate = Segs::kSingle || Segs::kHetero;      // plain and phased kernels: wait as late as possible
    constexpr bool kEarly = kLate && NB < kMmaMinBatch;         // ... and activations copied by the epilogue warp
    if (!kLate) asm volatile("griddepcontrol.wait;" ::: "memory");

    Segs src = segs;
    if constexpr (Segs::kHetero) {
        pbp = src.problem_ptr();
        plp = src.plan_ptr();
    }
    bool have = src.next(pr, wk);
    while (have && wk.count <= 0) have = src.next(pr, wk);
    auto next_segment = [&]() {
        if (Segs::kSingle) return false;
        bool more = src.next(pr, wk);
        while (more && wk.count <= 0) more = src.next(pr, wk);
        return more;
    };

    // activations of one or two tokens: kept whole in shared memory ([nb][K]), staged by these
    // warps while the producer starts the copies (plain kernels: one segment), or delivered with
    // every stage (grouped launch); the tensor-core path reads its fragments from global memory
    int xr[NB];
    auto token_rows = [&]() {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int bb = b < pr.nb(pb) ? b : 0;
            xr[b] = pr.xrow(pb) ? __ldg(pr.xrow(pb) + bb) : bb;
        }
    };
    if (have && !kLate) token_rows();
    const bool x_resident = L.x_bytes != 0;
    if (x_resident && have && !kEarly) {
        int4 *xs = reinterpret_cast<int4 *>(smem + L.x);
        const int per_tok = static_cast<int>(pb.K / 16);
        const int nthr = (pl.NW + 1) * 32;                   // the decoder warps and the epilogue warp
        const int tid = threadIdx.x;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            if (b < pr.nb(pb)) {
                const int4 *src = reinterpret_cast<const int4 *>(pb.x + static_cast<int64_t>(xr[b]) * pb.K);
                for (int q = tid; q < per_tok; q += nthr) xs[b * (per_tok + 1) + q] = __ldg(src + q);
            }
        }
    }
    __syncthreads();          // barriers initialised, activations in place
    if (!have) return;

    // ------------------------------------------------------------------ epilogue warp
    if (warp == pl.NW) {
        // the segment's activations into shared memory: one bulk copy per token (one or two tokens)
        auto fetch_x = [&]() {
            token_rows();
            if (kEarly && !kXQ && lane == 0) {
                mbar_expect_tx(bar0 + 8u * kBarX, static_cast<uint32_t>(pr.nb(pb)) * static_cast<uint32_t>(pb.K));
#pragma unroll
                for (int b = 0; b < NB; ++b)
                    if (b < pr.nb(pb))
                        bulk_copy(smem_addr(smem + L.x) + static_cast<uint32_t>(b) * static_cast<uint32_t>(x_stride(pb.K)),
                                  pb.x + static_cast<int64_t>(xr[b]) * pb.K, static_cast<uint32_t>(pb.K), bar0 + 8u * kBarX);
            }
        };
        if (kLate) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            if (lane == 0) BITCOS_TL(8, clock64());
            if (!Segs::kHetero) fetch_x();
        }
        float run[NB];          // running sum of the current row block over this block's items
#pragma unroll
        for (int b = 0; b < NB; ++b) run[b] = 0.f;
        // per-token activation scales, fetched once per segment (sixteen: a cached load per output block)
        constexpr bool kHoldScales = !kXG && NB <= 8;
        float xsc[kHoldScales ? NB : 1] = {};
        auto xscale = [&](int b) { return kBlend ? kBf16WeightInverse : kXG ? 1.f : kHoldScales ? xsc[kHoldScales ? b : 0] : __ldg(pb.x_scale + xr[b]); };
        Share pend[2];
        int n_pend = 0;
        ItemIter it;
        int kk = 0;             // items consumed so far, over all segments
        int es = 0;             // stage of the item the epilogue looks at next
        // The sums of n tiles, in an order that depends on n alone: neighbours first (with sixteen tokens neighbouring threes),
        // which is what a warp with several tiles has added up already (kPairs; see make_run_plan).  This one warp serves
        // every row block of the launch at the few issue slots the decoders leave it (one in six clocks or so), and with short
        // rows they come fast (six tiles a row block at K = 768): what counts there is its instructions, with long rows its latency at
        // the end of a launch.  Clocks per tile and multiprocessor at eight tokens against twenty guarded loads a sum and
        // a scale fetched per output: K = 768 300 -> 182, K = 2048 180 -> 148, K = 2560 163 -> 145.
        // Up to two tokens (spaced NB * 32 floats apart): a tree of pairs, all loads before the first addition.
        auto tree = [&](auto size, const float *base, int n) {
            constexpr int N = decltype(size)::value;
            float v[N];
#pragma unroll
            for (int j = 0; j < N; ++j) v[j] = (j < n) ? base[j * NB * kRows] : 0.f;
#pragma unroll
            for (int w2 = 1; w2 < N; w2 *= 2)
#pragma unroll
                for (int j = 0; j + w2 < N; j += 2 * w2) v[j] += v[j + w2];
            return v[0];
        };
        auto sum_groups20 = [&](const float *base, int n) {
            if (kPairs) return tree(std::integral_constant<int, 10>{}, base, n);
            if (n <= 8) return tree(std::integral_constant<int, 8>{}, base, n);
            return tree(std::integral_constant<int, kMaxWarps>{}, base, n);
        };
        // (up to 40 when a warp leaves the sums of two tiles: two trees)
        auto sum_groups = [&](const float *base, int n) {
            float t = sum_groups20(base, n);
            if (TPW == 2 && !kPairs && n > kMaxWarps) t += sum_groups20(base + kMaxWarps * NB * kRows, n - kMaxWarps);
            return t;
        };
        // Tensor-core layout: four tokens at a time, spaced one warp's rows apart; more than eight tiles in two batches of ten,
        // all loads of a batch before its first addition (three smaller batches cost the sixteen-token layer 3 %).
        constexpr int RF = NB;
        // (2-bit rows at eight tokens: packed additions and the short form of in_tens cost 25600 x 5120 20.9 -> 21.7 us, 12288 x 4096 9.5 -> 9.9, and give
        // rows of nine groups 6.2 -> 5.7)
        constexpr bool kShortSums = NB <= 8 && !kBlend && !(FMT == kBit2 && NB == 8);
        auto add4 = [](float4 a, float4 b) { return add_quads<kShortSums>(a, b); };
        const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
        auto batch = [&](auto full, const float *base, int n) {
            float4 v[10];
#pragma unroll
            for (int j = 0; j < 10; ++j) v[j] = decltype(full)::value || j < n ? *reinterpret_cast<const float4 *>(base + j * kRows * RF) : none;
#pragma unroll
            for (int w2 = 1; w2 < 10; w2 *= 2)
#pragma unroll
                for (int j = 0; j + w2 < 10; j += 2 * w2) v[j] = add4(v[j], v[j + w2]);
            return v[0];
        };
        // The second batch is left out of rows of nine or ten tiles (96 experts of 768 x 1152 | 1280 at eight tokens 11.0 | 11.7 -> 10.3 | 11.0 us).
        // Forms of a batch without guards grow this warp's code, which costs every length: with forms for full batches and for second ones
        // of six or eight, 4736 rows of 12 | 17 | 19 groups at eight tokens went from 4.9 | 5.3 | 5.3 to 5.1 | 5.5 | 5.5 us, without them 4.8 |
        // 5.2 | 5.2; 16 | 18 groups 5.3 | 5.3 -> 5.2 | 5.2 with and without.  Full batches alone pay at five-trit rows and eight tokens
        // (25600 x 5120 26.1 -> 24.7, 16384 x 5120 17.3 -> 16.9, 18944 x 1536 8.0 -> 8.2).
        auto in_tens = [&](const float *base, int n) {
            const float *second = base + 10 * kRows * RF;
            if constexpr (FMT == kTrit5 && NB == 8) {
                if (n >= 10) {
                    const float4 tot = batch(std::true_type{}, base, 10);
                    if (n == 10) return tot;
                    return add4(tot, n == 20 ? batch(std::true_type{}, second, 10) : batch(std::false_type{}, second, n - 10));
                }
            }
            const float4 tot = batch(std::false_type{}, base, n);
            if (kShortSums && n <= 10) return tot;
            return add4(tot, batch(std::false_type{}, second, n - 10));
        };
        auto sum_tiles4 = [&](const float *base, int n) {
            if (n > 8) return in_tens(base, n);
            auto at = [&](int j) { return *reinterpret_cast<const float4 *>(base + j * kRows * RF); };
            float4 tot = none;
#pragma unroll 1
            for (; n >= 4; n -= 4, base += 4 * kRows * RF) {
                const float4 a = at(0), b = at(1), c = at(2), d = at(3);
                tot = add4(tot, add4(add4(a, b), add4(c, d)));
            }
            if (n >= 1) {
                float4 a = at(0);
                if (n >= 2) {
                    const float4 b = at(1);
                    if (!kFrag && n == 3) tot = add4(tot, at(2));
                    if (kFrag) a = add4(a, b);
                    else tot = add4(tot, b);
                    if (kFrag && n == 3) a = add4(a, at(2));
                }
                tot = add4(tot, a);
            }
            return tot;
        };
        // the same from the sums of neighbouring tiles (n of them: nine tiles and more are five and more)
        // (Ten of them without guards: at four tokens large launches of rows of 14 | 19 | 20 groups 11.23 | 10.88 | 10.96 -> 11.10 | 10.84 | 10.90 us; at
        // eight the second form costs all lengths, 12 | 17 | 20 groups 12.8 | 11.4 | 11.5 -> 13.9 | 12.0 | 11.7.)
        auto sum_pairs4 = [&](const float *base, int n) {
            auto at = [&](int j) { return *reinterpret_cast<const float4 *>(base + j * kRows * RF); };
            if (n > 4) {
                float4 v[10];
                if (NB < 8 && n == 10) {
#pragma unroll
                    for (int j = 0; j < 10; ++j) v[j] = at(j);
                } else {
#pragma unroll
                    for (int j = 0; j < 10; ++j) v[j] = (j < 5 || j < n) ? at(j) : none;
                }
                return add4(add4(add4(add4(v[0], v[1]), add4(v[2], v[3])), v[4]), add4(add4(add4(v[5], v[6]), add4(v[7], v[8])), v[9]));
            }
            float4 tot = none;
#pragma unroll 1
            for (; n >= 2; n -= 2, base += 2 * kRows * RF) tot = add4(tot, add4(at(0), at(1)));
            if (n) tot = add4(tot, at(0));
            return tot;
        };
        // Sixteen tokens: by threes, the at most five threes by pairs; from n single tiles ..
        auto sum_threes4 = [&](const float *base, int n) {
            // (without branches, so that the loads of all tokens are under way together)
            auto up_to = [&](auto size) {
                constexpr int N = decltype(size)::value;
                float4 v[N], t[(N + 2) / 3];
#pragma unroll
                for (int i = 0; i < N; ++i) v[i] = i < n ? *reinterpret_cast<const float4 *>(base + i * kRows * RF) : none;
#pragma unroll
                for (int i = 0; i < N; ++i) t[i / 3] = i % 3 ? add4(t[i / 3], v[i]) : v[i];
                if constexpr (N <= 3) return t[0];
                else if constexpr (N <= 6) return add4(t[0], t[1]);
                else return add4(add4(add4(t[0], t[1]), add4(t[2], t[3])), t[4]);
            };
            if (n <= 3) return up_to(std::integral_constant<int, 3>{});
            if (n <= 6) return up_to(std::integral_constant<int, 6>{});
            return up_to(std::integral_constant<int, kWarps16>{});
        };
        // .. or from n sums of three (more than five only where rows are cut by their own width)
        auto sum_of_threes4 = [&](const float *base, int n) {
            auto at = [&](int j) { return *reinterpret_cast<const float4 *>(base + j * kRows * RF); };
            if (n > 5) return in_tens(base, n);
            if (n > 3) {
                const float4 a = at(0), b = at(1), c = at(2), d = at(3);
                float4 e = none;
                if (n > 4) e = at(4);
                return add4(add4(add4(a, b), add4(c, d)), e);
            }
            float4 a = at(0);
            if (n >= 2) a = add4(a, at(1));
            if (n == 3) a = add4(a, at(2));
            return a;
        };
        auto sum_groups4 = [&](const float *base, int n) {
            if constexpr (kFrag && NB > 8 && kPairs) return sum_of_threes4(base, n);
            else if constexpr (kFrag && NB > 8) return sum_threes4(base, n);
            else if constexpr (kPairs && !kBlend) return sum_pairs4(base, n);      // (the 16-bit variant has an order of its own)
            else return sum_tiles4(base, n);
        };
        // one row block's outputs: row m of every token, one M apart
        auto store_rows = [&](int64_t m, const float (&t)[NB]) {
            if (m >= pb.M) return;
            float *out = pb.y + pr.out_row0(pb) * pb.M + m;
            const int64_t step = pb.M;
            const int nb = pr.nb(pb);
#pragma unroll
            for (int b = 0; b < NB; ++b, out += step)
                if (b < nb) *out = xscale(b) * t[b];
        };
        // the sums of what warps j0 .. j0 + n - 1 left, for this lane's row and every token
        auto sums = [&](const float *rs, int j0, int n, float (&tot)[NB]) {
            if (NB >= kMmaMinBatch) {
#pragma unroll
                for (int t = 0; t < NB / 4; ++t) {
                    float4 v4 = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (4 * t < pr.nb(pb)) v4 = sum_groups4(rs + (j0 * kRows + lane) * RF + ((4 * t) ^ red_swizzle<NB>(lane)), n);
                    tot[4 * t + 0] = v4.x;
                    tot[4 * t + 1] = v4.y;
                    tot[4 * t + 2] = v4.z;
                    tot[4 * t + 3] = v4.w;
                }
            } else {
#pragma unroll
                for (int b = 0; b < NB; ++b)
                    tot[b] = (b < pr.nb(pb)) ? sum_groups(rs + (j0 * NB + b) * kRows + lane, n) : 0.f;
            }
        };
        // The same over n tiles of a row that begin at warp j0.  Several tiles per warp in fragment order (kSubs): one column block
        // of the one-tile plan after the other (two of them, sixteen tokens' up to three), added to tot (fresh: instead of it).
        constexpr bool kSubs = kPairs && !kBlend;
        auto row_sums = [&](const float *rs, int j0, int n, float (&tot)[NB], bool fresh) {
            if constexpr (kSubs) {
#pragma unroll 1
                for (; n > 0; n -= pl.sub, j0 += pl.wsub, fresh = false) {
                    float t[NB];
                    sums(rs, j0, ((n < pl.sub ? n : pl.sub) + TPW - 1) / TPW, t);
#pragma unroll
                    for (int b = 0; b < NB; ++b) tot[b] = fresh ? t[b] : tot[b] + t[b];
                }
            } else {
                sums(rs, j0, kPairs ? (n + TPW - 1) / TPW : n, tot);
            }
        };
        do {
        if constexpr (Segs::kHetero) {
            // A phased launch: this segment's activations (and whatever else its job reads) may be
            // written by the jobs of the phase before it, so they are fetched only once every thread
            // block has finished that phase.  All decoder warps have left the previous segment's
            // contractions by now (its last partial sums were consumed above), so the one activation
            // buffer is free.
            if (!src.wait_dependency(lane)) {
                if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
                return;
            }
            if (lane == 0) BITCOS_TLP(src, 0);
            fetch_x();
        }
        n_pend = 0;
        it.init(pl, wk.first);
        if (kHoldScales) {
#pragma unroll
            for (int b = 0; b < NB; ++b) xsc[kHoldScales ? b : 0] = __ldg(pb.x_scale + xr[b]);
        }
        for (int k = 0; k < wk.count; ++k, ++kk, it.next(pl, wk)) {
            const int slot = kk & rs_mask;
            const ItemRange r = item_range(pb, pl, it.c, it.cs);
            if (!mbar_wait(bar0 + 8u * (kBarRedFull + slot), static_cast<uint32_t>((kk >> rs_log2) & 1))) {
                if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
                return;
            }
            // every decoder warp has posted this item's sums, so none of them reads its stage any more:
            // one arrival per item hands the stage back to the producer
            if (lane == 0) mbar_arrive(bar0 + 8u * (kBarEmpty + es));
            if (++es == pl.stages) es = 0;
            const float *rs = red + slot * red_slot;
            if (pl.CS == 1) {
                // whole row blocks: one output per row.  The sums are formed first, the slot is
                // handed back, and only then are the outputs stored, so that the release of the
                // slot never waits for a global store.
                const int nrb = r.nt / pb.G, parts = kPairs ? pl.wrow : pb.G;
                for (int i = 0; i < nrb; ++i) {
                    const int64_t m = static_cast<int64_t>(r.rb0 + i) * kRows + lane;
                    float t_b[NB];
                    row_sums(rs, i * parts, pb.G, t_b, true);
                    if (i == nrb - 1) {
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar0 + 8u * (kBarRedEmpty + slot));
                    }
                    store_rows(m, t_b);
                }
                continue;
            }
            // one column block of row block rb0: add it to the running sum
            const bool starts = (r.cs == 0) || (k == 0);
            if constexpr (kSubs) {
                row_sums(rs, 0, r.nt, run, starts);
            } else {
                float t_b[NB];
                row_sums(rs, 0, r.nt, t_b, true);
#pragma unroll
                for (int b = 0; b < NB; ++b) run[b] = starts ? t_b[b] : run[b] + t_b[b];
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar0 + 8u * (kBarRedEmpty + slot));
            const bool ends = (r.cs == pl.CS - 1) || (k == wk.count - 1);
            if (!ends) continue;
            const int first_cs = (k >= r.cs) ? 0 : r.cs - k;       // first column block of rb0 seen by this block
            const int64_t m = static_cast<int64_t>(r.rb0) * kRows + lane;
            if (first_cs == 0 && r.cs == pl.CS - 1) {
                // the whole row block was ours
                store_rows(m, run);
            } else {
                // shared row block: publish our share, then count ourselves in
                Share sh;
                sh.rb = r.rb0;
                const int lo = owner_of(wk, r.rb0 * pl.CS), hi = owner_of(wk, r.rb0 * pl.CS + pl.CS - 1);
                sh.slot = src.block_in_job(block) - lo;
                sh.sharers = hi - lo + 1;
#pragma unroll
                for (int b = 0; b < NB; ++b)
                    if (b < pr.nb(pb))
                        pb.partial[((static_cast<int64_t>(sh.rb) * pl.CS + sh.slot) * pr.nb(pb) + b) * kRows + lane] = run[b];
                __syncwarp();
                sh.old = 0;
                if (lane == 0) {
                    __threadfence();
                    sh.old = atomicAdd(pb.counters + sh.rb, 1u);
                }
                pend[n_pend++] = sh;      // at most two per block: its first and its last row block
            }
        }
        for (int i = 0; i < n_pend; ++i) finish_share<NB, kXG, kBlend>(pb, pl, xr, pend[i], lane);
        if constexpr (Segs::kHetero) src.signal_done(lane);      // this block's outputs of the phase are written
        if (lane == 0) BITCOS_TLP(src, 5);
        have = next_segment();
        if (have && !Segs::kHetero) token_rows();
        } while (have);
        if (lane == 0) {
            BITCOS_TL(9, clock64());
            BITCOS_TL(11, global_timer_ns());
        }
        return;
    }

    // ------------------------------------------------------------------ decoder warps, fragment order
    // (tiles decoded straight into the A operands of the tensor cores, FragmentRows: no transposition through
    // shared memory, and two tokens come out of the products that one would need)
    if constexpr (kFrag) {
        constexpr int NC = NB < 8 ? NB : 8;              // tokens in the n dimension of one product
        constexpr int NH = NB > 8 ? 2 : 1;               // 8-token halves of the batch
        // The eight columns of a product hold the tokens over and over (column n: token n % NC), so with fewer than
        // eight tokens every lane has all of a tile's sums of its rows somewhere in its quad, and the quad
        // shares out the rows: of rows g + 8 s (g = lane / 4), lane t takes slots s0 .. s0 + NS - 1, and of the
        // tokens n0 and n0 + 1.
        constexpr int NS = NC == 8 ? 4 : NC == 4 ? 2 : 1;
        const int g8 = lane >> 2, t4 = lane & 3;
        const int s0 = NC == 8 ? 0 : NC == 4 ? 2 * (t4 >> 1) : t4;
        const int n0 = NC == 8 ? 2 * t4 : NC == 4 ? 2 * (t4 & 1) : 0;
        const uint32_t lane4 = static_cast<uint32_t>(lane) * 4u;
        // CS == 1: tile t of an item always is row block t / G of the chunk, group t % G
        // (a phased launch works these out again for every job)
        // several tiles: run number warp - wrow rbl of the row, the runs of a column block of the one-tile plan after those
        // of the one before it; the run has n_run tiles, fewer at the end of the column block or of the row
        int rbl = 0, g_first = 0, n_run = 1;
        auto place = [&]() {
            const int wr = kBlend ? (pb.G + TPW - 1) / TPW : kPairs ? pl.wrow : pb.G;      // warps per row block when items are whole rows
            rbl = pl.CS == 1 ? warp / wr : 0;
            g_first = warp - rbl * wr;
            if (kBlend) {
                g_first *= TPW;
            } else if (kPairs) {
                const int cb = g_first / pl.wsub;
                g_first = cb * pl.sub + (g_first - cb * pl.wsub) * TPW;
                int g_end = (cb + 1) * pl.sub;
                if (pl.CS == 1 && g_end > pb.G) g_end = pb.G;
                n_run = g_end - g_first < TPW ? g_end - g_first : TPW;
            }
        };
        place();
        int tile0 = rbl * pb.G + g_first;
        uint32_t x_parity = 0;      // phase parity of the activations' barrier: one phase per segment of a phased launch
        if (!mbar_wait(bar0 + 8u * kBarLut, 0)) {
            if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
            return;
        }
        if (warp == 0 && lane == 0) BITCOS_TL(3, clock64());
        bool tl_first = true;
        // B operand: of token g8 % NC (+ 8) this lane holds the 32 activations of presence word t4 of the group
        const int8_t *xfrag[NH];
        auto token_fragments = [&]() {
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                const int n = 8 * h + g8 % NC;
                xfrag[h] = nullptr;
                if (NB >= kMmaMinBatch && n < pr.nb(pb))
                    xfrag[h] = kBlend ? pb.x + 2 * (static_cast<int64_t>(n) * pb.K + 32 * t4)
                                      : pb.x + static_cast<int64_t>(pr.xrow(pb) ? __ldg(pr.xrow(pb) + n) : n) * pb.K + 32 * t4;
            }
        };
        uint32_t bf[NH][kBlend ? 16 : 8];
        float xg[NH][2];            // group scales of the tokens whose sums this lane keeps
        auto load_x = [&](int grp, const uint8_t *xs) {
            if constexpr (NB < kMmaMinBatch) {
                const uint4 *px = reinterpret_cast<const uint4 *>(xs + 32 * t4 + (g8 & 1) * (kXQ ? kGroup : static_cast<int>(x_stride(pb.K))));
                const uint4 u0 = px[0], u1 = px[1];
                bf[0][0] = u0.x; bf[0][1] = u0.y; bf[0][2] = u0.z; bf[0][3] = u0.w;
                bf[0][4] = u1.x; bf[0][5] = u1.y; bf[0][6] = u1.z; bf[0][7] = u1.w;
            } else if constexpr (kBlend) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    int4 u = make_int4(0, 0, 0, 0);
                    if (xfrag[0]) u = __ldg(reinterpret_cast<const int4 *>(xfrag[0] + static_cast<int64_t>(grp) * (2 * kGroup)) + q);
                    bf[0][4 * q] = u.x; bf[0][4 * q + 1] = u.y; bf[0][4 * q + 2] = u.z; bf[0][4 * q + 3] = u.w;
                }
            } else {
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    int4 u0 = make_int4(0, 0, 0, 0), u1 = make_int4(0, 0, 0, 0);
                    if (xfrag[h]) {
                        const int4 *px = reinterpret_cast<const int4 *>(xfrag[h] + static_cast<int64_t>(grp) * kGroup);
                        u0 = __ldg(px);
                        u1 = __ldg(px + 1);
                    }
                    bf[h][0] = u0.x; bf[h][1] = u0.y; bf[h][2] = u0.z; bf[h][3] = u0.w;
                    bf[h][4] = u1.x; bf[h][5] = u1.y; bf[h][6] = u1.z; bf[h][7] = u1.w;
                }
            }
            if constexpr (kXG && !kXQ && !kBlend) {
                // (after the dependency wait: the scales come from the kernel before this one)
#pragma unroll
                for (int h = 0; h < NH; ++h)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const int b = 8 * h + n0 + r;
                        xg[h][r] = (b < pr.nb(pb)) ? __ldg(pb.x_scale + static_cast<int64_t>(b) * pb.G + grp) : 0.f;
                    }
            }
        };
        // 16-bit activations: the group this warp has quantised last, its scales, and its buffer
        // ([token][128] int8 inside the activation area)
        int q_g = -1;
        float q_scale[2] = {};
        uint32_t *q_scr = reinterpret_cast<uint32_t *>(smem + L.x) + static_cast<uint32_t>(warp) * (NB * kRows);
        uint2 qv[2];
        auto fetch_group = [&](int grp) {
#pragma unroll
            for (int b = 0; b < 2; ++b)
                if (b < pr.nb(pb))
                    qv[b] = __ldg(reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(pb.x) + static_cast<int64_t>(b) * pb.K +
                                                                  static_cast<int64_t>(grp) * kGroup) + lane);
        };
        auto quantize_group = [&](int grp) {
            // this warp quantises the group its tile multiplies (four values per lane, largest magnitude by
            // shuffles) into its own 128 bytes per token
            __syncwarp();                     // the previous tile's fragments have been read
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                if (b < pr.nb(pb)) {
                    const uint2 v = qv[b];
                    float a = fmaxf(fmaxf(fabsf(bf16_lo(v.x)), fabsf(bf16_hi(v.x))), fmaxf(fabsf(bf16_lo(v.y)), fabsf(bf16_hi(v.y))));
#pragma unroll
                    for (int dd = 16; dd; dd >>= 1) a = fmaxf(a, __shfl_xor_sync(0xFFFFFFFFu, a, dd));
                    a = fmaxf(a, kAmaxFloor);
                    const float inv = __fdiv_rn(127.0f, a);
                    q_scale[b] = __fdiv_rn(a, 127.0f);
                    q_scr[b * kRows + lane] = quant_pair(v.x, inv) | (quant_pair(v.y, inv) << 16);
                }
            }
            __syncwarp();
            q_g = grp;
        };
        // byte offsets inside a stage that depend on nothing but the layout
        const uint32_t off_sign = L.payload_cap, off_scales = L.payload_cap + L.sign_cap;
        const uint32_t off_x = off_scales + L.scale_cap + L.off_cap;                     // activations inside a stage
        // where this lane leaves its partial sums inside a slot
        float *rd0 = red + (NB >= kMmaMinBatch ? static_cast<uint32_t>(warp * kRows + g8) * NB : static_cast<uint32_t>(warp * NB * kRows + g8 + 8 * s0));
        const uint8_t *stage = smem + L.stage;
        uint32_t full_bar = bar0 + 8u * static_cast<uint32_t>(kBarFull), phase = 0;
        int s = 0;
        int kk = 0;                 // items decoded so far, over all segments
        bool x_ready = false, x_held = false;
        bool more_segments = false;
        do {
        if (!kLate) {
            token_fragments();
            x_ready = true;
            x_held = false;
        }
        for (const int kk_end = kk + wk.count; kk < kk_end; ++kk) {
            if (!mbar_wait(full_bar, phase)) {
                if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
                return;
            }
            if (tl_first && warp == 0 && lane == 0) BITCOS_TL(4, clock64());
            if (tl_first && warp == 0 && lane == 0) BITCOS_TLP(src, 1);
            const uint4 d = reinterpret_cast<const uint4 *>(sign_base)[s];
            const int nt = static_cast<int>(d.x & 0xFFu);
            float ysum[NH][NS][2];
#pragma unroll
            for (int h = 0; h < NH; ++h)
#pragma unroll
                for (int j = 0; j < NS; ++j) ysum[h][j][0] = ysum[h][j][1] = 0.f;
#pragma unroll 1
            for (int ti = 0; ti < TPW; ++ti) {
                const int tile = tile0 + ti;
                if (tile >= nt || (kPairs && (kBlend ? pl.CS == 1 && g_first + ti >= pb.G : ti >= n_run))) break;
                // group: the item's first (0 when items are whole rows) + the tile's place in its row block
                const int grp = static_cast<int>(d.y) + g_first + ti;
                const uint8_t *xs = kXQ ? reinterpret_cast<const uint8_t *>(q_scr)
                                        : ((!Segs::kSingle && pl.x_in_stage) ? stage + off_x : smem + L.x) + static_cast<uint32_t>(grp) * kGroup;
                // from global memory: ahead of the decode, which hides the latency (not before the dependency is
                // resolved); a warp whose group never changes keeps its fragments
                if (NB >= kMmaMinBatch && x_ready && !(TPW == 1 && pl.CS == 1 && x_held)) {
                    load_x(grp, xs);
                    x_held = true;
                }
                if (kXQ && x_ready && grp != q_g) fetch_group(grp);
                const uint32_t toff = *reinterpret_cast<const uint32_t *>(stage + off_scales + L.scale_cap + 4u * static_cast<uint32_t>(tile) + ((d.x >> 8) << 2));
                FragmentRows rows;
                rows.open(stage + 512u * static_cast<uint32_t>(tile), stage + off_sign, toff - d.w, lane4);
                // One tile per warp: everything is decoded before the first product (launches of a few items, where a
                // block's first decode runs while it waits for its dependency).  Two tiles: product by product.
                // (The 16-bit variant always: its decoded row would be 64 registers.)
                constexpr bool kFused = TPW > 1 || kBlend;
                if (kBlend) rows.shift_presence();
                int e[kFused ? 1 : 4][8];
                if (!kFused) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) rows.step(k, lut, lane4, e[kFused ? 0 : k]);
                }
                if (!x_ready) {
                    // first contraction of this warp: the previous kernel must be complete before the activations
                    // are read (the decode above did not need them)
                    if (tl_first && warp == 0 && lane == 0) BITCOS_TL(5, clock64());
                    if (tl_first && warp == 0 && lane == 0) BITCOS_TLP(src, 2);
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                    if (kEarly && !kXQ && !mbar_wait(bar0 + 8u * kBarX, x_parity)) {
                        if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
                        return;
                    }
                    x_ready = true;
                    if (tl_first && warp == 0 && lane == 0) BITCOS_TL(6, clock64());
                    if (tl_first && warp == 0 && lane == 0) BITCOS_TLP(src, 3);
                    token_fragments();
                    if (NB >= kMmaMinBatch) {
                        load_x(grp, xs);
                        x_held = true;
                    }
                    if (kXQ) fetch_group(grp);
                }
                if (kXQ && grp != q_g) quantize_group(grp);
                if (NB < kMmaMinBatch) load_x(grp, xs);
                // int32 sums, or fp32 ones of the 16-bit variant: weights +-2^-8 against the activations as they are, the scale
                // applied to the group's sum (every product is exact).  Its table holds bf16 words, so that a lookup is two
                // fragment registers: 18944 -> 56832 x 5120 176 clocks per tile and multiprocessor at one token, 213 at four and
                // eight; 8192x5120 at four tokens 13.8 -> 11.3 us against rebuilding +-s from int8 weights and a pass
                // through shared memory.
                typename std::conditional<kBlend, float, int>::type acc[NH][2][4];
#pragma unroll
                for (int h = 0; h < NH; ++h)
#pragma unroll
                    for (int mh = 0; mh < 2; ++mh)
#pragma unroll
                        for (int r = 0; r < 4; ++r) acc[h][mh][r] = 0;
                if constexpr (kBlend) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        uint32_t ej[8];
                        rows.step_bf16(j, lut, 2u * lane4, ej);
#pragma unroll
                        for (int mh = 0; mh < 2; ++mh) {
                            const uint32_t a[4] = {ej[4 * mh], ej[4 * mh + 2], ej[4 * mh + 1], ej[4 * mh + 3]};
                            mma_bf16(acc[0][mh], a, bf[0][2 * j], bf[0][2 * j + 1]);
                        }
                    }
                } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    int(&ek)[8] = e[kFused ? 0 : k];
                    if (kFused) rows.step(k, lut, lane4, ek);
#pragma unroll
                    for (int mh = 0; mh < 2; ++mh) {
                        const uint32_t a[4] = {static_cast<uint32_t>(ek[4 * mh]), static_cast<uint32_t>(ek[4 * mh + 2]),
                                               static_cast<uint32_t>(ek[4 * mh + 1]), static_cast<uint32_t>(ek[4 * mh + 3])};
#pragma unroll
                        for (int h = 0; h < NH; ++h) mma_s8(acc[h][mh], a, bf[h][2 * k], bf[h][2 * k + 1]);
                    }
                }
                }
#pragma unroll
                for (int j = 0; j < NS; ++j) {
                    const float sc = bf16_to_float(*reinterpret_cast<const uint16_t *>(stage + off_scales + 2u * static_cast<uint32_t>(tile * kRows + g8 + 8 * (s0 + j))));
#pragma unroll
                    for (int h = 0; h < NH; ++h)
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            // row slot s of a token pair's accumulators: acc[h][s / 2][2 * (s % 2) + column]
                            typename std::conditional<kBlend, float, int>::type v;
                            if (NC == 8) v = acc[h][j >> 1][2 * (j & 1) + r];
                            else if (NC == 4) v = (t4 & 2) ? acc[h][1][2 * j + r] : acc[h][0][2 * j + r];
                            else {
                                const auto lo = (t4 & 1) ? acc[h][0][2 + r] : acc[h][0][r], hi = (t4 & 1) ? acc[h][1][2 + r] : acc[h][1][r];
                                v = (t4 & 2) ? hi : lo;
                            }
                            float y = sc * static_cast<float>(v);
                            // (a group scale makes the product inexact: rounded before it is added, as it is where a tile's
                            // sum is all that a warp leaves; bf16 scale times sum is exact, the 16-bit variant has one plan)
                            if (kXQ) y = kPairs ? __fmul_rn(y, q_scale[r]) : y * q_scale[r];
                            else if (kXG && !kBlend) y = kPairs ? __fmul_rn(y, xg[h][r]) : y * xg[h][r];
                            ysum[h][j][r] += y;
                            if constexpr (Segs::kDebug) if (pb.acc_debug) {
                                const int b = 8 * h + n0 + r;
                                const int64_t m = (static_cast<int64_t>(d.z) + rbl) * kRows + g8 + 8 * (s0 + j);
                                if (b < pr.nb(pb) && m < pb.M) pb.acc_debug[((pr.out_row0(pb) + b) * pb.M + m) * pb.G + grp] = v;
                            }
                        }
                }
            }
            // partial sums for the epilogue warp (several slots, so decoders may run ahead of it); the stage goes
            // back to the producer when the epilogue warp has seen them
            const int slot = kk & rs_mask;
            if ((kk >> rs_log2) > 0) {
                if (!mbar_wait(bar0 + 8u * (kBarRedEmpty + slot), static_cast<uint32_t>(((kk >> rs_log2) - 1) & 1))) {
                    if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
                    return;
                }
            }
            float *rd = rd0 + slot * red_slot;
            if (NB >= kMmaMinBatch) {
#pragma unroll
                for (int h = 0; h < NH; ++h)
#pragma unroll
                    for (int j = 0; j < NS; ++j)
                        *reinterpret_cast<float2 *>(rd + 8 * (s0 + j) * NB + ((8 * h + n0) ^ red_swizzle<NB>(g8 + 8 * (s0 + j)))) =
                            make_float2(ysum[h][j][0], ysum[h][j][1]);
            } else {
                rd[0] = ysum[0][0][0];
                rd[kRows] = ysum[0][0][1];
            }
            __syncwarp();
            mbar_arrive_lane0(bar0 + 8u * (kBarRedFull + slot), lane);
            if (tl_first && warp == 0 && lane == 0) BITCOS_TL(7, clock64());
            tl_first = false;
            stage += L.stage_bytes;
            full_bar += 8u;
            if (++s == pl.stages) {
                s = 0;
                stage = smem + L.stage;
                full_bar = bar0 + 8u * static_cast<uint32_t>(kBarFull);
                phase ^= 1u;
            }
        }
        if (warp == 0 && lane == 0) BITCOS_TL(10, clock64());
        if (warp == 0 && lane == 0) BITCOS_TLP(src, 4);
        if constexpr (Segs::kHetero) {
            // Every decoder warp passes every phase of the activations' barrier, a warp without a tile in
            // this segment included: a warp that skipped one could not tell the phase before from the
            // phase after by its parity.
            if (!x_ready && !mbar_wait(bar0 + 8u * kBarX, x_parity)) {
                if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
                return;
            }
            more_segments = next_segment();
            tl_first = true;
            if (more_segments) {
                x_ready = false;
                x_parity ^= 1u;
                place();
                tile0 = rbl * pb.G + g_first;
            }
        } else {
            more_segments = next_segment();
        }
        } while (more_segments);
        return;
    }

    // ------------------------------------------------------------------ decoder warps
    // CS == 1: tile t of an item always is row block t / G of the chunk, group t % G; this warp
    // decodes tile `warp` and, with two tiles per warp, tile `warp + NW`
    constexpr int tpw = TPW;
    // (a phased launch works these out again for every job)
    int my_rbl0 = (pl.CS == 1) ? warp / pb.G : 0;
    int g_fixed0 = warp - my_rbl0 * pb.G;
    int my_rbl1 = (pl.CS == 1) ? (warp + pl.NW) / pb.G : 0;
    int g_fixed1 = warp + pl.NW - my_rbl1 * pb.G;
    uint32_t x_parity = 0;      // phase parity of the activations' barrier: one phase per segment of a phased launch
    if (FMT != kBit2) {
        if (!mbar_wait(bar0 + 8u * kBarLut, 0)) {
            if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
            return;
        }
    }
    if (warp == 0 && lane == 0) BITCOS_TL(3, clock64());
    bool tl_first = true;
    constexpr bool kMma = NB >= kMmaMinBatch;          // contraction on the tensor cores
    static_assert(kFrag || !kXG || NB == 1, "group scales and 16-bit activations: one token here, from two on in fragment order");
    constexpr int NH = NB > 8 ? 2 : 1;                 // 8-token halves of the batch
    constexpr int NV = kMma ? NH * 8 : NB;             // partial sums a lane hands to the epilogue warp
    const uint32_t lane4 = static_cast<uint32_t>(lane) * 4u;
    // Tensor-core path.  The order of the 128 products inside a group is free, so it is chosen to
    // make the activation loads contiguous: of tokens lane / 4 and lane / 4 + 8 this lane holds
    // bytes 16 c .. 16 c + 15 and 64 + 16 c .. 64 + 16 c + 15 of the group (c = lane % 4, two 16-byte
    // loads), and k-block kb of the contraction pairs words 2 kb and 2 kb + 1 of those eight with
    // the matching weight words.  A operand: each lane stores the row it decoded into the warp's
    // buffer (32 int8 at a time, in that order), ldmatrix brings it back in fragment order.
    const int8_t *xfrag[NH];
    auto token_fragments = [&]() {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const int n = 8 * h + (lane >> 2);
            xfrag[h] = nullptr;
            if (kMma && n < pr.nb(pb))
                xfrag[h] = pb.x + static_cast<int64_t>(pr.xrow(pb) ? __ldg(pr.xrow(pb) + n) : n) * pb.K + 16 * (lane & 3);
        }
    };
    uint32_t bf[NH][8];
    auto load_bf = [&](int g) {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            int4 u0 = make_int4(0, 0, 0, 0), u1 = make_int4(0, 0, 0, 0);
            if (xfrag[h]) {
                const int4 *px = reinterpret_cast<const int4 *>(xfrag[h] + static_cast<int64_t>(g) * kGroup);
                u0 = __ldg(px);
                u1 = __ldg(px + 4);
            }
            bf[h][0] = u0.x; bf[h][1] = u0.y; bf[h][2] = u0.z; bf[h][3] = u0.w;
            bf[h][4] = u1.x; bf[h][5] = u1.y; bf[h][6] = u1.z; bf[h][7] = u1.w;
        }
    };

    const uint32_t scr0 = smem_addr(smem + L.scr) + static_cast<uint32_t>(warp) * kScrBytes;
    const uint32_t scr_st = scr0 + static_cast<uint32_t>(lane) * kScrRowBytes;
    const uint32_t scr_ld = scr0 + static_cast<uint32_t>((lane & 7) + ((lane >> 3) & 1) * 8) * kScrRowBytes +
                            static_cast<uint32_t>(lane >> 4) * 16u;
    const uint8_t *stage0 = smem + L.stage;
    const uint8_t *stage = stage0;
    const uint4 *desc = reinterpret_cast<const uint4 *>(sign_base);
    uint32_t full_bar = bar0 + 8u * kBarFull, phase = 0;
    int s = 0;
    // byte offsets inside a stage that do not change from item to item (first tile of this warp;
    // the second one lies NW tiles further)
    const uint32_t tile_lane0 = static_cast<uint32_t>(warp * kRows + lane);
    const uint32_t off_bm0 = tile_lane0 * 16u;                                       // this lane's four presence words
    const uint32_t off_scale0 = L.payload_cap + L.sign_cap + tile_lane0 * 2u;          // its row's group scale
    const uint32_t off_toff0 = L.payload_cap + L.sign_cap + L.scale_cap + static_cast<uint32_t>(warp) * 4u;
    const uint32_t off_sign = L.payload_cap;
    const uint32_t tile_step = static_cast<uint32_t>(pl.NW);
    const uint32_t off_x = L.payload_cap + L.sign_cap + L.scale_cap + L.off_cap;     // activations inside a stage
    const uint8_t *xs_base = smem + L.x;
    // where this lane leaves its partial sums inside a slot (one or two tokens)
    float *rd_lane0 = red + static_cast<uint32_t>(warp * NB) * kRows + lane;
    int kk = 0;                 // items decoded so far, over all segments
    bool x_ready = false;
    // 16-bit activations (one token): the group this warp has quantised last, its scale, and its buffer
    // (128 int8 inside the activation area)
    int q_g = -1;
    float q_scale = 0.f;
    uint32_t *q_scr = reinterpret_cast<uint32_t *>(smem + L.x) + static_cast<uint32_t>(warp) * kRows;
    bool more_segments = false;
    do {
    if (!(kLate && kMma)) {
        token_fragments();
        // whole rows per item: this warp's group never changes, neither do its activation fragments
        if (kMma && pl.CS == 1) load_bf(g_fixed0);
    }
    for (const int kk_end = kk + wk.count; kk < kk_end; ++kk) {
        if (!mbar_wait(full_bar, phase)) {
            if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
            return;
        }
        if (tl_first && warp == 0 && lane == 0) BITCOS_TL(4, clock64());
        if (tl_first && warp == 0 && lane == 0) BITCOS_TLP(src, 1);
        const uint4 d = desc[s];
        const int nt = static_cast<int>(d.x & 0xFFu);
        const int slot = kk & rs_mask;
        // Two tiles per warp: the partial sums of a tile are stored as soon as it is done, so the
        // slot must be free before the first one (with one tile per warp that wait comes after
        // the decode, further down).
        if (tpw == 2 && (kk >> rs_log2) > 0) {
            if (!mbar_wait(bar0 + 8u * (kBarRedEmpty + slot), static_cast<uint32_t>(((kk >> rs_log2) - 1) & 1))) {
                if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
                return;
            }
        }
        float ysum[NV];
#pragma unroll 1
        for (int ti = 0; ti < tpw; ++ti) {
        const int tile = warp + (ti ? pl.NW : 0);
        const bool busy = tile < nt;
        const int my_rbl = ti ? my_rbl1 : my_rbl0;
        // group of this tile: the item's first group (0 when items are whole rows) + the tile's
        // place in its row block
        const int g = static_cast<int>(d.y) + (ti ? g_fixed1 : g_fixed0);
        const uint32_t t_off = ti ? tile_step : 0u;
        const uint32_t off_bm = off_bm0 + t_off * (kRows * 16u);
        const uint32_t off_scale = off_scale0 + t_off * (kRows * 2u);
        const uint32_t off_toff = off_toff0 + t_off * 4u;
#pragma unroll
        for (int b = 0; b < NV; ++b) ysum[b] = 0.f;
        // early, so that the decode hides the latency (not before the dependency is resolved)
        if (kMma && pl.CS != 1 && busy && (!kLate || x_ready)) load_bf(g);
        // 16-bit activations of a group this warp has not quantised yet: fetched ahead of the decode too
        uint2 qv;
        bool q_have = false;
        auto fetch_group = [&]() {
            qv = __ldg(reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(pb.x) + static_cast<int64_t>(g) * kGroup) + lane);
            q_have = true;
        };
        if (kXQ && busy && x_ready && g != q_g) fetch_group();

        if (busy) {
            const float sc = bf16_to_float(*reinterpret_cast<const uint16_t *>(stage + off_scale));
            // activations of group g (one or two tokens: always in shared memory)
            // (only the grouped launch ever delivers activations with the stage)
            const uint8_t *xs = kXQ ? reinterpret_cast<const uint8_t *>(q_scr)
                                    : ((!Segs::kSingle && pl.x_in_stage) ? stage + off_x : xs_base) + static_cast<uint32_t>(g) * kGroup;
            int w[32];
            if (FMT == kBitcos) {
                const uint4 bm = *reinterpret_cast<const uint4 *>(stage + off_bm);
                const int c = __popc(bm.x) + __popc(bm.y) + __popc(bm.z) + __popc(bm.w);
                int incl = c;
#pragma unroll
                for (int dd = 1; dd < 32; dd <<= 1) {
                    const int v = __shfl_up_sync(0xFFFFFFFFu, incl, dd);
                    if (lane >= dd) incl += v;
                }
                // entry offset of this tile: word (t0 & 3) + warp of the stage's slice of tile_off
                const uint32_t toff = *reinterpret_cast<const uint32_t *>(stage + off_toff + ((d.x >> 8) << 2));
                const uint32_t cursor = toff + static_cast<uint32_t>(incl - c) - d.w;
                const uint32_t *sp = reinterpret_cast<const uint32_t *>(stage + off_sign + ((cursor >> 5) << 2));
                bitcos_decode_row_keyed(bm, sp, cursor & 31u, lut, lane4, w);
            } else if (FMT == kTrit5) {
                const int WPR = (26 * pb.G + 3) / 4;
                // words of the stage: row block my_rbl of the chunk, counted from the chunk's first word
                const int w_rel = my_rbl * WPR + ((26 * g) >> 2) - ((26 * static_cast<int>(d.y)) >> 2);
                const uint32_t *src = reinterpret_cast<const uint32_t *>(stage) + w_rel * kRows + lane;
                uint32_t wd[7];
#pragma unroll
                for (int i = 0; i < 7; ++i) wd[i] = src[i * kRows];
                trit5_decode_row(wd, g & 1, lut, static_cast<uint32_t>(lane) * 8u, w);
            } else {
                const uint4 *src = reinterpret_cast<const uint4 *>(stage) + (tile * 2) * kRows + lane;
                if (kMma) bit2_decode_row_s8(src[0], src[kRows], w);
                else bit2_decode_row(src[0], src[kRows], w);
            }
            if (kLate && kMma && !x_ready) {
                // first contraction of this warp: the previous kernel must be complete before the
                // activations are read (the decode above did not need them)
                asm volatile("griddepcontrol.wait;" ::: "memory");
                token_fragments();
                load_bf(g);
                x_ready = true;
            }
            if (kMma) {
                int acc[NH][2][4];
#pragma unroll
                for (int h = 0; h < NH; ++h)
#pragma unroll
                    for (int mh = 0; mh < 2; ++mh)
#pragma unroll
                        for (int r = 0; r < 4; ++r) acc[h][mh][r] = 0;
#pragma unroll
                for (int kb = 0; kb < 4; ++kb) {
                    // 32 weights of every row through the buffer: one k-block of the contraction
                    if (kb) __syncwarp();            // everyone has read the previous block back
                    const int w0 = (kb < 2) ? 2 * kb : 16 + 2 * (kb - 2);     // first weight word of this block
                    sts128(scr_st, w[w0], w[w0 + 4], w[w0 + 8], w[w0 + 12]);
                    sts128(scr_st + 16u, w[w0 + 1], w[w0 + 5], w[w0 + 9], w[w0 + 13]);
                    __syncwarp();
#pragma unroll
                    for (int mh = 0; mh < 2; ++mh) {
                        uint32_t a[4];
                        ldmatrix_x4(a, scr_ld + static_cast<uint32_t>(mh * 16 * kScrRowBytes));
#pragma unroll
                        for (int h = 0; h < NH; ++h) mma_s8(acc[h][mh], a, bf[h][2 * kb], bf[h][2 * kb + 1]);
                    }
                }
                // accumulator r of (h, mh): row 16 mh + lane / 4 + 8 (r / 2), token 8 h + 2 (lane % 4) + (r & 1)
                float scq[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) scq[j] = __shfl_sync(0xFFFFFFFFu, sc, (lane >> 2) + 8 * j);
#pragma unroll
                for (int h = 0; h < NH; ++h)
#pragma unroll
                    for (int mh = 0; mh < 2; ++mh)
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            ysum[(h * 2 + mh) * 4 + r] = scq[2 * mh + (r >> 1)] * static_cast<float>(acc[h][mh][r]);
                            if (Segs::kDebug && pb.acc_debug) {
                                const int b = 8 * h + 2 * (lane & 3) + (r & 1);
                                const int64_t m = (static_cast<int64_t>(d.z) + my_rbl) * kRows + 16 * mh + (lane >> 2) + 8 * (r >> 1);
                                if (b < pr.nb(pb) && m < pb.M) pb.acc_debug[((pr.out_row0(pb) + b) * pb.M + m) * pb.G + g] = acc[h][mh][r];
                            }
                        }
            }
            // decode first, contract afterwards: keeps the table lookups of the decode back to back
            // (interleaving them with the contraction's activation loads measured 20 % slower on the
            // five-trit path)
            if (!kMma) asm volatile("" ::: "memory");
            if (kEarly && !x_ready) {
                // first contraction of this warp: the previous kernel must be complete and the
                // activations in place (the decode above needed neither)
                if (tl_first && warp == 0 && lane == 0) BITCOS_TL(5, clock64());
                if (tl_first && warp == 0 && lane == 0) BITCOS_TLP(src, 2);
                asm volatile("griddepcontrol.wait;" ::: "memory");
                if (!kXQ && !mbar_wait(bar0 + 8u * kBarX, x_parity)) {
                    if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
                    return;
                }
                x_ready = true;
                if (tl_first && warp == 0 && lane == 0) BITCOS_TL(6, clock64());
                if (tl_first && warp == 0 && lane == 0) BITCOS_TLP(src, 3);
            }
            if (kXQ && g != q_g) {
                // 16-bit activations: this warp quantises the group its tile multiplies (four values
                // per lane, largest magnitude by shuffles) into its own 128 bytes
                if (!q_have) fetch_group();        // (first tile: the dependency has only just been resolved)
                __syncwarp();                     // the previous tile's contraction has read the buffer
                float a = fmaxf(fmaxf(fabsf(bf16_lo(qv.x)), fabsf(bf16_hi(qv.x))), fmaxf(fabsf(bf16_lo(qv.y)), fabsf(bf16_hi(qv.y))));
#pragma unroll
                for (int dd = 16; dd; dd >>= 1) a = fmaxf(a, __shfl_xor_sync(0xFFFFFFFFu, a, dd));
                a = fmaxf(a, kAmaxFloor);
                const float inv = __fdiv_rn(127.0f, a);
                q_scale = __fdiv_rn(a, 127.0f);
                q_scr[lane] = quant_pair(qv.x, inv) | (quant_pair(qv.y, inv) << 16);
                __syncwarp();
                q_g = g;
            }
            // (after the dependency wait: the scales come from the kernel before this one)
            const float xgs = kXQ ? q_scale : kXG ? __ldg(pb.x_scale + g) : 1.f;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                if (kMma) break;
                if (NB == 1 || b < pr.nb(pb)) {       // a call has at least one token
                    const int a = contract<FMT>(w, reinterpret_cast<const int4 *>(xs + static_cast<uint32_t>(b) * (kXQ ? static_cast<uint32_t>(kGroup) : static_cast<uint32_t>(x_stride(pb.K)))), lane);
                    ysum[b] = sc * static_cast<float>(a);
                    if (kXG) ysum[b] *= xgs;
                    if (Segs::kDebug && pb.acc_debug) {
                        const int64_t m = (static_cast<int64_t>(d.z) + my_rbl) * kRows + lane;
                        if (m < pb.M) pb.acc_debug[((pr.out_row0(pb) + b) * pb.M + m) * pb.G + g] = a;
                    }
                }
            }
        }
        if (tpw == 2) {
            // (one or two tokens only) this tile's partial sums, zeros if the item has no such tile
#pragma unroll
            for (int b = 0; b < NB; ++b)
                if (!kMma) rd_lane0[slot * red_slot + (t_off * NB + b) * kRows] = ysum[b];
        }
        }
        // (the stage goes back to the producer when the epilogue warp has seen this item's partial sums)
        stage += L.stage_bytes;
        full_bar += 8u;
        if (++s == pl.stages) {
            s = 0;
            stage = stage0;
            full_bar = bar0 + 8u * kBarFull;
            phase ^= 1u;
        }

        // partial sums for the epilogue warp (several slots, so decoders may run ahead of it)
        if (tpw == 1 && (kk >> rs_log2) > 0) {
            if (!mbar_wait(bar0 + 8u * (kBarRedEmpty + slot), static_cast<uint32_t>(((kk >> rs_log2) - 1) & 1))) {
                if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
                return;
            }
        }
        float *rd = red + slot * red_slot;
        if (tpw == 2) {
            // already stored, tile by tile
        } else if (kMma) {
#pragma unroll
            for (int i = 0; i < NV; i += 2) {
                const int b = 8 * (i >> 3) + 2 * (lane & 3);                          // and b + 1
                const int row = 16 * ((i >> 2) & 1) + (lane >> 2) + 8 * ((i >> 1) & 1);
                if (b < NB)
                    *reinterpret_cast<float2 *>(rd + (warp * kRows + row) * NB + (b ^ red_swizzle<NB>(row))) =
                        make_float2(ysum[i], ysum[i + 1]);
            }
        } else {
#pragma unroll
            for (int b = 0; b < NB; ++b) rd_lane0[slot * red_slot + b * kRows] = ysum[b];
        }
        __syncwarp();
        mbar_arrive_lane0(bar0 + 8u * (kBarRedFull + slot), lane);
        if (tl_first && warp == 0 && lane == 0) BITCOS_TL(7, clock64());
        tl_first = false;
    }
    if (warp == 0 && lane == 0) BITCOS_TL(10, clock64());
    if (warp == 0 && lane == 0) BITCOS_TLP(src, 4);
    if constexpr (Segs::kHetero) {
        // Every decoder warp passes every phase of the activations' barrier, a warp without a tile in
        // this segment included: a warp that skipped one could not tell the phase before from the
        // phase after by its parity.
        if (!x_ready && !mbar_wait(bar0 + 8u * kBarX, x_parity)) {
            if (lane == 0 && pr.status(pb)) *pr.status(pb) = 1u;
            return;
        }
        more_segments = next_segment();
        tl_first = true;
        if (more_segments) {
            x_ready = false;
            x_parity ^= 1u;
            my_rbl0 = (pl.CS == 1) ? warp / pb.G : 0;
            g_fixed0 = warp - my_rbl0 * pb.G;
            my_rbl1 = (pl.CS == 1) ? (warp + pl.NW) / pb.G : 0;
            g_fixed1 = warp + pl.NW - my_rbl1 * pb.G;
        }
    } else {
        more_segments = next_segment();
    }
    } while (more_segments);
#undef pb
#undef pl
}

// One problem, this block's share of its items.
template <int FMT, int NB, bool DEBUG = true, int TPW = 1, bool XG = false, bool XQ = false, bool BL = false>
__device__ __forceinline__ void run_problem(const Problem &pr, const Plan &pl, uint8_t *smem, const Walk &wk, int block,
                                            const FirstOff *fo = nullptr, int fo_index = 0, const PrefetchList *pf = nullptr,
                                            bool first_sent = false) {
    OneSegT<DEBUG, XG, XQ, BL> one;
    one.pr = &pr;
    one.wk = wk;
    one.used = false;
    run_segments<FMT, NB, TPW>(one, pl, smem, block, fo, fo_index, pf, first_sent);
}

// (DEBUG: the instantiation that also dumps the int32 accumulators.  The dump's addresses cost registers on the tile
// loop whether it is asked for or not, so calls without it run a kernel that has no such code; the plan, and with it the
// order of the sums, is the same.)
template <int FMT, int NB, int TPW = 1, bool XG = false, bool XQ = false, bool BL = false, bool DEBUG = false>
__global__ void __launch_bounds__(max_block_threads(NB), 1) gemv_kernel(const Problem pr, const Plan pl,
                                                                        const __grid_constant__ FirstOff fo) {
    extern __shared__ __align__(128) uint8_t smem[];
    run_problem<FMT, NB, DEBUG, TPW, XG, XQ, BL>(pr, pl, smem,
                         block_walk(fo, static_cast<int>(blockIdx.x), pl, static_cast<int>(blockIdx.x), static_cast<int>(gridDim.x)),
                         static_cast<int>(blockIdx.x), &fo, static_cast<int>(blockIdx.x));
}

// Several independent BITCOS problems in one launch: the grid is cut into one range of thread
// blocks per problem, and every block runs the ordinary kernel body on its problem.
constexpr int kMaxJobs = BITCOS_MAX_JOBS;
struct MultiArgs {
    Problem pr[kMaxJobs];
    Plan pl[kMaxJobs];
    int first_block[kMaxJobs + 1];
    int n;
    // mapped = 1: block b works on job job_of[b] as that job's block number rank[b] of nblk[job]
    // (the jobs' blocks interleaved); 0: job j owns blocks first_block[j] .. first_block[j + 1] - 1
    int mapped;
    int nblk[kMaxJobs];
    uint8_t job_of[kMaxGrid];
    uint8_t rank[kMaxGrid];
    PrefetchList pf;
};

template <int NB, int TPW = 1, bool XQ = false, bool XG = false, typename FC = NoFirstCopies>
__global__ void __launch_bounds__(max_block_threads(NB), 1) gemv_multi_kernel(const __grid_constant__ MultiArgs ma,
                                                                              const __grid_constant__ FirstOff fo,
                                                                              const __grid_constant__ FC fc) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int b = static_cast<int>(blockIdx.x);
    // The block's first copies, from the host's table: before anything else is read or worked out.
    const bool first_sent = first_copy<FC>::sent(fc, b);
    if constexpr (std::is_same<FC, FirstCopiesTable>::value)
    if (first_sent && threadIdx.x == blockDim.x - 32) {
        const FirstCopies &c = fc.c[b];
        const uint32_t base = smem_addr(smem);
        const uint32_t bar_full = base + c.bar + 8u * kBarFull, bar_lut = base + c.bar + 8u * kBarLut;
        mbar_init(bar_full, 1);
        mbar_init(bar_lut, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        // (the descriptor before the arrival below, which publishes it to the decoder warps)
        *reinterpret_cast<uint4 *>(smem + c.desc_off) = make_uint4(c.desc[0], c.desc[1], c.desc[2], c.desc[3]);
        mbar_expect_tx(bar_full, c.bytes[0] + c.bytes[1] + c.bytes[2] + c.bytes[3]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i != 2 || c.bytes[2]) bulk_copy(base + c.dst[i], c.src[i], c.bytes[i], bar_full);
        mbar_expect_tx(bar_lut, kLutBytes);
        bulk_copy(base, g_bitcos_lut.v, kLutBytes, bar_lut);
    }
#ifdef BITCOS_TIMELINE
    if (threadIdx.x == blockDim.x - 32 && ma.pf.tl) ma.pf.tl[static_cast<size_t>(blockIdx.x) * 32 + 1] = clock64();
#endif
    int j = 0, bj, nbj;
    if (ma.mapped) {
        j = ma.job_of[b];
        bj = ma.rank[b];
        nbj = ma.nblk[j];
    } else {
        while (j + 1 < ma.n && b >= ma.first_block[j + 1]) ++j;
        bj = b - ma.first_block[j];
        nbj = ma.first_block[j + 1] - ma.first_block[j];
    }
    const Plan pl = ma.pl[j];      // by value: read through the run-time index once, not at every use
    const Problem pr = ma.pr[j];
    const Walk wk0 = block_walk(fo, b, pl, bj, nbj);
    // (the multi launch has no accumulator dump)
#ifdef BITCOS_TIMELINE
    if (threadIdx.x == blockDim.x - 32 && ma.pf.tl) ma.pf.tl[static_cast<size_t>(blockIdx.x) * 32 + 20] = clock64();
#endif
    run_problem<kBitcos, NB, false, TPW, XG, XQ>(pr, pl, smem, wk0,
                             bj, &fo, b,
#ifdef BITCOS_TIMELINE
                             &ma.pf
#else
                             ma.pf.n ? &ma.pf : nullptr
#endif
                             , first_sent);
}

// ---------------------------------------------------------------------------------------------
// Phased launch: jobs in dependency order inside ONE launch.  The jobs of phase p may read what the
// jobs of phase p - 1 wrote (a decoder layer's o projection follows q, k and v; down follows gate
// and up), so a thread block fetches a job's activations only after every block has finished the
// phase before it.  Everything that does not depend on the phase before -- the packed weights, their
// decode -- runs ahead: the producer warp streams the next phase's tiles while the current one is
// being decoded, and every decoder warp decodes its first tile of the next phase before it waits.
// Blocks are persistent and at most one per multiprocessor, so all of them are resident together
// and the wait on the phase counter cannot starve; it is bounded like every other wait here.
// ---------------------------------------------------------------------------------------------
constexpr int kMaxPhases = BITCOS_MAX_PHASES;
struct PhasedArgs {
    Problem pr[kMaxJobs];
    Plan pl[kMaxJobs];                      // every plan with the layout's NW and stages
    Plan layout;                            // the widest plan: shared-memory layout, barrier counts, block size
    Problem shape;                          // K = the longest row (layout only)
    int job_first_block[kMaxJobs];          // a job's range of thread blocks inside its phase
    int job_blocks[kMaxJobs];
    int expect[kMaxPhases];                 // thread blocks that have items in the phase
    int n_phases;
    unsigned int *sync;                     // device: one arrival counter per phase, zero between launches
    uint8_t job_of[kMaxPhases][kMaxGrid];   // the job a thread block works on in a phase (0xFF: none)
#ifdef BITCOS_TIMELINE
    unsigned long long *tl;
#endif
};


__device__ __forceinline__ unsigned int load_acquire(const unsigned int *p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The segments of one thread block of a phased launch: in every phase, its share of one job.
template <bool XG>
struct PhasedSegs {
    typedef ParamView View;
    static constexpr bool kSingle = false;
    static constexpr bool kHetero = true;
    static constexpr bool kListsLate = false;
    static constexpr bool kDebug = false;
    static constexpr bool kGroupScales = XG;
    static constexpr bool kQuantize = false;
    static constexpr bool kBlend = false;
    const PhasedArgs *pa;
    int block;               // blockIdx.x
    int next_phase;          // phase the next call of next() looks at
    int phase;               // phase of the current segment
    int rel_block;           // this block's index inside the current job's range
    Problem cur_pb;
    Plan cur_pl;
    __device__ __forceinline__ const Problem &shape() const { return pa->shape; }
    __device__ __forceinline__ const Problem *problem_ptr() const { return &cur_pb; }
    __device__ __forceinline__ const Plan *plan_ptr() const { return &cur_pl; }
    __device__ __forceinline__ int block_in_job(int) const { return rel_block; }
    __device__ __forceinline__ bool next(View &, Walk &w) {
        while (next_phase < pa->n_phases) {
            const int p = next_phase++;
            const int j = pa->job_of[p][block];
            if (j == 0xFF) continue;
            const int rel = block - pa->job_first_block[j];
            const Walk wj = make_walk(pa->pl[j], rel, pa->job_blocks[j]);
            if (wj.count <= 0) continue;
            cur_pb = pa->pr[j];
            cur_pl = pa->pl[j];
            w = wj;
            phase = p;
            rel_block = rel;
            return true;
        }
        return false;
    }
    // Epilogue warp, before it fetches the current segment's activations: every block that has items
    // in the phase before must have written its outputs.  false if the wait ran out.
    __device__ __forceinline__ bool wait_dependency(int lane) const {
        if (phase == 0) return true;
        bool ok = true;
        if (lane == 0) {
            const unsigned int *ctr = pa->sync + (phase - 1);
            const unsigned int want = static_cast<unsigned int>(pa->expect[phase - 1]);
            uint64_t t0 = 0;
            for (uint32_t i = 0; load_acquire(ctr) < want; ++i) {
                if ((i & 15u) == 15u) {
                    const uint64_t now = global_timer_ns();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > kWaitLimitNs) {
                        ok = false;
                        break;
                    }
                }
            }
            // what the other blocks wrote, ordered before this block's asynchronous copies
            asm volatile("fence.proxy.async;" ::: "memory");
        }
        return __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0;
    }
    // Epilogue warp, after the last output of the current segment: count this block in.  The last
    // arrival of the last phase leaves every counter zero for the next launch (by then no block
    // reads an earlier counter any more: each one read it before it arrived here).
    __device__ __forceinline__ void signal_done(int lane) const {
        __syncwarp();
        if (lane != 0) return;
        __threadfence();
        const unsigned int old = atomicAdd(pa->sync + phase, 1u);
        if (phase == pa->n_phases - 1 && old + 1u == static_cast<unsigned int>(pa->expect[phase])) {
            for (int p = 0; p < pa->n_phases; ++p) pa->sync[p] = 0u;
        }
    }
};

template <int NB, bool XG = false>
__global__ void __launch_bounds__(max_block_threads(NB), 1) gemv_phased_kernel(const __grid_constant__ PhasedArgs pa) {
    extern __shared__ __align__(128) uint8_t smem[];
    PhasedSegs<XG> segs;
    segs.pa = &pa;
    segs.block = static_cast<int>(blockIdx.x);
    segs.next_phase = 0;
    segs.phase = 0;
    segs.rel_block = 0;
    run_segments<kBitcos, NB, 1>(segs, pa.layout, smem, static_cast<int>(blockIdx.x));
}

// Fills in what differs between the groups of a grouped product; false if the group is empty or
// names no expert.
template <int NB>
__device__ __forceinline__ bool grouped_problem(Problem &pr, const Problem &base, const GroupedArgs &ga, int grp) {
    const GroupDesc gd = read_group(ga, base.xrow, base.status, grp, NB);
    if (!gd.ok || gd.empty) return false;
    const int e = gd.e, begin = gd.begin, end = gd.end;
    const bitcos_weights wdesc = ga.experts[e];
    pr = base;
    pr.payload = wdesc.bitmap;
    pr.signs = wdesc.signs;
    pr.tile_off = wdesc.tile_off;
    pr.scales = wdesc.scales;
    pr.nb = min(end - begin, NB);
    pr.xrow = base.xrow + begin;
    pr.out_row0 = begin;
    uint8_t *ws = reinterpret_cast<uint8_t *>(base.status) + static_cast<size_t>(grp) * ga.ws_stride;
    pr.status = reinterpret_cast<unsigned int *>(ws);
    pr.counters = reinterpret_cast<unsigned int *>(ws + kHeaderBytes);
    pr.partial = reinterpret_cast<float *>(ws + kHeaderBytes + ((static_cast<size_t>(base.RB) * 4 + 255) / 256 * 256));
    return true;
}

// PARTS: groups have up to 2 NB tokens, those of more than NB run as two parts of at most NB: the groups' parts in order,
// found by a warp from the routing lists.  All lanes take part; the lists are read (and checked) again where they are used.
template <int NB>
__device__ __forceinline__ bool two_parts(const GroupedArgs &ga, int g) {
    return static_cast<int64_t>(__ldg(ga.group_begin + g + 1)) - __ldg(ga.group_begin + g) > NB;
}
template <int NB>
__device__ __forceinline__ int count_parts(const GroupedArgs &ga, int n_groups) {
    int extra = 0;
    for (int g = threadIdx.x & 31; g < n_groups; g += 32) extra += two_parts<NB>(ga, g) ? 1 : 0;
    return n_groups + __reduce_add_sync(0xFFFFFFFFu, extra);
}
// group and part of the part number `part` (< count_parts)
template <int NB>
__device__ __forceinline__ void find_part(const GroupedArgs &ga, int n_groups, int part, int &grp, int &half) {
    const int lane = threadIdx.x & 31;
    for (int base = 0; base < n_groups; base += 32) {
        const int g = base + lane;
        const bool in = g < n_groups, two = in && two_parts<NB>(ga, g);
        const uint32_t twos = __ballot_sync(0xFFFFFFFFu, two);
        const int at = lane + __popc(twos & ((1u << lane) - 1u));      // this group's first part, counted from the chunk's
        const uint32_t hit = __ballot_sync(0xFFFFFFFFu, in && at <= part && part <= at + (two ? 1 : 0));
        if (hit) {
            const int j = __ffs(hit) - 1;
            grp = base + j;
            half = part - __shfl_sync(0xFFFFFFFFu, at, j);
            return;
        }
        part -= 32 + __popc(twos);
    }
    grp = n_groups;
    half = 0;
}

// The pieces of the groups that fall into one thread block's range of the flat item list.
template <int NB, bool DEBUG, bool PARTS>
struct GroupedSegs {
    const Problem *base;
    const GroupedArgs *ga;
    int64_t lo, hi, ipg;      // this block's range of the list; items per group (or part)
    int grp;                  // group of item lo
    int half, shift;          // PARTS: which of the group's parts that is; parts beyond the first in front of it
    typedef GroupView View;
    static constexpr bool kSingle = false;
    static constexpr bool kHetero = false;
    static constexpr bool kListsLate = true;   // the routing lists are read only after the previous kernel has completed
    static constexpr bool kDebug = DEBUG;
    static constexpr bool kGroupScales = false;
    static constexpr bool kQuantize = false;
    static constexpr bool kBlend = false;
    __device__ __forceinline__ const Problem &shape() const { return *base; }
    __device__ __forceinline__ int block_in_job(int block) const { return block; }
    __device__ __forceinline__ bool next(View &v, Walk &w) {
        while (lo < hi) {
            const int64_t g_lo = static_cast<int64_t>(PARTS ? grp + shift + half : grp) * ipg;
            const int64_t seg_hi = hi < g_lo + ipg ? hi : g_lo + ipg;
            w.first = static_cast<int>(lo - g_lo);
            w.count = static_cast<int>(seg_hi - lo);
            w.cstride = 1;
            w.q = 1;
            w.rem = 0;
            lo = seg_hi;
            const int g = grp, h = PARTS ? half : 0;
            const GroupDesc gd = read_group(*ga, base->xrow, base->status, g, PARTS ? 2 * NB : NB);
            if (PARTS && h == 0 && static_cast<int64_t>(gd.end) - gd.begin > NB) {
                half = 1;
            } else {
                ++grp;
                if (PARTS) {
                    shift += h;
                    half = 0;
                }
            }
            if (!gd.ok || gd.empty) continue;
            const int begin = gd.begin + h * NB;
            const bitcos_weights *wd = ga->experts + gd.e;
            v.payload_ = wd->bitmap;
            v.signs_ = wd->signs;
            v.tile_off_ = wd->tile_off;
            v.scales_ = wd->scales;
            v.xrow_ = base->xrow + begin;
            v.status_ = reinterpret_cast<unsigned int *>(reinterpret_cast<uint8_t *>(base->status) +
                                                         static_cast<size_t>(g) * ga->ws_stride);
            v.begin_ = begin;
            v.nb_ = min(gd.end - begin, NB);
            return true;
        }
        return false;
    }
};

// Grouped product.  Two launch shapes.  Flat (rows in one piece, no cross-block sums): the items
// of all groups form one list, cut into equal contiguous ranges, one per thread block; a block
// that crosses from one group to the next keeps its pipeline running (the producer is already
// copying the next group's weights while the last tiles of this one are decoded).  Otherwise:
// blockIdx.y = group, and the blocks of a row of the grid share that group's items.
template <int FMT, int NB, bool DEBUG, bool PARTS>
__global__ void __launch_bounds__(max_block_threads(NB), 1) gemv_grouped_kernel(const __grid_constant__ Problem base, const Plan pl,
                                                                                const __grid_constant__ GroupedArgs ga) {
    extern __shared__ __align__(128) uint8_t smem[];
    int n_groups = ga.n_groups;
    if (ga.n_groups_dev) {
        // the number of groups itself comes from the device (a grouping kernel earlier in the stream)
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const int n = __ldg(ga.n_groups_dev);
        n_groups = n < 0 ? 0 : (n < n_groups ? n : n_groups);
    }
    if (!ga.flat) {
        // the routing lists may come from the previous kernel in the stream
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (static_cast<int>(blockIdx.y) >= n_groups) return;
        Problem pr;
        if (!grouped_problem<NB>(pr, base, ga, static_cast<int>(blockIdx.y))) return;
        run_problem<FMT, NB, DEBUG>(pr, pl, smem, make_walk(pl, static_cast<int>(blockIdx.x), static_cast<int>(gridDim.x)),
                                 static_cast<int>(blockIdx.x));
        return;
    }
    int parts = n_groups;
    if constexpr (PARTS) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        parts = count_parts<NB>(ga, n_groups);
    }
    const int64_t ipg = pl.items, total = ipg * parts;
    const int64_t nblk = gridDim.x, b = blockIdx.x;
    const int64_t q = total / nblk, rem = total - q * nblk;
    GroupedSegs<NB, DEBUG, PARTS> segs;
    segs.base = &base;
    segs.ga = &ga;
    segs.ipg = ipg;
    segs.lo = b * q + (b < rem ? b : rem);
    segs.hi = segs.lo + q + (b < rem ? 1 : 0);
    segs.grp = static_cast<int>(segs.lo / ipg);
    segs.half = segs.shift = 0;
    if constexpr (PARTS) {
        const int part = segs.grp;
        find_part<NB>(ga, n_groups, part, segs.grp, segs.half);
        segs.shift = part - segs.half - segs.grp;
    }
    run_segments<FMT, NB, 1>(segs, pl, smem, static_cast<int>(b));
}

// ---------------------------------------------------------------------------------------------
// Host side of the device entry points.
// ---------------------------------------------------------------------------------------------
inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline int check_cuda(cudaError_t e) {
    if (e == cudaSuccess) return BITCOS_OK;
    g_last_cuda_error = static_cast<int>(e);
    return BITCOS_ERR_CUDA;
}

// Number of multiprocessors of the current device.  The opt-in to large dynamic shared memory is
// done on the first call for a given kernel instantiation and device and remembered (so that
// first call must not happen during stream capture; later calls only read the cache).
template <auto kernel>
int prepare_kernel(int *sms_out, int *smem_budget_out) {
    constexpr int kMaxDev = 32;
    static int cache[kMaxDev][2];      // [0] multiprocessor count (0 = not prepared yet), [1] dynamic smem budget
    int dev = 0;
    int rc = check_cuda(cudaGetDevice(&dev));
    if (rc) return rc;
    if (dev < kMaxDev && cache[dev][0] > 0) {
        *sms_out = cache[dev][0];
        *smem_budget_out = cache[dev][1];
        return BITCOS_OK;
    }
    int sms = 0, max_smem = 0;
    rc = check_cuda(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (rc) return rc;
    rc = check_cuda(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    if (rc) return rc;
    const int budget = max_smem - 1024;
    rc = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, budget));
    if (rc) return rc;
    if (dev < kMaxDev) {
        cache[dev][1] = budget;
        cache[dev][0] = sms;
    }
    *sms_out = sms;
    *smem_budget_out = budget;
    return BITCOS_OK;
}

// Ring depth: as many stages as fit next to the tables, activations and partial sums (the loaded
// DRAM latency of this part needs on the order of 100 KB in flight per multiprocessor).
inline int choose_stages(int fmt, const Plan &pl, int G, int nb, int64_t K, int smem_budget, bool scr) {
    Plan p = pl;
    for (int st = kMaxStages; st > 2; --st) {
        p.stages = st;
        if (static_cast<int>(smem_layout(fmt, p, G, nb, K, scr).total) <= smem_budget) return st;
    }
    return 2;
}

// How the items are handed to thread blocks, and how many blocks to launch (persistent: at most
// one per multiprocessor).  Cost model in units of one item's time: round robin over row-block
// chunks costs ceil(chunks / blocks) * CS items per block and never shares a row block; a
// contiguous balanced split costs ceil(items / blocks) items plus, when rows are split into
// column blocks, the cross-block hand-shake at the end (worth about 2.5 items).
// BITCOS_WALK=cyclic|contiguous overrides the choice (for A/B runs).
// A launch with no more items than multiprocessors would give every block one item and spread
// over most of the machine.  Under programmatic dependent launch the NEXT kernel's blocks start
// early (table, first weights, first decode, all before its dependency is resolved) only on
// multiprocessors this launch leaves free, and blocks that start late pay their whole start-up
// after the dependency; so such a launch takes a little under half of the multiprocessors and two
// items per block instead (measured on the decoder-layer sequence: 16.5 -> 16.05 us per pass; the
// step is sharp: the blocks of two consecutive small launches must fit side by side).
inline int small_launch_cap(int64_t items, int sms) {
    if (items > sms) return sms;
    const int cap = sms * 46 / 100;
    static const char *env = std::getenv("BITCOS_SMALL_FULL");
    if ((!env || env[0] != '0') && items <= sms - cap) return static_cast<int>(items);
    return cap < 1 ? 1 : cap;
}

inline void choose_walk(Plan &pl, int sms, int *grid) {
    static const char *force = std::getenv("BITCOS_WALK");
    const int64_t chunks = pl.items / pl.CS;
    const int64_t g_cyc = chunks < sms ? chunks : sms, g_con = pl.items < sms ? pl.items : sms;
    const double cost_cyc = static_cast<double>((chunks + g_cyc - 1) / g_cyc) * pl.CS;
    const double cost_con = static_cast<double>((pl.items + g_con - 1) / g_con) + (pl.CS > 1 ? 2.5 : 0.0);
    int cyclic = cost_cyc <= cost_con ? 1 : 0;
    if (force && force[0] == 'c' && force[1] == 'y') cyclic = 1;
    if (force && force[0] == 'c' && force[1] == 'o') cyclic = 0;
    pl.cyclic = cyclic;
    *grid = static_cast<int>(cyclic ? g_cyc : g_con);
    pl.wq = cyclic ? 1 : static_cast<int>(pl.items / *grid);
    pl.wrem = cyclic ? 0 : static_cast<int>(pl.items - static_cast<int64_t>(pl.wq) * *grid);
}

// Launches with programmatic stream serialization, so that this kernel's prologue (barrier
// set-up, table and first weight copies) may overlap the tail of the previous kernel in the
// stream.  BITCOS_PDL=0 turns it off (for A/B runs).
// (arguments of exactly the kernel's types, taken by reference: the largest are 7 KB, and every copy on the way counts
// against launches of 2 us)
template <typename... KArgs, typename... Args>
int launch_pdl(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t stream, const Args &...args) {
    static_assert(std::is_same<std::tuple<typename std::remove_cv<KArgs>::type...>, std::tuple<Args...>>::value, "the kernel's own types");
    static const char *env = std::getenv("BITCOS_PDL");
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = (env && env[0] == '0') ? 0 : 1;
    void *pointers[] = {const_cast<void *>(static_cast<const void *>(&args))...};
    return check_cuda(cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(kernel), pointers));
}

// While a launch sequence is being recorded for replay (bitcos_gemv_phases_host), every value a
// plan takes from a host copy of tile_off is noted here, so that a replay can make sure that the
// values it was built from are still there.
inline thread_local std::vector<std::pair<const uint32_t *, uint32_t>> *g_offset_log = nullptr;
inline uint32_t host_offset(const uint32_t *off_host, int64_t i) {
    const uint32_t v = off_host[i];
    if (g_offset_log) g_offset_log->emplace_back(off_host + i, v);
    return v;
}

// Fills fo.lo / fo.hi [base .. base + grid) from a host copy of tile_off: the sign-vector range of
// the first item of each of the `grid` thread blocks that share the problem.
inline void fill_first_off(FirstOff &fo, int base, const uint32_t *off_host, const Problem &pr, const Plan &pl, int grid) {
    if (base + grid > kMaxGrid) {
        fo.valid = 0;
        fo.walks = 0;
        return;
    }
    if (!off_host) fo.valid = 0;
    // (make_walk for every block, with its divisions once: 148 blocks took 3 us of the caller's time)
    const int items = static_cast<int>(pl.items), units = pl.cyclic ? items / pl.CS : items;
    const int q = units / grid, rem = units - q * grid;
    for (int b = 0, first = 0; b < grid; ++b) {
        const int count = q + (b < rem ? 1 : 0);
        fo.first[base + b] = pl.cyclic ? b * pl.CS : first;
        fo.count[base + b] = pl.cyclic ? count * pl.CS : count;
        if (fo.valid) {
            fo.lo[base + b] = fo.hi[base + b] = 0;
            if (count > 0) {
                ItemIter it;
                if (pl.cyclic) {
                    it.c = b;
                    it.cs = 0;
                } else {
                    it.init(pl, first);
                }
                const ItemRange r = item_range(pr, pl, it.c, it.cs);
                fo.lo[base + b] = host_offset(off_host, r.t0);
                fo.hi[base + b] = host_offset(off_host, r.t0 + r.nt);
            }
        }
        first += count;
    }
}

// Large matrices, one or two tokens: items of twice the size, two tiles per decoder warp, so that
// what a decoder warp does per item (barrier waits, descriptor, stage advance, hand-off of the
// partial sums: about 50 of its 364 instructions per tile) is paid once per two tiles.  Only when
// every block still gets several items: from eight of the one-tile items per multiprocessor on.  (Between
// three and eight the gain depends on the shape and the format: 8192x5120 -3 % at one token but +6 % at
// two, 4096x12288 +3 %, 2-bit +3 %; so those keep one tile per warp.)
// In fragment order a warp's two tiles also share one set of partial sums (added in registers: half the stores, and
// half the additions of the epilogue warp) and the decode runs product by product, so the line lies lower, from 64
// tiles per multiprocessor on.  Below it, 2x6912x2560 in one launch (58 tiles): layer pass 17.2 -> 17.9 us at two
// tokens, 20.2 -> 22.2 at eight; above it, 8192x5120 (69 tiles): 6.80 -> 6.77, 8.41 -> 7.93, 12.0 -> 11.4 at sixteen;
// 25600x5120 (216): 15.8 -> 15.5, 19.8 -> 18.1, 31.1 -> 27.1.
inline bool wants_two_tiles(int fmt, int64_t items, int64_t tiles, int nb_template, int sms) {
    if (fragment_order(fmt, nb_template)) return tiles >= 64 * static_cast<int64_t>(sms);
    return nb_template < kMmaMinBatch && items >= 8 * static_cast<int64_t>(sms);
}
inline int64_t tile_count(int64_t M, int64_t K) { return padded_rows(M) / kRows * (K / kGroup); }
// The plan of such a product.
inline Plan two_tile_plan(int fmt, int64_t M, int64_t K, int nb_template, bool own_order = false) {
    return fragment_order(fmt, nb_template) ? make_run_plan(M, K, decoder_warps(nb_template), wide_tiles(fmt, nb_template), own_order)
                                            : make_plan(M, K, decoder_warps(nb_template), 2);
}

// A launch of one product's kernel (set up for large shared memory on its first use).
template <auto kernel>
int launch_single(const Problem &pr, const Plan &plw, const FirstOff &fo, int grid, uint32_t smem, cudaStream_t stream) {
    int sms = 0, budget = 0;
    const int rc = prepare_kernel<kernel>(&sms, &budget);
    return rc ? rc : launch_pdl(kernel, dim3(grid), (plw.NW + 2) * 32, smem, stream, pr, plw, fo);
}

template <int FMT, int NB, bool XG = false, bool XQ = false, bool BL = false>
int launch(const Problem &pr, const Plan &pl_in, cudaStream_t stream, const uint32_t *off_host = nullptr) {
    // the one- and two-token instantiations keep the activations in shared memory (nb_bucket sees to it)
    if (NB < kMmaMinBatch && static_cast<int64_t>(NB) * pr.K > kXResidentBytes) return BITCOS_ERR_SHAPE;
    constexpr bool kTwo = NB < kMmaMinBatch || fragment_order(FMT, NB);      // a two-tile instantiation exists
    constexpr bool kScr = NB >= kMmaMinBatch && !fragment_order(FMT, NB);
    int sms = 0, budget = 0;
    int rc = prepare_kernel<gemv_kernel<FMT, NB, 1, XG, XQ, BL>>(&sms, &budget);
    if (rc) return rc;
    // (with and without the accumulator dump: the same plan, so the same order of the sums)
    const bool two = kTwo && wants_two_tiles(FMT, pl_in.items, tile_count(pr.M, pr.K), NB, sms);
    const Plan pl = two ? two_tile_plan(FMT, pr.M, pr.K, NB, BL) : pl_in;
    int grid = 1;
    Plan plw = pl;
    choose_walk(plw, small_launch_cap(pl.items, sms), &grid);
    plw.stages = choose_stages(FMT, pl, pr.G, NB, pr.K, budget, kScr);
    const SmemLayout L = smem_layout(FMT, plw, pr.G, NB, pr.K, kScr);
    FirstOff fo;
    fo.valid = (FMT == kBitcos && off_host) ? 1 : 0;
    fo.walks = 1;
    fill_first_off(fo, 0, off_host, pr, plw, grid);
    if constexpr (kTwo) {
        constexpr int kWide = wide_tiles(FMT, NB);
        if constexpr (!BL) {
            if (two && pr.acc_debug) return launch_single<gemv_kernel<FMT, NB, kWide, XG, XQ, false, true>>(pr, plw, fo, grid, L.total, stream);
        }
        if (two) return launch_single<gemv_kernel<FMT, NB, kWide, XG, XQ, BL>>(pr, plw, fo, grid, L.total, stream);
    }
    if constexpr (!BL) {
        if (pr.acc_debug) return launch_single<gemv_kernel<FMT, NB, 1, XG, XQ, false, true>>(pr, plw, fo, grid, L.total, stream);
    }
    return launch_pdl(gemv_kernel<FMT, NB, 1, XG, XQ, BL>, dim3(grid), (pl.NW + 2) * 32, L.total, stream, pr, plw, fo);
}

// The copies of a thread block's first item, as issue_item<kBitcos> would issue them into stage 0
// (first = the block's first item, o_lo / o_hi = entry offsets of its first tile and of the tile
// after its last).
inline void fill_first_copies(FirstCopies &c, const Problem &pr, const Plan &pl, const SmemLayout &L, int first, uint32_t o_lo,
                              uint32_t o_hi) {
    ItemIter it;
    it.init(pl, first);
    const ItemRange r = item_range(pr, pl, it.c, it.cs);
    const uint32_t b_lo = (o_lo >> 7) << 4, b_hi = ((o_hi + 127u) >> 7) << 4;
    const uint32_t o_first = static_cast<uint32_t>(r.t0 & 3);
    c.src[0] = pr.tile_off + (r.t0 - o_first);
    c.bytes[0] = ((o_first + static_cast<uint32_t>(r.nt) + 1u + 3u) & ~3u) * 4u;
    c.src[1] = reinterpret_cast<const uint8_t *>(pr.payload) + r.t0 * 512;
    c.bytes[1] = static_cast<uint32_t>(r.nt) * 512u;
    c.src[2] = reinterpret_cast<const uint8_t *>(pr.signs) + b_lo;
    c.bytes[2] = b_hi - b_lo;
    c.src[3] = reinterpret_cast<const uint8_t *>(pr.scales) + r.t0 * 64;
    c.bytes[3] = static_cast<uint32_t>(r.nt) * 64u;
    c.dst[1] = L.stage;
    c.dst[2] = c.dst[1] + L.payload_cap;
    c.dst[3] = c.dst[2] + L.sign_cap;
    c.dst[0] = c.dst[3] + L.scale_cap;
    c.desc[0] = static_cast<uint32_t>(r.nt) | (o_first << 8);
    c.desc[1] = static_cast<uint32_t>(r.g0);
    c.desc[2] = static_cast<uint32_t>(r.rb0);
    c.desc[3] = b_lo * 8u;
    c.desc_off = L.bar + 384u;
    c.bar = L.bar;
}

// Multiprocessors shared between n jobs in proportion to their items: cap[j] of at most sms altogether, at least one each.  (The
// blocks that the smallest jobs are rounded up to come from the largest: no launch is wider than the machine, and of a
// phased launch every block is resident.)
inline void share_multiprocessors(const int64_t *items, int n, int sms, int64_t *cap) {
    int64_t total = 0, sum = 0;
    for (int j = 0; j < n; ++j) total += items[j];
    for (int j = 0; j < n; ++j) {
        cap[j] = items[j];
        if (total > sms) cap[j] = std::max<int64_t>(1, items[j] * sms / total);
        sum += cap[j];
    }
    for (; sum > std::max(sms, n); --sum) --*std::max_element(cap, cap + n);
}

// Grids of a multi launch: whether it runs two tiles per decoder warp, and each job's plan, walk
// and number of thread blocks (the multiprocessors shared between the jobs in proportion to their
// item counts).  Returns the total number of blocks.
inline int plan_multi(MultiArgs &ma, int nb_template, int sms, bool *two_out, int *grids) {
    int64_t total_items = 0;
    for (int j = 0; j < ma.n; ++j) {
        ma.pl[j] = one_tile_plan(kBitcos, ma.pr[j].M, ma.pr[j].K, nb_template);
        total_items += ma.pl[j].items;
    }
    // enough items altogether: every problem with two tiles per decoder warp
    int64_t tiles = 0;
    for (int j = 0; j < ma.n; ++j) tiles += tile_count(ma.pr[j].M, ma.pr[j].K);
    const bool two = wants_two_tiles(kBitcos, total_items, tiles, nb_template, sms);
    if (two) {
        total_items = 0;
        for (int j = 0; j < ma.n; ++j) {
            ma.pl[j] = two_tile_plan(kBitcos, ma.pr[j].M, ma.pr[j].K, nb_template);
            total_items += ma.pl[j].items;
        }
    }
    *two_out = two;
    sms = small_launch_cap(total_items, sms);
    int64_t items[kMaxJobs], cap[kMaxJobs];
    for (int j = 0; j < ma.n; ++j) items[j] = ma.pl[j].items;
    share_multiprocessors(items, ma.n, sms, cap);
    int next = 0;
    for (int j = 0; j < ma.n; ++j) {
        choose_walk(ma.pl[j], static_cast<int>(cap[j]), &grids[j]);
        next += grids[j];
    }
    return next;
}

// A launch whose first `early` thread blocks (of `grid`) find a free multiprocessor at once while
// the others have to wait for the blocks of the kernel before it to leave: by the time a late
// block has gone through its start-up, an early one -- which did all of that, first decode
// included, while it waited for its dependency -- is about kLateLagItems items ahead.  So early
// blocks take that many items more.  Only for jobs whose items are whole row blocks (nothing is
// shared between thread blocks, so the split has no influence on any sum).  counts[r] = items of
// the job's block number r; its early blocks come first.
constexpr int kLateLagItems = 2;
inline void skewed_counts(int64_t items, int n_early, int n_late, int *counts) {
    const int n = n_early + n_late;
    int64_t a = (items + static_cast<int64_t>(n_late) * kLateLagItems + n - 1) / n;
    if (a < 1) a = 1;
    int64_t sum = 0;
    for (int r = 0; r < n; ++r) {
        int64_t c = r < n_early ? a : a - kLateLagItems;
        if (c < 0) c = 0;
        counts[r] = static_cast<int>(c);
        sum += c;
    }
    // too many by rounding: taken back one at a time, from the last block backwards
    for (int r = n - 1; sum > items; r = (r == 0 ? n - 1 : r - 1))
        if (counts[r] > 0) {
            --counts[r];
            --sum;
        }
    for (int r = 0; sum < items; r = (r + 1) % n) {       // (too few: only when a - lag was cut at zero)
        ++counts[r];
        ++sum;
    }
}

// Whether a launch's blocks are split into early and late ones, and if so the split: block b works on
// job job_of[b] as that job's block number rank[b] and takes count[b] items from item first[b] of the job
// (early blocks are dealt to the jobs in proportion to their grids, job after job, then the late ones;
// inside a job, contiguous ranges of its items, early blocks first).
inline bool skewed_assignment(MultiArgs &ma, const int *grids, int total, bool two, int sms, int busy_sms, int *first, int *count) {
    // late starters: only when part of the grid starts early and part late, and every job's items are whole rows
    const int early = sms - busy_sms;
    bool skew = busy_sms > 0 && early > 0 && early < total && total <= kMaxGrid && !two;
    for (int j = 0; j < ma.n; ++j) skew = skew && ma.pl[j].CS == 1 && ma.pl[j].items >= grids[j];
    if (!skew) return false;
    int ne[kMaxJobs], given = 0;
    for (int j = 0; j < ma.n; ++j) {
        ne[j] = static_cast<int>(static_cast<int64_t>(early) * grids[j] / total);
        given += ne[j];
    }
    for (int j = 0; given < early; j = (j + 1) % ma.n)
        if (ne[j] < grids[j]) {
            ++ne[j];
            ++given;
        }
    int b = 0;
    for (int pass = 0; pass < 2; ++pass)
        for (int j = 0; j < ma.n; ++j) {
            const int r0 = pass ? ne[j] : 0, r1 = pass ? grids[j] : ne[j];
            for (int r = r0; r < r1; ++r, ++b) {
                ma.job_of[b] = static_cast<uint8_t>(j);
                ma.rank[b] = static_cast<uint8_t>(r);
            }
        }
    static thread_local int counts[kMaxJobs][kMaxGrid], firsts[kMaxJobs][kMaxGrid];
    for (int j = 0; j < ma.n; ++j) {
        ma.nblk[j] = grids[j];
        ma.pl[j].cyclic = 0;
        skewed_counts(ma.pl[j].items, ne[j], grids[j] - ne[j], counts[j]);
        int f = 0;
        for (int r = 0; r < grids[j]; ++r) {
            firsts[j][r] = f;
            f += counts[j][r];
        }
    }
    for (b = 0; b < total; ++b) {
        first[b] = firsts[ma.job_of[b]][ma.rank[b]];
        count[b] = counts[ma.job_of[b]][ma.rank[b]];
    }
    ma.first_block[ma.n] = total;
    ma.mapped = 1;
    return true;
}

// busy_sms: multiprocessors the caller expects the kernel before this one in the stream to hold on
// to when this launch's blocks are scheduled (0: unknown or none).
template <int NB, bool XQ = false, bool XG = false>
int launch_multi(MultiArgs &ma, cudaStream_t stream, const uint32_t *const *off_host, int busy_sms = 0) {
    for (int j = 0; j < ma.n; ++j)
        if (NB < kMmaMinBatch && static_cast<int64_t>(NB) * ma.pr[j].K > kXResidentBytes) return BITCOS_ERR_SHAPE;
    int sms = 0, budget = 0;
    int rc = prepare_kernel<gemv_multi_kernel<NB, 1, XQ, XG>>(&sms, &budget);
    if (rc) return rc;
    if constexpr (!XQ && !XG && NB <= 2) {
        // (the variant that is only launched while a graph is being recorded is set up here, on whichever call comes first)
        rc = prepare_kernel<gemv_multi_kernel<NB, 1, false, false, FirstCopiesTable>>(&sms, &budget);
        if (rc) return rc;
    }
    bool two = false;
    int grids[kMaxJobs];
    const int total = plan_multi(ma, NB, sms, &two, grids);
    if (two) {
        rc = prepare_kernel<gemv_multi_kernel<NB, wide_tiles(kBitcos, NB), XQ, XG>>(&sms, &budget);
        if (rc) return rc;
    }
    int nw = 0;
    uint32_t smem = 0;
    FirstOff fo;
    fo.valid = 1;
    fo.walks = 1;
    for (int j = 0; j < ma.n; ++j) fo.valid = (fo.valid && off_host[j]) ? 1 : 0;
    for (int j = 0; j < ma.n; ++j) {
        ma.pl[j].stages = choose_stages(kBitcos, ma.pl[j], ma.pr[j].G, NB, ma.pr[j].K, budget, false);
        const SmemLayout L = smem_layout(kBitcos, ma.pl[j], ma.pr[j].G, NB, ma.pr[j].K, false);
        if (L.total > smem) smem = L.total;
        if (ma.pl[j].NW > nw) nw = ma.pl[j].NW;
    }
    if (!skewed_assignment(ma, grids, total, two, sms, busy_sms, fo.first, fo.count)) {
        int next = 0;
        for (int j = 0; j < ma.n; ++j) {
            ma.first_block[j] = next;
            fill_first_off(fo, next, fo.valid ? off_host[j] : nullptr, ma.pr[j], ma.pl[j], grids[j]);
            next += grids[j];
        }
        ma.first_block[ma.n] = next;
        ma.mapped = 0;
    } else {
        for (int b = 0; b < total; ++b) {
            const int j = ma.job_of[b];
            fo.lo[b] = fo.hi[b] = 0;
            if (fo.valid && fo.count[b] > 0) {
                ItemIter it;
                it.init(ma.pl[j], fo.first[b]);
                const ItemRange ir = item_range(ma.pr[j], ma.pl[j], it.c, it.cs);
                fo.lo[b] = host_offset(off_host[j], ir.t0);
                fo.hi[b] = host_offset(off_host[j], ir.t0 + ir.nt);
            }
        }
    }
    // every block's first copies, when the entry offsets are known on the host
    static thread_local FirstCopiesTable fc;
    static const char *fc_env = std::getenv("BITCOS_FIRST_COPIES");      // 0: never, 1: also on plain stream launches (A/B runs)
    fc.valid = 0;
    bool recording = false;
    {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &cs) == cudaSuccess) recording = cs == cudaStreamCaptureStatusActive;
        else cudaGetLastError();
    }
    const bool with_table = !XQ && !XG && NB <= 2 && !two && (recording || (fc_env && fc_env[0] == '1')) && !(fc_env && fc_env[0] == '0');
    if (with_table && fo.valid && fo.walks && total <= kMaxGrid) {
        fc.valid = 1;
        int jb = 0;
        for (int b = 0; b < total; ++b) {
            int j;
            if (ma.mapped) {
                j = ma.job_of[b];
            } else {
                while (jb + 1 < ma.n && b >= ma.first_block[jb + 1]) ++jb;
                j = jb;
            }
            fc.c[b] = FirstCopies{};
            if (fo.count[b] <= 0) continue;
            const SmemLayout L = smem_layout(kBitcos, ma.pl[j], ma.pr[j].G, NB, ma.pr[j].K, false);
            fill_first_copies(fc.c[b], ma.pr[j], ma.pl[j], L, fo.first[b], fo.lo[b], fo.hi[b]);
        }
    }
    if constexpr (!XQ && !XG && NB <= 2) {
        if (fc.valid) {
            return launch_pdl(gemv_multi_kernel<NB, 1, false, false, FirstCopiesTable>, dim3(total), (nw + 2) * 32, smem, stream, ma, fo, fc);
        }
    }
    const NoFirstCopies none{0};
    if (two) return launch_pdl(gemv_multi_kernel<NB, wide_tiles(kBitcos, NB), XQ, XG>, dim3(total), (nw + 2) * 32, smem, stream, ma, fo, none);
    return launch_pdl(gemv_multi_kernel<NB, 1, XQ, XG>, dim3(total), (nw + 2) * 32, smem, stream, ma, fo, none);
}

// Which instantiation serves a batch: 1, 2, 4, 8 or 16 tokens.  The one- and two-token paths read
// the activations from shared memory; when those do not fit there (K beyond 48 K / 24 K), the
// tensor-core path, which takes its activation fragments from global memory, is the faster one.
inline int nb_bucket(int batch, int64_t K) {
    if (batch <= 2 && static_cast<int64_t>(batch) * K > kXResidentBytes) return 4;
    return batch <= 1 ? 1 : batch <= 2 ? 2 : batch <= 4 ? 4 : batch <= 8 ? 8 : 16;
}

template <int FMT, bool XG = false>
int launch_nb(const Problem &pr, const Plan &pl, cudaStream_t stream, const uint32_t *off_host) {
    const int nbk = nb_bucket(pr.nb, pr.K);
    if (nbk == 1) return launch<FMT, 1, XG>(pr, pl, stream, off_host);
    if (nbk == 2) return launch<FMT, 2, XG>(pr, pl, stream, off_host);
    if (pr.nb <= 4) return launch<FMT, 4, XG>(pr, pl, stream, off_host);
    if (pr.nb <= 8) return launch<FMT, 8, XG>(pr, pl, stream, off_host);
    return launch<FMT, 16, XG>(pr, pl, stream, off_host);
}

template <int FMT, int NB, bool PARTS = false>
int launch_grouped(const Problem &pr, const Plan &pl, const GroupedArgs &ga, int n_groups, cudaStream_t stream) {
    if (NB < kMmaMinBatch && static_cast<int64_t>(NB) * pr.K > kXResidentBytes) return BITCOS_ERR_SHAPE;
    constexpr bool kScr = NB >= kMmaMinBatch && !fragment_order(FMT, NB);
    int sms = 0, budget = 0;
    auto kernel = gemv_grouped_kernel<FMT, NB, false, PARTS>;
    int rc = prepare_kernel<gemv_grouped_kernel<FMT, NB, false, PARTS>>(&sms, &budget);
    if (pr.acc_debug) {
        kernel = gemv_grouped_kernel<FMT, NB, true, PARTS>;
        if (!rc) rc = prepare_kernel<gemv_grouped_kernel<FMT, NB, true, PARTS>>(&sms, &budget);
    }
    if (rc) return rc;
    Plan plw = pl;
    plw.stages = choose_stages(FMT, pl, pr.G, NB, pr.K, budget, kScr);
    const SmemLayout L = smem_layout(FMT, plw, pr.G, NB, pr.K, kScr);
    GroupedArgs gaw = ga;
    gaw.n_groups = n_groups;
    if (pl.CS == 1) {
        // rows in one piece: one balanced list of all groups' items; one or two tokens per group:
        // their activation rows travel with every stage
        const int64_t total = pl.items * n_groups;
        gaw.flat = 1;
        plw.cyclic = 0;
        plw.x_in_stage = NB < kMmaMinBatch ? 1 : 0;
        plw.stages = choose_stages(FMT, plw, pr.G, NB, pr.K, budget, kScr);
        const SmemLayout Lf = smem_layout(FMT, plw, pr.G, NB, pr.K, kScr);
        return launch_pdl(kernel, dim3(static_cast<unsigned>(total < sms ? total : sms)), (pl.NW + 2) * 32,
                          Lf.total, stream, pr, plw, gaw);
    }
    // the machine is shared by all groups: spread its multiprocessors over them
    int per_group = (sms + n_groups - 1) / n_groups;
    if (per_group < 1) per_group = 1;
    int gx = 1;
    choose_walk(plw, per_group, &gx);
    gaw.flat = 0;
    return launch_pdl(kernel, dim3(gx, n_groups), (pl.NW + 2) * 32, L.total, stream, pr, plw, gaw);
}

template <int NB>
int launch_phased(PhasedArgs &pa, int n_jobs, const int *job_phase, cudaStream_t stream) {
    for (int j = 0; j < n_jobs; ++j)
        if (static_cast<int64_t>(NB) * pa.pr[j].K > kXResidentBytes) return BITCOS_ERR_SHAPE;
    int sms = 0, budget = 0;
    int rc = prepare_kernel<gemv_phased_kernel<NB>>(&sms, &budget);
    if (rc) return rc;
    if (sms > kMaxGrid) sms = kMaxGrid;
    // the layout every job shares: the widest plan, the longest row
    Plan layout{};
    layout.tpw = 1;
    int64_t kmax = 0;
    int gmax = 0;
    for (int j = 0; j < n_jobs; ++j) {
        if (pa.pl[j].NW > layout.NW) layout.NW = pa.pl[j].NW;
        if (pa.pr[j].K > kmax) kmax = pa.pr[j].K;
        if (pa.pr[j].G > gmax) gmax = pa.pr[j].G;
    }
    layout.stages = choose_stages(kBitcos, layout, gmax, NB, kmax, budget, false);
    pa.layout = layout;
    pa.shape = Problem{};
    pa.shape.K = kmax;
    pa.shape.G = gmax;
    for (int p = 0; p < kMaxPhases; ++p) {
        pa.expect[p] = 0;
        for (int b = 0; b < kMaxGrid; ++b) pa.job_of[p][b] = 0xFF;
    }
    int grid = 1;
    for (int p = 0; p < pa.n_phases; ++p) {
        // the multiprocessors are shared between the phase's jobs in proportion to their item counts
        int64_t items[kMaxJobs], cap[kMaxJobs];
        int n = 0, next = 0;
        for (int j = 0; j < n_jobs; ++j)
            if (job_phase[j] == p) items[n++] = pa.pl[j].items;
        share_multiprocessors(items, n, sms, cap);
        for (int j = 0, i = 0; j < n_jobs; ++j) {
            if (job_phase[j] != p) continue;
            int blocks = 1;
            choose_walk(pa.pl[j], static_cast<int>(cap[i++]), &blocks);
            if (next + blocks > kMaxGrid) return BITCOS_ERR_SHAPE;
            pa.pl[j].NW = layout.NW;
            pa.pl[j].stages = layout.stages;
            pa.job_first_block[j] = next;
            pa.job_blocks[j] = blocks;
            for (int b = 0; b < blocks; ++b) {
                pa.job_of[p][next + b] = static_cast<uint8_t>(j);
                if (make_walk(pa.pl[j], b, blocks).count > 0) ++pa.expect[p];
            }
            next += blocks;
        }
        if (next > grid) grid = next;
    }
    const SmemLayout L = smem_layout(kBitcos, layout, gmax, NB, kmax, false);
    if (static_cast<int>(L.total) > budget) return BITCOS_ERR_SHAPE;
    return launch_pdl(gemv_phased_kernel<NB>, dim3(static_cast<unsigned>(grid)), (layout.NW + 2) * 32, L.total, stream, pa);
}
}  // namespace bitcos_kernels

#endif  // BITCOS_GEMV_CUH
