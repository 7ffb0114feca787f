// C entry points of the BITCOS library's device side (bitcos_gemv, trit5_gemv, bit2_gemv, bitcos_gemv_grouped, the
// launches of several products, the host-buffer forms, the activation quantiser, the routing and probe kernels).
// The products' kernels are in gemv.cuh; their instantiations are compiled part by part from gemv_inst.cu.
#include "gemv.cuh"
#include "gemv_inst.cuh"

#include <cuda.h>

namespace {

using namespace bitcos_kernels;

// ---------------------------------------------------------------------------------------------
// Decode-rate probe: what the paper's roofline calls gamma -- the cost of the unpack sequence when
// every operand is already on chip (Section III-B.1, Eq. 6).  Each warp decodes one synthetic tile
// that sits in shared memory, `iters` times, with the same code the GEMV kernels run (popcounts,
// prefix sum, sign windows, table lookups, dp4a); nothing is read from global memory inside the
// timed loop.  cycles[block] receives the block's elapsed clock cycles, sums (if not NULL) the accumulators of
// block 0's last pass, so that a test can hold them against the tile.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t probe_hash(uint32_t v) {
    v ^= v >> 16; v *= 0x7FEB352Du; v ^= v >> 15; v *= 0x846CA68Bu; v ^= v >> 16;
    return v;
}

template <int FMT>
__global__ void __launch_bounds__((kMaxWarps + 2) * 32, 1) decode_probe_kernel(int iters, unsigned long long *cycles, int32_t *sums) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    uint8_t *lut = smem;
    uint8_t *tiles = smem + (FMT == kBit2 ? 0 : kLutBytes);          // per warp: 1024 B payload + 640 B signs + 64 B scales
    uint8_t *xs = tiles + nw * 1792;                                   // 128 activations
    constexpr uint32_t kTile = 1792;
    if (FMT != kBit2) {
        const uint32_t *src = FMT == kBitcos ? g_bitcos_lut.v : g_trit5_lut.v;
        for (int i = threadIdx.x; i < kLutBytes / 4; i += blockDim.x) reinterpret_cast<uint32_t *>(lut)[i] = src[i];
    }
    // synthetic tile: presence bits set with probability 0.5625, random sign bits, valid five-trit bytes
    uint32_t *mine = reinterpret_cast<uint32_t *>(tiles + warp * kTile);
    for (int i = lane; i < kTile / 4; i += 32) {
        const uint32_t h1 = probe_hash(i * 4u + 1), h2 = probe_hash(i * 4u + 2), h3 = probe_hash(i * 4u + 3),
                       h4 = probe_hash(i * 4u + 4);
        uint32_t v = h1 | (h2 & h3 & h4);
        if (FMT == kTrit5) v = ((h1 & 0xFFu) % 243u) | (((h2 & 0xFFu) % 243u) << 8) | (((h3 & 0xFFu) % 243u) << 16) |
                               (((h4 & 0xFFu) % 243u) << 24);
        if (FMT == kBit2) v = (h1 | (h2 & h3 & h4)) & 0x55555555u;
        mine[i] = v;
    }
    for (int i = threadIdx.x; i < 32; i += blockDim.x) reinterpret_cast<uint32_t *>(xs)[i] = probe_hash(1000u + i);
    __syncthreads();
    const uint8_t *stage = tiles + warp * kTile;
    const uint32_t lane4 = static_cast<uint32_t>(lane) * 4u;
    int total = 0, last = 0;
    const long long t0 = clock64();
    for (int it = 0; it < iters; ++it) {
        int w[32];
        int a;
        if (FMT == kBitcos) {
            const uint4 bm = reinterpret_cast<const uint4 *>(stage)[lane];
            const int c = __popc(bm.x) + __popc(bm.y) + __popc(bm.z) + __popc(bm.w);
            int incl = c;
#pragma unroll
            for (int dd = 1; dd < 32; dd <<= 1) {
                const int v = __shfl_up_sync(0xFFFFFFFFu, incl, dd);
                if (lane >= dd) incl += v;
            }
            const uint32_t cursor = static_cast<uint32_t>(incl - c) + static_cast<uint32_t>(it & 1);
            const uint32_t *sp = reinterpret_cast<const uint32_t *>(stage + 1024) + (cursor >> 5);
            bitcos_decode_row_keyed(bm, sp, cursor & 31u, lut, lane4, w);
            asm volatile("" ::: "memory");
            a = contract<kBitcos>(w, reinterpret_cast<const int4 *>(xs), lane);
        } else if (FMT == kTrit5) {
            const uint32_t *src = reinterpret_cast<const uint32_t *>(stage) + lane;
            uint32_t wd[7];
#pragma unroll
            for (int i = 0; i < 7; ++i) wd[i] = src[i * kRows];
            trit5_decode_row(wd, it & 1, lut, static_cast<uint32_t>(lane) * 8u, w);
            a = contract<kTrit5>(w, reinterpret_cast<const int4 *>(xs), lane);
        } else {
            const uint4 *src = reinterpret_cast<const uint4 *>(stage) + lane + (it & 1);   // keep the loads in the loop
            bit2_decode_row(src[0], src[kRows], w);
            a = contract<kBit2>(w, reinterpret_cast<const int4 *>(xs), lane);
        }
        const float sc = bf16_to_float(reinterpret_cast<const uint16_t *>(stage + 1024 + 640)[lane]);
        total += __float_as_int(sc * static_cast<float>(a));
        last = a;
    }
    const long long t1 = clock64();
    __shared__ unsigned long long s_max;
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    if (lane == 0) atomicMax(&s_max, static_cast<unsigned long long>(t1 - t0));
    __syncthreads();
    if (threadIdx.x == 0) cycles[blockIdx.x] = s_max;
    if (sums && blockIdx.x == 0) sums[warp * 32 + lane] = last;
    if (total == 0x12345678) cycles[blockIdx.x] = 0;      // keeps the sum alive; never true in practice
}

// ---------------------------------------------------------------------------------------------
// Give-up path of the bounded waits, exercised without a fault: one warp arms an mbarrier for bytes
// that no copy ever delivers and waits for it with the kernels' own polling loop and a short limit.
// The wait runs out, the warp sets the workspace's status word exactly as the products do, and the
// kernel returns normally; the context stays usable.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(32, 1) wait_probe_kernel(unsigned int *status, unsigned long long limit_ns, unsigned long long *waited_ns) {
    __shared__ __align__(8) unsigned long long bar_word;
    const uint32_t bar = smem_addr(&bar_word);
    const int lane = threadIdx.x & 31;
    if (lane == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(bar, 64);                  // 64 bytes are announced; nothing is ever copied
    }
    __syncwarp();
    const uint64_t t0 = global_timer_ns();
    const bool ok = mbar_wait_limited(bar, 0, limit_ns);
    const uint64_t t1 = global_timer_ns();
    if (!ok && lane == 0) {
        *status = 1u;
        if (waited_ns) *waited_ns = t1 - t0;
    }
}

// ---------------------------------------------------------------------------------------------
// Routing pairs grouped by expert on the device (a stable counting sort in one thread block), so
// that a decode loop whose router runs on the GPU never has to bring the pairs to the host: count
// the pairs of every expert, give every expert that has any a group (experts ascending), place
// every pair behind the pairs of the same expert that precede it in the input.  A pair whose expert
// id is out of range is dropped: it gets no group.  What the groups leave of the output lists is
// filled (0, order -1), so that the caller need not.
// Latency is all there is to it (a few KB), so every step is one round of the block: the experts are
// scanned by all threads, four to a thread at most, and one warp finds the stable places 32 pairs at a
// time (match_any: the earlier lanes with the same expert), without reading global memory.
// 64 pairs, 128 experts: 8.6 -> 2.2 us against one thread that walks the experts, every pair counting the pairs
// before it, and the caller's five fill kernels.
// ---------------------------------------------------------------------------------------------
constexpr int kGroupPairsThreads = 256;
constexpr int kExpertsPerThread = BITCOS_GROUP_EXPERTS_MAX / kGroupPairsThreads;
__global__ void __launch_bounds__(kGroupPairsThreads) group_pairs_kernel(const int32_t *__restrict__ pair_expert,
                                                                         const int32_t *__restrict__ pair_xrow, int n_pairs, int n_experts,
                                                                         int32_t *__restrict__ group_expert, int32_t *__restrict__ group_begin,
                                                                         int32_t *__restrict__ pair_xrow_sorted, int32_t *__restrict__ order,
                                                                         int32_t *__restrict__ n_groups) {
    __shared__ int count[BITCOS_GROUP_EXPERTS_MAX];      // pairs per expert, then the expert's next free position
    __shared__ int16_t place[BITCOS_GROUP_PAIRS_MAX];    // a pair's expert (-1: out of range), then its position
    __shared__ uint32_t warp_sum[kGroupPairsThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int e = tid; e < BITCOS_GROUP_EXPERTS_MAX; e += kGroupPairsThreads) count[e] = 0;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    for (int i = tid; i < n_pairs; i += kGroupPairsThreads) {
        const int e = __ldg(pair_expert + i);
        const bool in = e >= 0 && e < n_experts;
        place[i] = static_cast<int16_t>(in ? e : -1);
        if (in) atomicAdd(&count[e], 1);
    }
    __syncthreads();
    // pairs (low half: at most 4096) and groups (high half: at most 1024) in front of every expert
    int c[kExpertsPerThread];
    uint32_t mine = 0;
#pragma unroll
    for (int j = 0; j < kExpertsPerThread; ++j) {
        c[j] = count[tid * kExpertsPerThread + j];
        mine += static_cast<uint32_t>(c[j]) + (c[j] ? 0x10000u : 0u);
    }
    const uint32_t upto = warp_scan_add(mine);
    if (lane == 31) warp_sum[warp] = upto;
    __syncthreads();
    uint32_t before = upto - mine, total = 0;
#pragma unroll
    for (int w = 0; w < kGroupPairsThreads / 32; ++w) {
        if (w < warp) before += warp_sum[w];
        total += warp_sum[w];
    }
#pragma unroll
    for (int j = 0; j < kExpertsPerThread; ++j) {
        const int pos = static_cast<int>(before & 0xFFFFu), g = static_cast<int>(before >> 16);
        count[tid * kExpertsPerThread + j] = pos;
        if (c[j]) {
            group_expert[g] = tid * kExpertsPerThread + j;
            group_begin[g] = pos;
        }
        before += static_cast<uint32_t>(c[j]) + (c[j] ? 0x10000u : 0u);
    }
    const int kept = static_cast<int>(total & 0xFFFFu), groups = static_cast<int>(total >> 16);
    const int cap = n_pairs < n_experts ? n_pairs : n_experts;
    for (int g = groups + tid; g <= cap; g += kGroupPairsThreads) {
        group_begin[g] = g == groups ? kept : 0;
        if (g < cap) group_expert[g] = 0;
    }
    for (int i = kept + tid; i < n_pairs; i += kGroupPairsThreads) {
        pair_xrow_sorted[i] = 0;
        order[i] = -1;
    }
    if (tid == 0) *n_groups = groups;
    __syncthreads();
    if (warp == 0) {
        for (int base = 0; base < n_pairs; base += 32) {
            const int i = base + lane;
            const int e = i < n_pairs ? place[i] : -1;
            const uint32_t same = __match_any_sync(0xFFFFFFFFu, e);
            const int at = e >= 0 ? count[e] + __popc(same & ((1u << lane) - 1u)) : -1;      // input order inside a group
            __syncwarp();
            if (e >= 0 && lane == __ffs(same) - 1) count[e] += __popc(same);
            if (i < n_pairs) place[i] = static_cast<int16_t>(at);
            __syncwarp();
        }
    }
    __syncthreads();
    for (int i = tid; i < n_pairs; i += kGroupPairsThreads) {
        const int at = place[i];
        if (at < 0) continue;
        pair_xrow_sorted[at] = __ldg(pair_xrow + i);
        order[at] = i;
    }
}

// Validates the arguments every product shares; fills nothing.
int check_common(int fmt, const uint32_t *payload, const uint32_t *signs, const uint32_t *tile_off,
                 const uint16_t *scales, int64_t M, int64_t K, const int8_t *x, const float *x_scale, int batch,
                 const float *y, const int32_t *acc_debug, const void *workspace, size_t workspace_bytes) {
    if (!payload || !scales || !x || !x_scale || !y || !workspace) return BITCOS_ERR_NULL;
    if (fmt == kBitcos && (!signs || !tile_off)) return BITCOS_ERR_NULL;
    if (M < 1 || K < kGroup || K % kGroup != 0 || batch < 1 || batch > BITCOS_MAX_BATCH) return BITCOS_ERR_SHAPE;
    if (K / kGroup > 0x7FFFFF || make_plan(M, K, kWarps16).items > 0x3FFFFFFF) return BITCOS_ERR_SHAPE;
    if (!aligned16(payload) || !aligned16(scales) || !aligned16(x) || !aligned16(y) || !aligned16(workspace) ||
        (signs && !aligned16(signs)) || (tile_off && !aligned16(tile_off)) || (acc_debug && !aligned16(acc_debug)))
        return BITCOS_ERR_ALIGN;
    if (workspace_bytes < workspace_bytes_for(M, K)) return BITCOS_ERR_CAPACITY;
    return BITCOS_OK;
}

void fill_problem(Problem &pr, const uint32_t *payload, const uint32_t *signs, const uint32_t *tile_off,
                  const uint16_t *scales, int64_t M, int64_t K, const int8_t *x, const float *x_scale, int batch,
                  float *y, int32_t *acc_debug, void *workspace) {
    pr.payload = payload;
    pr.signs = signs;
    pr.tile_off = tile_off;
    pr.scales = scales;
    pr.x = x;
    pr.x_scale = x_scale;
    pr.xrow = nullptr;
    pr.y = y;
    pr.acc_debug = acc_debug;
    pr.M = M;
    pr.K = K;
    pr.G = static_cast<int>(K / kGroup);
    pr.RB = static_cast<int>(padded_rows(M) / kRows);
    pr.nb = batch;
    pr.out_row0 = 0;
    uint8_t *ws = static_cast<uint8_t *>(workspace);
    pr.status = reinterpret_cast<unsigned int *>(ws);
    pr.counters = reinterpret_cast<unsigned int *>(ws + kHeaderBytes);
    pr.partial = reinterpret_cast<float *>(ws + kHeaderBytes + counters_bytes(pr.RB));
}

int gemv_common(int fmt, const uint32_t *payload, const uint32_t *signs, const uint32_t *tile_off,
                const uint16_t *scales, int64_t M, int64_t K, const int8_t *x, const float *x_scale, int batch,
                float *y, int32_t *acc_debug, void *workspace, size_t workspace_bytes, void *cuda_stream,
                const uint32_t *off_host = nullptr, bool group_scales = false) {
    const int bad = check_common(fmt, payload, signs, tile_off, scales, M, K, x, x_scale, batch, y, acc_debug, workspace,
                                 workspace_bytes);
    if (bad) return bad;
    const Plan pl = one_tile_plan(fmt, M, K, nb_bucket(batch, K));
    Problem pr{};
    fill_problem(pr, payload, signs, tile_off, scales, M, K, x, x_scale, batch, y, acc_debug, workspace);
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (group_scales) return fmt == kBitcos ? launch_nb<kBitcos, true>(pr, pl, stream, off_host) : BITCOS_ERR_SHAPE;
    if (fmt == kBitcos) return launch_nb<kBitcos>(pr, pl, stream, off_host);
    if (fmt == kTrit5) return launch_nb<kTrit5>(pr, pl, stream, nullptr);
    return launch_nb<kBit2>(pr, pl, stream, nullptr);
}


// ------------------------------------------------------------------ activation quantiser
// bf16 activations -> int8 codes and float scales, one scale per group of 128 or per token:
//   a = max(max |x| over the group, 2^-100),  scale = a / 127,  code = rint(x * (127 / a))
// with IEEE float32 quotient and product and ties to even (the explicit intrinsics keep the
// compiler from contracting or approximating them, so the codes do not depend on build flags).
// One warp per group of 128: a lane holds four consecutive values.
__global__ void __launch_bounds__(256) quantize_groups_kernel(const uint16_t *__restrict__ x, int8_t *__restrict__ q,
                                                              float *__restrict__ scale, int64_t n_groups) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    for (int64_t grp = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); grp < n_groups; grp += warps) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(x + grp * kGroup) + lane);
        float a = fmaxf(fmaxf(fabsf(bf16_lo(v.x)), fabsf(bf16_hi(v.x))), fmaxf(fabsf(bf16_lo(v.y)), fabsf(bf16_hi(v.y))));
#pragma unroll
        for (int d = 16; d; d >>= 1) a = fmaxf(a, __shfl_xor_sync(0xFFFFFFFFu, a, d));
        a = fmaxf(a, kAmaxFloor);
        const float inv = __fdiv_rn(127.0f, a);
        reinterpret_cast<uint32_t *>(q + grp * kGroup)[lane] = quant_pair(v.x, inv) | (quant_pair(v.y, inv) << 16);
        if (lane == 0) scale[grp] = __fdiv_rn(a, 127.0f);
    }
}

// One thread block per token: largest magnitude of the row, then the codes (the row is read
// twice, the second time from cache).
constexpr int kQuantThreads = 512;
__global__ void __launch_bounds__(kQuantThreads) quantize_tokens_kernel(const uint16_t *__restrict__ x, int8_t *__restrict__ q,
                                                                        float *__restrict__ scale, int64_t K) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __shared__ float warp_max[kQuantThreads / 32];
    const int64_t row = blockIdx.x;
    const uint4 *src = reinterpret_cast<const uint4 *>(x + row * K);      // eight values per load
    const int64_t n = K / 8;
    float a = 0.f;
    for (int64_t i = threadIdx.x; i < n; i += kQuantThreads) {
        const uint4 v = __ldg(src + i);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) a = fmaxf(a, fmaxf(fabsf(bf16_lo(w[j])), fabsf(bf16_hi(w[j]))));
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) a = fmaxf(a, __shfl_xor_sync(0xFFFFFFFFu, a, d));
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = a;
    __syncthreads();
    a = warp_max[0];
#pragma unroll
    for (int j = 1; j < kQuantThreads / 32; ++j) a = fmaxf(a, warp_max[j]);
    a = fmaxf(a, kAmaxFloor);
    const float inv = __fdiv_rn(127.0f, a);
    uint2 *dst = reinterpret_cast<uint2 *>(q + row * K);
    for (int64_t i = threadIdx.x; i < n; i += kQuantThreads) {
        const uint4 v = __ldg(src + i);
        dst[i] = make_uint2(quant_pair(v.x, inv) | (quant_pair(v.y, inv) << 16),
                            quant_pair(v.z, inv) | (quant_pair(v.w, inv) << 16));
    }
    if (threadIdx.x == 0) scale[row] = __fdiv_rn(a, 127.0f);
}

}  // namespace

namespace bitcos_detail {
// for the library's other translation units: the error bitcos_last_cuda_error reports
void record_cuda_error(int e) { bitcos_kernels::g_last_cuda_error = e; }

// Where a kernel finds the host memory [p, p + bytes): its device address if all of it lies in one pinned allocation (or
// one registered range) that is mapped into the device, else NULL.  Asked before every launch that is going to touch host
// memory, because a range that was mapped at an earlier call may have been unregistered or freed since
// (0.2 us a call: one driver call without a lock on the stream).
void *mapped_host(const void *p, size_t bytes) {
    typedef CUresult (*Attributes)(unsigned int, CUpointer_attribute *, void **, CUdeviceptr);
    static const Attributes attributes = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 7000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<Attributes>(f);
    }();
    if (!attributes) return nullptr;
    CUpointer_attribute ask[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                 CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    unsigned int type = 0, managed = 0;
    CUdeviceptr at = 0, start = 0;
    size_t size = 0;
    void *answers[] = {&type, &managed, &at, &start, &size};
    if (attributes(5, ask, answers, reinterpret_cast<CUdeviceptr>(p)) != CUDA_SUCCESS || type != CU_MEMORYTYPE_HOST || (managed & 0xFFu) || !at)
        return nullptr;
    // (the range is given at the address asked for, host and device addresses being the same ones, or at the mapped one)
    const CUdeviceptr host = reinterpret_cast<CUdeviceptr>(p);
    const CUdeviceptr in = host >= start && host - start < size ? host : at;
    if (in < start || in - start > size || bytes > size - (in - start)) return nullptr;
    return reinterpret_cast<void *>(at);
}
}  // namespace bitcos_detail

extern "C" {

int bitcos_last_cuda_error(void) { return g_last_cuda_error; }

size_t bitcos_gemv_workspace_bytes(int64_t M, int64_t K) {
    if (M < 1 || K < kGroup || K % kGroup != 0) return 0;
    return workspace_bytes_for(M, K);
}

int bitcos_workspace_init(void *workspace, size_t workspace_bytes, void *cuda_stream) {
    if (!workspace) return BITCOS_ERR_NULL;
    return check_cuda(cudaMemsetAsync(workspace, 0, workspace_bytes, static_cast<cudaStream_t>(cuda_stream)));
}

int bitcos_workspace_status(const void *workspace, void *cuda_stream, int *status) {
    if (!workspace || !status) return BITCOS_ERR_NULL;
    unsigned int v = 0;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    int rc = check_cuda(cudaMemcpyAsync(&v, workspace, sizeof v, cudaMemcpyDeviceToHost, stream));
    if (rc) return rc;
    rc = check_cuda(cudaStreamSynchronize(stream));
    if (rc) return rc;
    *status = static_cast<int>(v);
    return BITCOS_OK;
}

int bitcos_decode_probe_sums(int format, int warps_per_block, int iters, int blocks, uint64_t *cycles, int32_t *sums, void *cuda_stream) {
    if (!cycles) return BITCOS_ERR_NULL;
    if (format < 0 || format > 2 || warps_per_block < 1 || warps_per_block > kMaxWarps + 2 || iters < 1 ||
        iters > (1 << 20) || blocks < 1 || blocks > 4096)
        return BITCOS_ERR_SHAPE;
    const size_t smem = (format == kBit2 ? 0 : kLutBytes) + static_cast<size_t>(warps_per_block) * 1792 + 256;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    unsigned long long *out = reinterpret_cast<unsigned long long *>(cycles);
    auto launch = [&](auto *kernel) {
        const int rc = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
        if (rc) return rc;
        kernel<<<blocks, warps_per_block * 32, smem, stream>>>(iters, out, sums);
        return check_cuda(cudaGetLastError());
    };
    if (format == kBitcos) return launch(decode_probe_kernel<kBitcos>);
    if (format == kTrit5) return launch(decode_probe_kernel<kTrit5>);
    return launch(decode_probe_kernel<kBit2>);
}

int bitcos_decode_probe(int format, int warps_per_block, int iters, int blocks, uint64_t *cycles, void *cuda_stream) {
    return bitcos_decode_probe_sums(format, warps_per_block, iters, blocks, cycles, nullptr, cuda_stream);
}

int bitcos_gemv(const bitcos_weights *W, const int8_t *x, const float *x_scale, int batch, float *y,
                int32_t *acc_debug, void *workspace, size_t workspace_bytes, void *cuda_stream) {
    if (!W) return BITCOS_ERR_NULL;
    return gemv_common(kBitcos, W->bitmap, W->signs, W->tile_off, W->scales, W->M, W->K, x, x_scale, batch, y,
                       acc_debug, workspace, workspace_bytes, cuda_stream, W->tile_off_host);
}

// ---------------------------------------------------------------------------------------------
// bitcos_gemv_static: the same product with the scratch memory taken from a fixed array that is
// part of the library image, for callers that must not (or cannot) allocate device memory.
// ---------------------------------------------------------------------------------------------
}  // extern "C"

namespace {
// Scratch of the no-allocation entry point.  Every device that loads the library carries these
// bytes until the process exits.  In host code the name below is only a handle for
// cudaGetSymbolAddress; it is not a device address and is never passed to a kernel.
static __device__ __align__(256) unsigned char g_static_workspace[BITCOS_STATIC_WORKSPACE_BYTES];

// Device address of g_static_workspace on the current device, looked up once per device.  (The cache is
// written without a lock: two threads that race on a device's first call both store the same address.)
int static_workspace_ptr(void **out) {
    constexpr int kMaxDev = 32;
    static void *cache[kMaxDev];
    int dev = 0;
    int rc = check_cuda(cudaGetDevice(&dev));
    if (rc) return rc;
    if (dev < kMaxDev && cache[dev]) {
        *out = cache[dev];
        return BITCOS_OK;
    }
    void *ptr = nullptr;
    rc = check_cuda(cudaGetSymbolAddress(&ptr, g_static_workspace));
    if (rc) return rc;
    if (!ptr) return BITCOS_ERR_CUDA;
    if (dev < kMaxDev) cache[dev] = ptr;
    *out = ptr;
    return BITCOS_OK;
}
}  // namespace

extern "C" {

int bitcos_gemv_static(const bitcos_weights *W, const int8_t *x, const float *x_scale, int batch, float *y,
                       void *cuda_stream) {
    if (!W) return BITCOS_ERR_NULL;
    if (W->M < 1 || W->K < kGroup || W->K % kGroup != 0) return BITCOS_ERR_SHAPE;
    const size_t need = workspace_bytes_for(W->M, W->K);
    if (need > static_cast<size_t>(BITCOS_STATIC_WORKSPACE_BYTES)) return BITCOS_ERR_CAPACITY;
    void *ws = nullptr;
    int rc = static_workspace_ptr(&ws);
    if (rc) return rc;
    // (nothing is enqueued for a call that is going to be refused)
    rc = check_common(kBitcos, W->bitmap, W->signs, W->tile_off, W->scales, W->M, W->K, x, x_scale, batch, y, nullptr, ws,
                      BITCOS_STATIC_WORKSPACE_BYTES);
    if (rc) return rc;
    // The array keeps whatever the last call left.  The status word and the arrival counters must
    // start at zero, so they are cleared on the caller's stream ahead of the kernel (the partial
    // sums behind them are always written before they are read).
    const size_t head = kHeaderBytes + counters_bytes(padded_rows(W->M) / kRows);
    rc = check_cuda(cudaMemsetAsync(ws, 0, head, static_cast<cudaStream_t>(cuda_stream)));
    if (rc) return rc;
    return gemv_common(kBitcos, W->bitmap, W->signs, W->tile_off, W->scales, W->M, W->K, x, x_scale, batch, y,
                       nullptr, ws, BITCOS_STATIC_WORKSPACE_BYTES, cuda_stream, W->tile_off_host);
}

int bitcos_gemv_static_status(void *cuda_stream, int *status) {
    if (!status) return BITCOS_ERR_NULL;
    void *ws = nullptr;
    const int rc = static_workspace_ptr(&ws);
    if (rc) return rc;
    return bitcos_workspace_status(ws, cuda_stream, status);
}

int bitcos_wait_probe(void *workspace, uint64_t limit_ns, uint64_t *waited_ns, void *cuda_stream) {
    if (!workspace) return BITCOS_ERR_NULL;
    if (limit_ns < 1000 || limit_ns > 100ull * 1000 * 1000) return BITCOS_ERR_SHAPE;      // 1 us .. 100 ms
    wait_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>(static_cast<unsigned int *>(workspace), limit_ns,
                                                                        reinterpret_cast<unsigned long long *>(waited_ns));
    return check_cuda(cudaGetLastError());
}

int bitcos_quantize_activations(const uint16_t *x_bf16, int batch, int64_t K, int group, int8_t *xq, float *x_scale,
                                void *cuda_stream) {
    if (!x_bf16 || !xq || !x_scale) return BITCOS_ERR_NULL;
    if (batch < 1 || batch > BITCOS_MAX_BATCH || K < kGroup || K % kGroup != 0) return BITCOS_ERR_SHAPE;
    if (group != 0 && group != kGroup) return BITCOS_ERR_SHAPE;
    if (!aligned16(x_bf16) || !aligned16(xq)) return BITCOS_ERR_ALIGN;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (group == 0)
        return launch_pdl(quantize_tokens_kernel, dim3(static_cast<unsigned>(batch)), kQuantThreads, 0, stream, x_bf16, xq,
                          x_scale, K);
    const int64_t n_groups = static_cast<int64_t>(batch) * (K / kGroup);
    const int64_t blocks = (n_groups + 7) / 8;
    return launch_pdl(quantize_groups_kernel, dim3(static_cast<unsigned>(blocks)), 256, 0, stream, x_bf16, xq, x_scale,
                      n_groups);
}

int bitcos_gemv_group_scales(const bitcos_weights *W, const int8_t *x, const float *x_group_scale, int batch, float *y,
                             int32_t *acc_debug, void *workspace, size_t workspace_bytes, void *cuda_stream) {
    if (!W) return BITCOS_ERR_NULL;
    return gemv_common(kBitcos, W->bitmap, W->signs, W->tile_off, W->scales, W->M, W->K, x, x_group_scale, batch, y,
                       acc_debug, workspace, workspace_bytes, cuda_stream, W->tile_off_host, true);
}

}  // extern "C"

namespace {
// bf16 = true: every job's x holds 16-bit activations (x_scale is not used) and the decoder warps
// quantise them per group of 128; one or two tokens.
#ifdef BITCOS_TIMELINE
unsigned long long *g_tl_buf = nullptr;
int g_tl_slots = 0, g_tl_next = 0;
#endif

int gemv_multi_common(const bitcos_gemv_job *jobs, int n_jobs, int batch, void *cuda_stream, bool bf16,
                      bool group_scales = false, const bitcos_weights *const *next = nullptr, int n_next = 0,
                      const bitcos_weights *const *prev = nullptr, int n_prev = 0) {
    if (!jobs) return BITCOS_ERR_NULL;
    if (n_jobs < 1 || n_jobs > kMaxJobs) return BITCOS_ERR_SHAPE;
    if (bf16 && batch > 2) return BITCOS_ERR_SHAPE;
    if (n_next < 0 || n_next * 4 > kMaxPrefetch || (n_next > 0 && !next)) return BITCOS_ERR_SHAPE;
    if (n_prev < 0 || n_prev > kMaxJobs || (n_prev > 0 && !prev)) return BITCOS_ERR_SHAPE;
    // thread blocks of the launch the caller says runs directly before this one (same batch)
    int busy = 0;
    if (n_prev > 0) {
        MultiArgs pm{};
        pm.n = n_prev;
        int64_t kprev = 0;
        for (int i = 0; i < n_prev; ++i) {
            const bitcos_weights *w = prev[i];
            if (!w) return BITCOS_ERR_NULL;
            if (w->M < 1 || w->K < kGroup || w->K % kGroup) return BITCOS_ERR_SHAPE;
            pm.pr[i].M = w->M;
            pm.pr[i].K = w->K;
            kprev = w->K > kprev ? w->K : kprev;
        }
        int dev = 0, sms = 0;
        int rc = check_cuda(cudaGetDevice(&dev));
        if (!rc) rc = check_cuda(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        if (rc) return rc;
        bool two = false;
        int grids[kMaxJobs];
        busy = plan_multi(pm, nb_bucket(batch, kprev), sms, &two, grids);
    }
    MultiArgs ma{};
    ma.n = n_jobs;
#ifdef BITCOS_TIMELINE
    if (g_tl_buf) ma.pf.tl = g_tl_buf + static_cast<size_t>(g_tl_next++ % g_tl_slots) * kMaxGrid * 32;
#endif
    for (int i = 0; i < n_next; ++i) {
        const bitcos_weights *w = next[i];
        if (!w || !w->bitmap || !w->signs || !w->tile_off || !w->scales) return BITCOS_ERR_NULL;
        if (w->M < 1 || w->K < kGroup || w->K % kGroup) return BITCOS_ERR_SHAPE;
        const uint64_t tiles = static_cast<uint64_t>(padded_rows(w->M) / kRows) * static_cast<uint64_t>(w->K / kGroup);
        auto add = [&](const void *p, uint64_t bytes) {
            bytes &= ~static_cast<uint64_t>(15);
            if (bytes > 0xFFFFFFF0ull) bytes = 0xFFFFFFF0ull;
            if (!bytes || (reinterpret_cast<uintptr_t>(p) & 15)) return;
            ma.pf.ptr[ma.pf.n] = static_cast<const uint8_t *>(p);
            ma.pf.bytes[ma.pf.n++] = static_cast<uint32_t>(bytes);
        };
        add(w->bitmap, tiles * 512);
        add(w->scales, tiles * kRows * sizeof(uint16_t));
        add(w->tile_off, (tiles + 1) * sizeof(uint32_t));
        // the length of the sign vector is only known from the host copy of the entry offsets
        if (w->tile_off_host)
            add(w->signs, (static_cast<uint64_t>(host_offset(w->tile_off_host, static_cast<int64_t>(tiles))) + 31) / 32 * 4);
    }
    // The request pays when the launches are short and the later one starts from L2 instead of device
    // memory (a 2B model's layer: requests of 3.8 and 7.6 MB, 0.45 us of 16 gained); asking for more
    // only competes with the launch's own stream (a 32B model's layer, requests of 9 to 54 MB: 1-3 %
    // slower), so a large request is dropped whole.
    {
        uint64_t requested = 0;
        for (int i = 0; i < ma.pf.n; ++i) requested += ma.pf.bytes[i];
        if (requested > BITCOS_PREFETCH_MAX_BYTES) ma.pf.n = 0;
    }
    for (int j = 0; j < n_jobs; ++j) {
        bitcos_gemv_job jb = jobs[j];
        if (!jb.W) return BITCOS_ERR_NULL;
        if (bf16) jb.x_scale = reinterpret_cast<const float *>(jb.x);        // never read; passes the NULL check
        const int bad = check_common(kBitcos, jb.W->bitmap, jb.W->signs, jb.W->tile_off, jb.W->scales, jb.W->M, jb.W->K,
                                     jb.x, jb.x_scale, batch, jb.y, nullptr, jb.workspace, jb.workspace_bytes);
        if (bad) return bad;
        for (int i = 0; i < j; ++i)
            if (jobs[i].workspace == jb.workspace) return BITCOS_ERR_SHAPE;      // jobs run concurrently
        fill_problem(ma.pr[j], jb.W->bitmap, jb.W->signs, jb.W->tile_off, jb.W->scales, jb.W->M, jb.W->K, jb.x,
                     jb.x_scale, batch, jb.y, nullptr, jb.workspace);
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    int64_t kmax = 0;
    for (int j = 0; j < n_jobs; ++j) kmax = jobs[j].W->K > kmax ? jobs[j].W->K : kmax;
    const int nbk = nb_bucket(batch, kmax);
    const uint32_t *off_host[kMaxJobs];
    for (int j = 0; j < n_jobs; ++j) off_host[j] = jobs[j].W->tile_off_host;
    if (bf16) {
        if (nbk == 1) return launch_multi<1, true>(ma, stream, off_host);
        if (nbk == 2) return launch_multi<2, true>(ma, stream, off_host);
        return BITCOS_ERR_SHAPE;          // rows too long for the one- and two-token kernels
    }
    if (group_scales) {
        if (nbk == 1) return launch_multi<1, false, true>(ma, stream, off_host);
        if (nbk == 2) return launch_multi<2, false, true>(ma, stream, off_host);
        if (batch <= 4) return launch_multi<4, false, true>(ma, stream, off_host);
        if (batch <= 8) return launch_multi<8, false, true>(ma, stream, off_host);
        return launch_multi<16, false, true>(ma, stream, off_host);
    }
    if (nbk == 1) return launch_multi<1>(ma, stream, off_host, busy);
    if (nbk == 2) return launch_multi<2>(ma, stream, off_host, busy);
    if (batch <= 4) return launch_multi<4>(ma, stream, off_host, busy);
    if (batch <= 8) return launch_multi<8>(ma, stream, off_host, busy);
    return launch_multi<16>(ma, stream, off_host, busy);
}
}  // namespace

extern "C" {

int bitcos_gemv_phased(const bitcos_gemv_job *jobs, const int *job_phase, int n_jobs, int batch, void *sync,
                       void *cuda_stream) {
    if (!jobs || !job_phase || !sync) return BITCOS_ERR_NULL;
    if (n_jobs < 1 || n_jobs > kMaxJobs || batch < 1 || batch > 2) return BITCOS_ERR_SHAPE;
    if (!aligned16(sync)) return BITCOS_ERR_ALIGN;
    if (job_phase[0] != 0) return BITCOS_ERR_SHAPE;
    for (int j = 1; j < n_jobs; ++j)
        if (job_phase[j] < job_phase[j - 1] || job_phase[j] > job_phase[j - 1] + 1) return BITCOS_ERR_SHAPE;
    if (job_phase[n_jobs - 1] >= kMaxPhases) return BITCOS_ERR_SHAPE;
    static PhasedArgs pa_storage;      // (large: kept off the stack; calls are serialised by the lock below)
    static std::mutex lock;
    std::lock_guard<std::mutex> guard(lock);
    PhasedArgs &pa = pa_storage;
    pa.n_phases = job_phase[n_jobs - 1] + 1;
    pa.sync = static_cast<unsigned int *>(sync);
#ifdef BITCOS_TIMELINE
    pa.tl = g_tl_buf ? g_tl_buf + static_cast<size_t>(g_tl_next++ % g_tl_slots) * kMaxGrid * 32 : nullptr;
#endif
    for (int j = 0; j < n_jobs; ++j) {
        const bitcos_gemv_job &jb = jobs[j];
        if (!jb.W) return BITCOS_ERR_NULL;
        const int bad = check_common(kBitcos, jb.W->bitmap, jb.W->signs, jb.W->tile_off, jb.W->scales, jb.W->M, jb.W->K,
                                     jb.x, jb.x_scale, batch, jb.y, nullptr, jb.workspace, jb.workspace_bytes);
        if (bad) return bad;
        for (int i = 0; i < j; ++i)
            if (jobs[i].workspace == jb.workspace) return BITCOS_ERR_SHAPE;
        pa.pl[j] = one_tile_plan(kBitcos, jb.W->M, jb.W->K, batch);
        fill_problem(pa.pr[j], jb.W->bitmap, jb.W->signs, jb.W->tile_off, jb.W->scales, jb.W->M, jb.W->K, jb.x,
                     jb.x_scale, batch, jb.y, nullptr, jb.workspace);
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (batch == 1) return launch_phased<1>(pa, n_jobs, job_phase, stream);
    return launch_phased<2>(pa, n_jobs, job_phase, stream);
}

#ifdef BITCOS_TIMELINE
// Debug build only: device buffer of slots x 160 blocks x 16 stamps; every multi launch takes the next slot.
__attribute__((visibility("default"))) void bitcos_debug_timeline(unsigned long long *buf, int slots) {
    g_tl_buf = buf;
    g_tl_slots = slots;
    g_tl_next = 0;
}
#endif

int bitcos_gemv_multi_plan(const int64_t *M, const int64_t *K, int n_jobs, int batch, int multiprocessors,
                           int busy_multiprocessors, int capacity, int *block_job, int *block_first_item, int *block_items,
                           int *job_items, int *job_tiles_per_item, int *job_column_blocks, int *job_chunk_stride,
                           int *n_blocks) {
    if (!M || !K || !block_job || !block_first_item || !block_items || !job_items || !job_tiles_per_item ||
        !job_column_blocks || !job_chunk_stride || !n_blocks)
        return BITCOS_ERR_NULL;
    if (n_jobs < 1 || n_jobs > kMaxJobs || batch < 1 || batch > BITCOS_MAX_BATCH || multiprocessors < 1 ||
        multiprocessors > kMaxGrid || busy_multiprocessors < 0)
        return BITCOS_ERR_SHAPE;
    static thread_local MultiArgs ma;
    ma = MultiArgs{};
    ma.n = n_jobs;
    int64_t kmax = 0;
    for (int j = 0; j < n_jobs; ++j) {
        if (M[j] < 1 || K[j] < kGroup || K[j] % kGroup) return BITCOS_ERR_SHAPE;
        ma.pr[j].M = M[j];
        ma.pr[j].K = K[j];
        ma.pr[j].G = static_cast<int>(K[j] / kGroup);
        ma.pr[j].RB = static_cast<int>(padded_rows(M[j]) / kRows);
        kmax = K[j] > kmax ? K[j] : kmax;
    }
    bool two = false;
    int grids[kMaxJobs];
    const int total = plan_multi(ma, nb_bucket(batch, kmax), multiprocessors, &two, grids);
    if (total > capacity) return BITCOS_ERR_CAPACITY;
    static thread_local int first[kMaxGrid], count[kMaxGrid];
    if (skewed_assignment(ma, grids, total, two, multiprocessors, busy_multiprocessors, first, count)) {
        for (int b = 0; b < total; ++b) {
            block_job[b] = ma.job_of[b];
            block_first_item[b] = first[b];
            block_items[b] = count[b];
        }
    } else {
        int b = 0;
        for (int j = 0; j < n_jobs; ++j)
            for (int r = 0; r < grids[j]; ++r, ++b) {
                const Walk w = make_walk(ma.pl[j], r, grids[j]);
                block_job[b] = j;
                block_first_item[b] = w.first;
                block_items[b] = w.count;
            }
    }
    for (int j = 0; j < n_jobs; ++j) {
        job_items[j] = static_cast<int>(ma.pl[j].items);
        job_tiles_per_item[j] = ma.pl[j].NW * ma.pl[j].tpw;
        job_column_blocks[j] = ma.pl[j].CS;
        job_chunk_stride[j] = ma.pl[j].cyclic ? grids[j] : 1;
    }
    *n_blocks = total;
    return BITCOS_OK;
}

int bitcos_gemv_multi_chained(const bitcos_gemv_job *jobs, int n_jobs, int batch, const bitcos_weights *const *prev,
                              int n_prev, const bitcos_weights *const *next, int n_next, void *cuda_stream) {
    return gemv_multi_common(jobs, n_jobs, batch, cuda_stream, false, false, next, n_next, prev, n_prev);
}

int bitcos_gemv_multi(const bitcos_gemv_job *jobs, int n_jobs, int batch, void *cuda_stream) {
    return gemv_multi_common(jobs, n_jobs, batch, cuda_stream, false);
}

int bitcos_gemv_multi_group_scales(const bitcos_gemv_job *jobs, int n_jobs, int batch, void *cuda_stream) {
    return gemv_multi_common(jobs, n_jobs, batch, cuda_stream, false, true);
}

int bitcos_gemv_multi_bf16(const bitcos_gemv_job *jobs, int n_jobs, int batch, void *cuda_stream) {
    return gemv_multi_common(jobs, n_jobs, batch, cuda_stream, true);
}

int bitcos_gemv_blend_bf16(const bitcos_weights *W, const uint16_t *x_bf16, int batch, float *y, void *workspace,
                           size_t workspace_bytes, void *cuda_stream) {
    if (!W) return BITCOS_ERR_NULL;
    if (batch > 8) return BITCOS_ERR_SHAPE;
    const int8_t *x = reinterpret_cast<const int8_t *>(x_bf16);
    const int bad = check_common(kBitcos, W->bitmap, W->signs, W->tile_off, W->scales, W->M, W->K, x,
                                 reinterpret_cast<const float *>(x), batch, y, nullptr, workspace, workspace_bytes);
    if (bad) return bad;
    const Plan pl = one_tile_plan(kBitcos, W->M, W->K, batch <= 4 ? 4 : 8);
    Problem pr{};
    fill_problem(pr, W->bitmap, W->signs, W->tile_off, W->scales, W->M, W->K, x, nullptr, batch, y, nullptr, workspace);
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (batch <= 4) return launch<kBitcos, 4, false, false, true>(pr, pl, stream, W->tile_off_host);
    return launch<kBitcos, 8, false, false, true>(pr, pl, stream, W->tile_off_host);
}

int bitcos_gemv_bf16(const bitcos_weights *W, const uint16_t *x_bf16, int batch, float *y, int32_t *acc_debug,
                     void *workspace, size_t workspace_bytes, void *cuda_stream) {
    if (!W) return BITCOS_ERR_NULL;
    if (batch > 2) return BITCOS_ERR_SHAPE;
    const int8_t *x = reinterpret_cast<const int8_t *>(x_bf16);
    const int bad = check_common(kBitcos, W->bitmap, W->signs, W->tile_off, W->scales, W->M, W->K, x,
                                 reinterpret_cast<const float *>(x), batch, y, acc_debug, workspace, workspace_bytes);
    if (bad) return bad;
    const Plan pl = one_tile_plan(kBitcos, W->M, W->K, nb_bucket(batch, W->K));
    Problem pr{};
    fill_problem(pr, W->bitmap, W->signs, W->tile_off, W->scales, W->M, W->K, x, nullptr, batch, y, acc_debug, workspace);
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    const int nbk = nb_bucket(batch, W->K);
    if (nbk == 1) return launch<kBitcos, 1, false, true>(pr, pl, stream, W->tile_off_host);
    if (nbk == 2) return launch<kBitcos, 2, false, true>(pr, pl, stream, W->tile_off_host);
    return BITCOS_ERR_SHAPE;              // rows too long for the one- and two-token kernels
}

size_t bitcos_gemv_host_staging_bytes(int64_t M, int64_t K, int batch) {
    if (M < 1 || K < kGroup || K % kGroup != 0 || batch < 1 || batch > BITCOS_MAX_BATCH) return 0;
    const size_t xb = (static_cast<size_t>(batch) * K + 255) / 256 * 256;
    return xb + 256 + static_cast<size_t>(batch) * M * sizeof(float);
}

int bitcos_gemv_host(const bitcos_weights *W, const int8_t *x_host, const float *x_scale_host, int batch,
                     float *y_host, void *staging, size_t staging_bytes, void *workspace,
                     size_t workspace_bytes, void *cuda_stream) {
    if (!W || !x_host || !x_scale_host || !y_host || !staging) return BITCOS_ERR_NULL;
    const size_t need = bitcos_gemv_host_staging_bytes(W->M, W->K, batch);
    if (need == 0) return BITCOS_ERR_SHAPE;
    if (staging_bytes < need) return BITCOS_ERR_CAPACITY;
    if (!aligned16(staging)) return BITCOS_ERR_ALIGN;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    uint8_t *base = static_cast<uint8_t *>(staging);
    const size_t xb = (static_cast<size_t>(batch) * W->K + 255) / 256 * 256;
    int8_t *x_dev = reinterpret_cast<int8_t *>(base);
    float *xs_dev = reinterpret_cast<float *>(base + xb);
    float *y_dev = reinterpret_cast<float *>(base + xb + 256);
    int rc = check_cuda(cudaMemcpyAsync(x_dev, x_host, static_cast<size_t>(batch) * W->K, cudaMemcpyHostToDevice, stream));
    if (rc) return rc;
    rc = check_cuda(cudaMemcpyAsync(xs_dev, x_scale_host, static_cast<size_t>(batch) * sizeof(float),
                                    cudaMemcpyHostToDevice, stream));
    if (rc) return rc;
    rc = bitcos_gemv(W, x_dev, xs_dev, batch, y_dev, nullptr, workspace, workspace_bytes, cuda_stream);
    if (rc) return rc;
    rc = check_cuda(cudaMemcpyAsync(y_host, y_dev, static_cast<size_t>(batch) * W->M * sizeof(float),
                                    cudaMemcpyDeviceToHost, stream));
    if (rc) return rc;
    return check_cuda(cudaStreamSynchronize(stream));
}

int bitcos_gemv_multi_host(const bitcos_gemv_host_job *jobs, int n_jobs, int batch, void *cuda_stream) {
    if (!jobs) return BITCOS_ERR_NULL;
    if (n_jobs < 1 || n_jobs > kMaxJobs) return BITCOS_ERR_SHAPE;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    bitcos_gemv_job dev_jobs[kMaxJobs];
    float *y_dev[kMaxJobs];
    for (int j = 0; j < n_jobs; ++j) {
        const bitcos_gemv_host_job &jb = jobs[j];
        if (!jb.W || !jb.x_host || !jb.x_scale_host || !jb.y_host || !jb.staging) return BITCOS_ERR_NULL;
        const size_t need = bitcos_gemv_host_staging_bytes(jb.W->M, jb.W->K, batch);
        if (need == 0) return BITCOS_ERR_SHAPE;
        if (jb.staging_bytes < need) return BITCOS_ERR_CAPACITY;
        if (!aligned16(jb.staging)) return BITCOS_ERR_ALIGN;
        uint8_t *base = static_cast<uint8_t *>(jb.staging);
        const size_t xb = (static_cast<size_t>(batch) * jb.W->K + 255) / 256 * 256;
        dev_jobs[j].W = jb.W;
        dev_jobs[j].x = reinterpret_cast<const int8_t *>(base);
        dev_jobs[j].x_scale = reinterpret_cast<const float *>(base + xb);
        y_dev[j] = reinterpret_cast<float *>(base + xb + 256);
        dev_jobs[j].y = y_dev[j];
        dev_jobs[j].workspace = jb.workspace;
        dev_jobs[j].workspace_bytes = jb.workspace_bytes;
    }
    for (int j = 0; j < n_jobs; ++j) {
        uint8_t *base = static_cast<uint8_t *>(jobs[j].staging);
        const size_t xb = (static_cast<size_t>(batch) * jobs[j].W->K + 255) / 256 * 256;
        int rc = check_cuda(cudaMemcpyAsync(base, jobs[j].x_host, static_cast<size_t>(batch) * jobs[j].W->K,
                                            cudaMemcpyHostToDevice, stream));
        if (rc) return rc;
        rc = check_cuda(cudaMemcpyAsync(base + xb, jobs[j].x_scale_host, static_cast<size_t>(batch) * sizeof(float),
                                        cudaMemcpyHostToDevice, stream));
        if (rc) return rc;
    }
    int rc = bitcos_gemv_multi(dev_jobs, n_jobs, batch, cuda_stream);
    if (rc) return rc;
    for (int j = 0; j < n_jobs; ++j) {
        rc = check_cuda(cudaMemcpyAsync(jobs[j].y_host, y_dev[j], static_cast<size_t>(batch) * jobs[j].W->M * sizeof(float),
                                        cudaMemcpyDeviceToHost, stream));
        if (rc) return rc;
    }
    return check_cuda(cudaStreamSynchronize(stream));
}

}  // extern "C"

namespace {
// Copies pieces of a block between host memory that is mapped into the device and device memory.  In a recorded step these
// copies stand between kernels that are a few microseconds long, and a copy node is a hand-over to a copy engine and
// back with nothing overlapping; a kernel is launched like the products (the one behind it starts up while it
// runs, it starts up while the one before it runs) and moves the tens of kilobytes of a decode step in one trip over
// the bus.  2B-model layer, 22 KB in and 91 KB out: 40.3 -> 31.5 us a call, 30.8 with the outputs of every phase but
// the last copied while the later phases run (32B-model layer at sixteen tokens, 4.6 MB out: 236 -> 231 -> 196).
struct CopyPieces {
    const uint8_t *src;
    uint8_t *dst;
    int n;
    size_t off[kMaxJobs + 1], bytes[kMaxJobs + 1];      // pieces of both blocks at the same offsets
};
__global__ void __launch_bounds__(128) copy_pieces_kernel(const __grid_constant__ CopyPieces c) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const size_t i0 = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x, step = static_cast<size_t>(gridDim.x) * blockDim.x;
    for (int p = 0; p < c.n; ++p) {
        const uint8_t *src = c.src + c.off[p];
        uint8_t *dst = c.dst + c.off[p];
        size_t done = 0;
        if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0) {
            for (size_t i = i0; i < c.bytes[p] / 16; i += step) reinterpret_cast<uint4 *>(dst)[i] = __ldcv(reinterpret_cast<const uint4 *>(src) + i);
            done = c.bytes[p] / 16 * 16;
        }
        for (size_t i = done + i0; i < c.bytes[p]; i += step) dst[i] = __ldcv(reinterpret_cast<const unsigned char *>(src) + i);
    }
}
int launch_copy(const CopyPieces &c, cudaStream_t stream) {
    size_t total = 0;
    for (int p = 0; p < c.n; ++p) total += c.bytes[p];
    if (!total) return BITCOS_OK;
    const size_t blocks = (total / 16 + 127) / 128;
    return launch_pdl(copy_pieces_kernel, dim3(static_cast<unsigned>(blocks < 1 ? 1 : blocks < 256 ? blocks : 256)), 128, 0, stream, c);
}

// What a recorded step needs besides its arguments: the host blocks as the device sees them, a stream for the copies that
// run beside the products, and an event per fork and join.
struct RecordedCopies {
    const void *in_mapped;
    void *out_mapped;
    cudaStream_t side;
    cudaEvent_t event[BITCOS_MAX_PHASES + 1];
};

// The work of bitcos_gemv_phases_host on a stream: copy in, one launch per phase (each told which
// launch runs before it and which comes after it), copy out.  rec: given while the step is being recorded, else NULL (plain copies).
int host_step_enqueue(const bitcos_gemv_job *jobs, const int *job_phase, int n_jobs, int batch, const void *in_host,
                      void *in_device, size_t in_bytes, void *out_host, const void *out_device, size_t out_bytes,
                      const RecordedCopies *rec, cudaStream_t stream) {
    int rc;
    if (rec) {
        CopyPieces in{static_cast<const uint8_t *>(rec->in_mapped), static_cast<uint8_t *>(in_device), 1, {0}, {in_bytes}};
        rc = launch_copy(in, stream);
    } else {
        rc = check_cuda(cudaMemcpyAsync(in_device, in_host, in_bytes, cudaMemcpyHostToDevice, stream));
    }
    if (rc) return rc;
    // the outputs already on their way, as [begin, end) offsets of the block
    std::pair<size_t, size_t> sent[kMaxJobs];
    int n_sent = 0, forks = 0;
    auto output_range = [&](int j) {
        const size_t off = static_cast<size_t>(reinterpret_cast<const uint8_t *>(jobs[j].y) - static_cast<const uint8_t *>(out_device));
        return std::pair<size_t, size_t>(off, off + static_cast<size_t>(batch) * static_cast<size_t>(jobs[j].W->M) * sizeof(float));
    };
    const bitcos_weights *w[kMaxJobs];
    for (int j = 0; j < n_jobs; ++j) w[j] = jobs[j].W;
    int prev_first = 0, prev_n = 0;
    for (int first = 0; first < n_jobs;) {
        int last = first;
        while (last + 1 < n_jobs && job_phase[last + 1] == job_phase[first]) ++last;
        int next_n = 0;
        while (last + 1 + next_n < n_jobs && job_phase[last + 1 + next_n] == job_phase[last + 1] && next_n < kMaxPrefetch / 4) ++next_n;
        rc = bitcos_gemv_multi_chained(jobs + first, last - first + 1, batch, w + prev_first, prev_n, w + last + 1, next_n, stream);
        if (rc) return rc;
        if (rec && last + 1 < n_jobs && forks < BITCOS_MAX_PHASES) {
            // this phase's outputs go out beside the phases that follow, those that a later job writes over excepted
            // (what the caller gets is the block after the last phase)
            CopyPieces out{static_cast<const uint8_t *>(out_device), static_cast<uint8_t *>(rec->out_mapped), 0, {}, {}};
            for (int j = first; j <= last; ++j) {
                const std::pair<size_t, size_t> r = output_range(j);
                bool final = true;
                for (int i = last + 1; i < n_jobs; ++i) {
                    const std::pair<size_t, size_t> later = output_range(i);
                    final = final && (later.second <= r.first || r.second <= later.first);
                }
                if (!final) continue;
                out.off[out.n] = r.first;
                out.bytes[out.n++] = r.second - r.first;
                sent[n_sent++] = r;
            }
            if (out.n) {
                rc = check_cuda(cudaEventRecord(rec->event[forks], stream));
                if (!rc) rc = check_cuda(cudaStreamWaitEvent(rec->side, rec->event[forks], 0));
                if (!rc) rc = launch_copy(out, rec->side);
                if (rc) return rc;
                ++forks;
            }
        }
        prev_first = first;
        prev_n = last - first + 1;
        first = last + 1;
    }
    if (rec) {
        // everything that is not on its way yet: the last phase's outputs, and whatever else the block holds
        std::sort(sent, sent + n_sent);
        CopyPieces out{static_cast<const uint8_t *>(out_device), static_cast<uint8_t *>(rec->out_mapped), 0, {}, {}};
        size_t at = 0;
        for (int i = 0; i <= n_sent; ++i) {
            const size_t end = i < n_sent ? sent[i].first : out_bytes;
            if (end > at) {
                out.off[out.n] = at;
                out.bytes[out.n++] = end - at;
            }
            if (i < n_sent && sent[i].second > at) at = sent[i].second;
        }
        rc = launch_copy(out, stream);
        if (!rc && forks) rc = check_cuda(cudaEventRecord(rec->event[BITCOS_MAX_PHASES], rec->side));
        if (!rc && forks) rc = check_cuda(cudaStreamWaitEvent(stream, rec->event[BITCOS_MAX_PHASES], 0));
        return rc;
    }
    return check_cuda(cudaMemcpyAsync(out_host, out_device, out_bytes, cudaMemcpyDeviceToHost, stream));
}

// Recorded steps.  A record is keyed by everything the enqueued work depends on, by value: the job
// list, the descriptors behind it, the blocks and their sizes, the device; and it remembers every
// entry offset its plans took from the host copies of tile_off and where the host blocks were mapped, which a
// replay compares with what is there now (packed arrays in device memory may change freely between calls: the kernels read
// them when they run).  Anything that does not match is simply enqueued directly.
struct alignas(8) HostStepKey {
    int n_jobs, batch, device, pad;
    int phase[kMaxJobs];
    bitcos_gemv_job jobs[kMaxJobs];
    bitcos_weights w[kMaxJobs];
    const void *in_host, *out_device;
    void *in_device, *out_host;
    size_t in_bytes, out_bytes;
};
struct HostStepRecord {
    HostStepKey key;
    uint64_t hash = 0;
    std::vector<std::pair<const uint32_t *, uint32_t>> offsets;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    const void *in_mapped = nullptr;      // the host blocks as the record's copies address them
    void *out_mapped = nullptr;
    uint64_t last_use = 0;
    int seen = 0;          // calls with this key so far
    bool failed = false;   // recording did not work for this key: never tried again
};
constexpr int kHostStepRecords = 64;
HostStepRecord g_host_steps[kHostStepRecords];
std::mutex g_host_steps_lock;
uint64_t g_host_steps_clock = 0;
cudaStream_t g_record_stream = nullptr;
RecordedCopies g_recorded_copies;       // (used under the lock)

void host_step_key(HostStepKey &k, const bitcos_gemv_job *jobs, const int *job_phase, int n_jobs, int batch, const void *in_host,
                   void *in_device, size_t in_bytes, void *out_host, const void *out_device, size_t out_bytes) {
    std::memset(&k, 0, sizeof(k));
    k.n_jobs = n_jobs;
    k.batch = batch;
    cudaGetDevice(&k.device);
    for (int j = 0; j < n_jobs; ++j) {
        k.phase[j] = job_phase[j];
        std::memcpy(&k.jobs[j], &jobs[j], sizeof(bitcos_gemv_job));
        std::memcpy(&k.w[j], jobs[j].W, sizeof(bitcos_weights));
    }
    k.in_host = in_host;
    k.in_device = in_device;
    k.in_bytes = in_bytes;
    k.out_host = out_host;
    k.out_device = out_device;
    k.out_bytes = out_bytes;
}

// true: the step was launched on `stream` as a recorded graph.  false: the caller enqueues it directly
// (first sight of these arguments, a stale record, or recording is not possible).
bool host_step_replay(const bitcos_gemv_job *jobs, const int *job_phase, int n_jobs, int batch, const void *in_host,
                      void *in_device, size_t in_bytes, void *out_host, const void *out_device, size_t out_bytes,
                      cudaStream_t stream) {
    static const char *env = std::getenv("BITCOS_HOST_GRAPH");
    if (env && env[0] == '0') return false;
    static thread_local HostStepKey key;
    host_step_key(key, jobs, job_phase, n_jobs, batch, in_host, in_device, in_bytes, out_host, out_device, out_bytes);
    uint64_t hash = 1469598103934665603ull;      // (FNV-1a over the key's words: only to skip most comparisons)
    {
        const uint64_t *kw = reinterpret_cast<const uint64_t *>(&key);
        for (size_t i = 0; i < sizeof(key) / 8; ++i) hash = (hash ^ kw[i]) * 1099511628211ull;
    }
    std::lock_guard<std::mutex> guard(g_host_steps_lock);
    HostStepRecord *rec = nullptr, *oldest = &g_host_steps[0];
    for (HostStepRecord &r : g_host_steps) {
        if (r.seen && r.hash == hash && std::memcmp(&r.key, &key, sizeof(key)) == 0) rec = &r;
        if (r.last_use < oldest->last_use) oldest = &r;
    }
    if (!rec) {
        // first sight: remember the arguments (in the least recently used slot), enqueue directly this time
        rec = oldest;
        if (rec->exec) cudaGraphExecDestroy(rec->exec);
        if (rec->graph) cudaGraphDestroy(rec->graph);
        rec->exec = nullptr;
        rec->graph = nullptr;
        rec->offsets.clear();
        rec->key = key;
        rec->hash = hash;
        rec->seen = 1;
        rec->failed = false;
        rec->last_use = ++g_host_steps_clock;
        return false;
    }
    rec->last_use = ++g_host_steps_clock;
    if (rec->failed) return false;
    const void *in_mapped = bitcos_detail::mapped_host(in_host, in_bytes);
    void *out_mapped = bitcos_detail::mapped_host(out_host, out_bytes);
    if (rec->exec) {
        // the host blocks where the record's copies expect them, the entry offsets as its plans took them
        bool stale = in_mapped != rec->in_mapped || out_mapped != rec->out_mapped;
        for (size_t i = 0; !stale && i < rec->offsets.size(); ++i) stale = *rec->offsets[i].first != rec->offsets[i].second;
        if (stale) {
            cudaGraphExecDestroy(rec->exec);
            cudaGraphDestroy(rec->graph);
            rec->exec = nullptr;
            rec->graph = nullptr;
            rec->offsets.clear();
            rec->seen = 1;
            return false;
        }
        return cudaGraphLaunch(rec->exec, stream) == cudaSuccess;
    }
    // second sight: record the step on a stream of the library's own (nothing runs), then replay it
    ++rec->seen;
    if (!in_mapped || !out_mapped) return false;       // pageable host blocks: their copies are not recorded
    if (!g_record_stream) {
        bool ok = cudaStreamCreateWithFlags(&g_recorded_copies.side, cudaStreamNonBlocking) == cudaSuccess;
        for (cudaEvent_t &e : g_recorded_copies.event) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
        ok = ok && cudaStreamCreateWithFlags(&g_record_stream, cudaStreamNonBlocking) == cudaSuccess;
        if (!ok) {
            cudaGetLastError();
            g_record_stream = nullptr;
            rec->failed = true;
            return false;
        }
    }
    g_recorded_copies.in_mapped = rec->in_mapped = in_mapped;
    g_recorded_copies.out_mapped = rec->out_mapped = out_mapped;
    if (cudaStreamBeginCapture(g_record_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        cudaGetLastError();
        rec->failed = true;
        return false;
    }
    g_offset_log = &rec->offsets;
    const int rc = host_step_enqueue(jobs, job_phase, n_jobs, batch, in_host, in_device, in_bytes, out_host, out_device, out_bytes,
                                     &g_recorded_copies, g_record_stream);
    g_offset_log = nullptr;
    cudaGraph_t graph = nullptr;
    const cudaError_t ce = cudaStreamEndCapture(g_record_stream, &graph);
    if (rc || ce != cudaSuccess || !graph || cudaGraphInstantiate(&rec->exec, graph, 0) != cudaSuccess) {
        cudaGetLastError();
        if (graph) cudaGraphDestroy(graph);
        rec->exec = nullptr;
        rec->offsets.clear();
        rec->failed = true;
        return false;
    }
    rec->graph = graph;
    // (neighbouring blocks share entry offsets: every address once)
    std::sort(rec->offsets.begin(), rec->offsets.end());
    rec->offsets.erase(std::unique(rec->offsets.begin(), rec->offsets.end()), rec->offsets.end());
    return cudaGraphLaunch(rec->exec, stream) == cudaSuccess;
}
}  // namespace

extern "C" {

int bitcos_gemv_phases_host(const bitcos_gemv_job *jobs, const int *job_phase, int n_jobs, int batch, const void *in_host,
                            void *in_device, size_t in_bytes, void *out_host, const void *out_device, size_t out_bytes,
                            void *cuda_stream) {
    if (!jobs || !job_phase || !in_host || !in_device || !out_host || !out_device) return BITCOS_ERR_NULL;
    if (n_jobs < 1 || n_jobs > kMaxJobs || in_bytes == 0 || out_bytes == 0) return BITCOS_ERR_SHAPE;
    if (job_phase[0] != 0) return BITCOS_ERR_SHAPE;
    for (int j = 1; j < n_jobs; ++j)
        if (job_phase[j] < job_phase[j - 1] || job_phase[j] > job_phase[j - 1] + 1) return BITCOS_ERR_SHAPE;
    // every job's activations, scales and outputs must lie inside the two blocks that are copied
    const uintptr_t in0 = reinterpret_cast<uintptr_t>(in_device), out0 = reinterpret_cast<uintptr_t>(out_device);
    for (int j = 0; j < n_jobs; ++j) {
        if (!jobs[j].W || !jobs[j].x || !jobs[j].x_scale || !jobs[j].y) return BITCOS_ERR_NULL;
        const uintptr_t x = reinterpret_cast<uintptr_t>(jobs[j].x), xs = reinterpret_cast<uintptr_t>(jobs[j].x_scale),
                        y = reinterpret_cast<uintptr_t>(jobs[j].y);
        const size_t xb = static_cast<size_t>(batch) * static_cast<size_t>(jobs[j].W->K), yb = static_cast<size_t>(batch) * static_cast<size_t>(jobs[j].W->M) * 4;
        if (x < in0 || x + xb > in0 + in_bytes || xs < in0 || xs + static_cast<size_t>(batch) * 4 > in0 + in_bytes) return BITCOS_ERR_CAPACITY;
        if (y < out0 || y + yb > out0 + out_bytes) return BITCOS_ERR_CAPACITY;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    // A step that was seen before, argument for argument, is replayed as one CUDA graph (one call
    // into the driver instead of six); the first time round the work is enqueued directly.
    if (host_step_replay(jobs, job_phase, n_jobs, batch, in_host, in_device, in_bytes, out_host, out_device, out_bytes, stream))
        return check_cuda(cudaStreamSynchronize(stream));
    const int rc = host_step_enqueue(jobs, job_phase, n_jobs, batch, in_host, in_device, in_bytes, out_host, out_device,
                                     out_bytes, nullptr, stream);
    if (rc) return rc;
    return check_cuda(cudaStreamSynchronize(stream));
}

int trit5_gemv(const uint32_t *words, const uint16_t *scales_tiled, int64_t M, int64_t K, const int8_t *x,
               const float *x_scale, int batch, float *y, int32_t *acc_debug, void *workspace,
               size_t workspace_bytes, void *cuda_stream) {
    return gemv_common(kTrit5, words, nullptr, nullptr, scales_tiled, M, K, x, x_scale, batch, y, acc_debug,
                       workspace, workspace_bytes, cuda_stream);
}

int bit2_gemv(const uint32_t *words, const uint16_t *scales_tiled, int64_t M, int64_t K, const int8_t *x,
              const float *x_scale, int batch, float *y, int32_t *acc_debug, void *workspace,
              size_t workspace_bytes, void *cuda_stream) {
    return gemv_common(kBit2, words, nullptr, nullptr, scales_tiled, M, K, x, x_scale, batch, y, acc_debug,
                       workspace, workspace_bytes, cuda_stream);
}

}  // extern "C"

namespace {
template <int FMT>
int grouped_common(const bitcos_weights *experts, int n_experts, int64_t M, int64_t K, const int32_t *group_expert,
                   const int32_t *group_begin, int n_groups, const int32_t *pair_xrow, int n_pairs, int max_group_size,
                   const int8_t *x, int n_xrows, const float *x_scale, float *y, int32_t *acc_debug, void *workspace,
                   size_t workspace_bytes, void *cuda_stream, const int32_t *n_groups_dev = nullptr) {
    if (!experts || !group_expert || !group_begin || !pair_xrow || !x || !x_scale || !y || !workspace)
        return BITCOS_ERR_NULL;
    if (M < 1 || K < kGroup || K % kGroup != 0 || n_experts < 1 || n_groups < 1 || n_groups > 65535 ||
        (!n_groups_dev && n_pairs < n_groups) || n_pairs < 1 || n_xrows < 1 || max_group_size < 1 || max_group_size > BITCOS_MAX_BATCH)
        return BITCOS_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(y) || !aligned16(workspace) || (acc_debug && !aligned16(acc_debug)))
        return BITCOS_ERR_ALIGN;
    const size_t stride = workspace_bytes_for(M, K);
    if (workspace_bytes < stride * static_cast<size_t>(n_groups)) return BITCOS_ERR_CAPACITY;

    const Plan pl = make_plan(M, K, decoder_warps(max_group_size));
    Problem pr{};
    pr.x = x;
    pr.x_scale = x_scale;
    pr.xrow = pair_xrow;
    pr.y = y;
    pr.acc_debug = acc_debug;
    pr.M = M;
    pr.K = K;
    pr.G = static_cast<int>(K / kGroup);
    pr.RB = static_cast<int>(padded_rows(M) / kRows);
    pr.status = static_cast<unsigned int *>(workspace);
    GroupedArgs ga{experts, group_expert, group_begin, stride, n_experts, n_groups, 0, n_pairs, n_xrows, n_groups_dev};
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    const int nbk = nb_bucket(max_group_size, K);
    // BITCOS, up to 16 tokens per group, rows in one piece: the eight-token kernel, larger groups in two parts (their
    // weights are read twice, the second time from L2).  A routed group of more than eight tokens is rare, and the
    // sixteen-token kernel has 14 decoder warps instead of 20 and cuts rows of more than 14 groups in two: 128 experts of
    // 768x2048, 16 tokens x top-8: 55.3 -> 23.7 us, of 2048x768 40.6 -> 29.3.
    if constexpr (FMT == kBitcos) {
        const Plan p8 = make_plan(M, K, decoder_warps(8));
        if (max_group_size > 8 && p8.CS == 1) return launch_grouped<FMT, 8, true>(pr, p8, ga, n_groups, stream);
    }
    if (nbk == 1) return launch_grouped<FMT, 1>(pr, pl, ga, n_groups, stream);
    if (nbk == 2) return launch_grouped<FMT, 2>(pr, pl, ga, n_groups, stream);
    if (nbk == 4) return launch_grouped<FMT, 4>(pr, pl, ga, n_groups, stream);
    if (nbk == 8) return launch_grouped<FMT, 8>(pr, pl, ga, n_groups, stream);
    return launch_grouped<FMT, 16>(pr, pl, ga, n_groups, stream);
}
}  // namespace

extern "C" {

int bitcos_gemv_grouped(const bitcos_weights *experts, int n_experts, int64_t M, int64_t K, const int32_t *group_expert,
                        const int32_t *group_begin, int n_groups, const int32_t *pair_xrow, int n_pairs,
                        int max_group_size, const int8_t *x, int n_xrows, const float *x_scale, float *y,
                        int32_t *acc_debug, void *workspace, size_t workspace_bytes, void *cuda_stream) {
    return grouped_common<kBitcos>(experts, n_experts, M, K, group_expert, group_begin, n_groups, pair_xrow, n_pairs,
                                   max_group_size, x, n_xrows, x_scale, y, acc_debug, workspace, workspace_bytes, cuda_stream);
}

int bitcos_gemv_grouped_lists(const bitcos_weights *experts, int n_experts, int64_t M, int64_t K, const int32_t *group_expert,
                              const int32_t *group_begin, const int32_t *n_groups_device, int max_groups,
                              const int32_t *pair_xrow, int n_pairs, int max_group_size, const int8_t *x, int n_xrows,
                              const float *x_scale, float *y, int32_t *acc_debug, void *workspace, size_t workspace_bytes,
                              void *cuda_stream) {
    if (!n_groups_device) return BITCOS_ERR_NULL;
    return grouped_common<kBitcos>(experts, n_experts, M, K, group_expert, group_begin, max_groups, pair_xrow, n_pairs,
                                   max_group_size, x, n_xrows, x_scale, y, acc_debug, workspace, workspace_bytes, cuda_stream,
                                   n_groups_device);
}

int bitcos_group_pairs_device(const int32_t *pair_expert, const int32_t *pair_xrow, int n_pairs, int n_experts,
                              int32_t *group_expert, int32_t *group_begin, int32_t *pair_xrow_sorted, int32_t *order,
                              int32_t *n_groups, void *cuda_stream) {
    if (!pair_expert || !pair_xrow || !group_expert || !group_begin || !pair_xrow_sorted || !order || !n_groups)
        return BITCOS_ERR_NULL;
    if (n_pairs < 1 || n_pairs > BITCOS_GROUP_PAIRS_MAX || n_experts < 1 || n_experts > BITCOS_GROUP_EXPERTS_MAX) return BITCOS_ERR_SHAPE;
    return launch_pdl(group_pairs_kernel, dim3(1), kGroupPairsThreads, 0, static_cast<cudaStream_t>(cuda_stream), pair_expert,
                      pair_xrow, n_pairs, n_experts, group_expert, group_begin, pair_xrow_sorted, order, n_groups);
}

int trit5_gemv_grouped(const bitcos_weights *experts, int n_experts, int64_t M, int64_t K, const int32_t *group_expert,
                       const int32_t *group_begin, int n_groups, const int32_t *pair_xrow, int n_pairs,
                       int max_group_size, const int8_t *x, int n_xrows, const float *x_scale, float *y,
                       int32_t *acc_debug, void *workspace, size_t workspace_bytes, void *cuda_stream) {
    return grouped_common<kTrit5>(experts, n_experts, M, K, group_expert, group_begin, n_groups, pair_xrow, n_pairs,
                                  max_group_size, x, n_xrows, x_scale, y, acc_debug, workspace, workspace_bytes, cuda_stream);
}

int bit2_gemv_grouped(const bitcos_weights *experts, int n_experts, int64_t M, int64_t K, const int32_t *group_expert,
                      const int32_t *group_begin, int n_groups, const int32_t *pair_xrow, int n_pairs,
                      int max_group_size, const int8_t *x, int n_xrows, const float *x_scale, float *y,
                      int32_t *acc_debug, void *workspace, size_t workspace_bytes, void *cuda_stream) {
    return grouped_common<kBit2>(experts, n_experts, M, K, group_expert, group_begin, n_groups, pair_xrow, n_pairs,
                                 max_group_size, x, n_xrows, x_scale, y, acc_debug, workspace, workspace_bytes, cuda_stream);
}

}  // extern "C"
