// batch_noalloc.cu -- the batched launch for callers that cannot allocate.
//
// wxpy_batch_plan_create() allocates device memory for its tile list, and the
// one-shot wxpy_batch() takes stream-ordered scratch with cudaMallocAsync.
// Some callers can do neither: code whose device memory is entirely owned by
// another allocator (a framework's caching pool or a server's fixed arena)
// that must not see a cudaMalloc it did not make, one that could fail or
// synchronise the device in the middle of its work; and hot loops that cannot
// afford an allocation call at all.  wxpy_batch_noalloc() serves them: it
// computes the same results as wxpy_batch() from the caller's device table,
// and its only scratch is the fixed file-scope device array below, which
// every GPU that loads the library holds until the process exits.
//
// The plan is made on the device, in the caller's stream, in two launches:
//   1. a cluster of blocks sums the table's lengths, picks the tile length that
//      spreads the batch over the GPU (spread_tile), and
//      scans the tile counts into a per-segment plan;
//   2. a grid of warps runs the tiles; a warp finds its first tile's segment
//      in the plan, so no per-tile list is written and read.
// Descriptors with n <= 0, or with a null or misaligned pointer, get no
// tiles: they are skipped, never dereferenced.  Nothing else is checked: the
// caller guarantees that within each descriptor w is x, is y, or overlaps
// neither, and that no descriptor writes what another one reads or writes.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <mutex>

#include "cluster.cuh"
#include "internal.h"
#include "seg_search.cuh"

namespace wx {
namespace {

constexpr int64_t kNaMaxSegments = 65536;  // largest table this entry accepts
constexpr int kPlanBlocks = 8;             // one cluster plans a table
constexpr int kPer = 8;                    // segments per thread of it, at most
static_assert((int64_t)kPlanBlocks * 1024 * kPer >= kNaMaxSegments, "the plan holds the table");

struct NaScratch {
    SegPlan plan[kNaMaxSegments + 1];  // the last used one holds the tile count
};

// The scratch: about 1.5 MiB, fixed, shared by every call of the process on a
// device.  Host code must not use this name as an address (it is a host-side
// stand-in); the address comes from cudaGetSymbolAddress below.
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NaScratch)];

__device__ __forceinline__ bool usable(const wxpy_desc &d) {
    const uintptr_t bits = (uintptr_t)d.x | (uintptr_t)d.y | (uintptr_t)d.w;
    return d.n > 0 && d.x && d.y && d.w && (bits & 7u) == 0;
}

__device__ __forceinline__ int64_t warp_sum(int64_t v) {
    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// The value v of every block of the cluster, by all threads: slot[r] is block
// r's after the call.  v counts in thread 0.
template <int BLOCKS>
__device__ __forceinline__ void cluster_gather(int64_t *slot, int64_t v, int rank) {
    if constexpr (BLOCKS == 1) {
        if (threadIdx.x == 0) slot[0] = v;
        __syncthreads();
        return;
    }
    if (threadIdx.x == 0) {
        const uint32_t local = (uint32_t)__cvta_generic_to_shared(slot + rank);
        for (int r = 0; r < BLOCKS; ++r) {
            uint32_t remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(r));
            asm volatile("st.shared::cluster.s64 [%0], %1;" ::"r"(remote), "l"(v) : "memory");
        }
    }
    cluster_arrive();
    cluster_wait();
}

// 1. Tile length, tile counts, exclusive prefix over the segments, by one
// cluster: thread (block r, t) holds the lengths of up to kPer neighbouring
// segments in registers, so the table is read once.  Latency-bound: one table
// read, two scans and two exchanges through the cluster.  40000 segments up to
// 1024 elements take 85 us in all on GB300, against 195 with one block that
// reads the table twice, 4096 segments a round.
template <int BLOCKS>
__global__ void __cluster_dims__(BLOCKS, 1, 1) __launch_bounds__(1024)
    na_plan_kernel(const wxpy_desc *table, int64_t count, NaScratch *sc) {
    __shared__ int64_t warp_sums[32];
    __shared__ int64_t elems[BLOCKS], tiles_of[BLOCKS];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, rank = blockIdx.x;
    // no block's shared memory is written before it has started
    cluster_arrive();
    pdl_enter();
    cluster_wait();
    const int per = (int)((count + BLOCKS * 1024 - 1) / (BLOCKS * 1024));  // <= kPer
    const int64_t s0 = ((int64_t)rank * 1024 + tid) * per;
    int64_t n[kPer], total = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        n[k] = 0;
        if (k < per && s0 + k < count) {
            const wxpy_desc d = table[s0 + k];
            if (usable(d)) n[k] = d.n;
        }
        total += n[k];
    }
    total = warp_sum(total);
    if (lane == 0) warp_sums[wid] = total;
    __syncthreads();
    total = warp_sum(warp_sums[lane]);
    cluster_gather<BLOCKS>(elems, total, rank);
    total = 0;
    for (int r = 0; r < BLOCKS; ++r) total += elems[r];
    const int64_t len = spread_tile(total);
    const int shift = 63 - __clzll(len);
    int64_t mine = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) mine += (n[k] + len - 1) >> shift;
    int64_t v = mine;  // inclusive scan across the block
    for (int off = 1; off < 32; off <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += u;
    }
    if (lane == 31) warp_sums[wid] = v;
    __syncthreads();
    int64_t ws = warp_sums[lane];
    for (int off = 1; off < 32; off <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, ws, off);
        if (lane >= off) ws += u;
    }
    int64_t at = v - mine + (wid ? __shfl_sync(0xffffffffu, ws, wid - 1) : 0);
    cluster_gather<BLOCKS>(tiles_of, __shfl_sync(0xffffffffu, ws, 31), rank);
    int64_t all = 0;
    for (int r = 0; r < BLOCKS; ++r) {
        if (r == rank) at += all;
        all += tiles_of[r];
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (k < per && s0 + k < count) sc->plan[s0 + k] = seg_plan_of(n[k], at, len, 2);
        at += (n[k] + len - 1) >> shift;
    }
    if (rank == 0 && tid == 0) sc->plan[count] = seg_plan_of(0, all, len, 2);
}

// 2. The tiles, by the batched kernel's tile body with every product in the
// integer pipelines.  Bound as that kernel: HBM, once the batch fills the GPU.
// GB300, 1024 segments up to 2^16 elements stored back to back (6.0e6 in all):
// 34 us, against 77 with 8192-element tiles, a tile list written and
// read by two kernels, and FP64 products.
__global__ void __launch_bounds__(256, 3) na_run_kernel(const wxpy_desc *table, int64_t count,
                                                        const NaScratch *sc) {
    pdl_enter();
    run_plan_tiles<3, kTileU>(table, sc->plan, count);
}

constexpr int kMaxDev = 64;
// Device address of the scratch array per device: null until a lookup has
// succeeded.  Only a successful lookup is kept, so a lookup that failed (a
// first call made during a stream capture, or with an error pending) is
// simply tried again by the next call.
std::atomic<void *> g_na_ptr[kMaxDev];
std::mutex g_na_mu;

// The scratch's device address on device `dev` (current); nullptr and the
// error recorded when the lookup fails.
NaScratch *scratch_address(int dev, int *status) {
    void *p = g_na_ptr[dev].load(std::memory_order_acquire);
    if (p) return (NaScratch *)p;
    std::lock_guard<std::mutex> lk(g_na_mu);
    p = g_na_ptr[dev].load(std::memory_order_relaxed);
    if (!p) {
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            cudaGetLastError();  // clear a non-sticky error; the next call retries
            *status = fail_cuda(e != cudaSuccess ? e : cudaErrorInvalidSymbol,
                                "cudaGetSymbolAddress(scratch)");
            return nullptr;
        }
        g_na_ptr[dev].store(p, std::memory_order_release);
    }
    return (NaScratch *)p;
}

}  // namespace
}  // namespace wx

using namespace wx;

extern "C" int wxpy_batch_noalloc(const wxpy_desc *dev_table, int64_t count, void *stream) {
    if (count < 0) return fail(WXPY_EINVAL, "negative segment count");
    if (count == 0) return WXPY_OK;
    if (count > kNaMaxSegments)
        return fail(WXPY_EINVAL,
                    "%lld segments exceed the %lld that the fixed scratch of "
                    "wxpy_batch_noalloc holds; use wxpy_batch or split the table",
                    (long long)count, (long long)kNaMaxSegments);
    if (!dev_table || ((uintptr_t)dev_table & 7u))
        return fail(WXPY_EINVAL, "null or misaligned device table");
    int st = WXPY_OK;
    const DeviceProps *dp = current_device(&st);
    if (!dp) return st;
    const int dev = dp->device;
    if (dev >= kMaxDev) return fail(WXPY_EINVAL, "device ordinal %d out of range", dev);
    // With the device current: the device address of the scratch array,
    // looked up on the first successful call for this device.
    NaScratch *sc = scratch_address(dev, &st);
    if (!sc) return st;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = injected_launch_error();
    if (e == cudaSuccess) {
        // a table of one or two segments per thread of one block does without the
        // cluster's exchanges (about a microsecond)
        e = count <= 2048 ? launch_pdl(&na_plan_kernel<1>, 1u, 1024u, s, dev_table, count, sc)
                          : launch_pdl(&na_plan_kernel<kPlanBlocks>, (unsigned)kPlanBlocks, 1024u, s,
                                       dev_table, count, sc);
    }
    if (e == cudaSuccess)
        e = launch_pdl(&na_run_kernel, (unsigned)dp->sm_count * 8u, 256u, s, dev_table, count,
                       (const NaScratch *)sc);
    if (e != cudaSuccess) return fail_cuda(e, "wxpy_batch_noalloc launch");
    return WXPY_OK;
}
