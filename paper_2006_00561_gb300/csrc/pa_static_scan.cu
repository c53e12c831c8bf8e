// pa_static_scan.cu -- copy counts and their exclusive scan without any
// device allocation (pa_copy_counts_scan_noalloc in include/pa.h).
//
// Some callers cannot allocate device memory at all, not even through a
// caller-side allocator: code that runs while a CUDA graph is being captured,
// plugins whose host process owns every allocation, and embedded callers with
// a fixed memory budget.  For them this entry point computes the
// nearest-integer copy counts and their exclusive scan from buffers the
// caller already has, and keeps the only scratch it needs (one word per tile
// of the scan) in the file-scope array below.  That array is part of the library's image:
// every GPU that loads the library holds it until the process exits.
#include <mutex>

#include "pa_internal.cuh"

namespace pa {
namespace {

constexpr int SS_THREADS = 256;
constexpr int SS_ITEMS = 8;
constexpr int SS_TILE = SS_THREADS * SS_ITEMS;  // replicas per tile
constexpr int SS_MAX_TILES = PA_NOALLOC_MAX_REPLICAS / SS_TILE;
static_assert(SS_MAX_TILES * SS_TILE == PA_NOALLOC_MAX_REPLICAS, "whole tiles");

struct StaticScanScratch {
    // per tile: the sum of its counts, bit 32 set if a level was out of range
    unsigned long long tile[SS_MAX_TILES];
};

// The scratch.  Shared by every call in the process.
static __device__ __align__(256) StaticScanScratch g_scan_scratch;

// Two passes, no CTA waits on another: k_static_counts writes the counts and
// every tile's sum, k_static_offsets adds up the sums of the tiles before its
// own (at most 16 loads a thread, all independent), scans its tile's counts,
// which are still in L2, and writes the offsets.  A single pass with a decoupled
// lookback saves re-reading the counts, but its prefix moves from tile to
// tile in L2 round trips: 3 000 017 replicas (1465 tiles) took 64.4 us on GB300
// with one descriptor at a time, 51.2 us with 32, 42.6 us with 256; the two passes
// take 12.6 us a call (2.9 TB/s over the caller's arrays), 16.4 as single launches
// instead of a chain; up to 10^6 replicas a call is 6.1 to 6.6 us (8.2 to 12.3), its
// launches and each pass's two dependent L2 round trips.
//
// VEC: the caller's three arrays are 16-byte aligned, so a thread's eight
// replicas move as 16-byte words.
template <bool VEC>
__global__ void __launch_bounds__(SS_THREADS)
    k_static_counts(StaticScanScratch* s, const uint32_t* ebin, uint32_t R, const uint32_t* tab_n,
                    const uint32_t* tab_F, uint32_t bins, uint32_t step, uint32_t ctr3, uint32_t k0,
                    uint32_t k1, uint32_t* counts) {
    __shared__ uint32_t s_warp[SS_THREADS / 32];
    chain_wait();
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const uint32_t base = blockIdx.x * SS_TILE;
    uint32_t sum = 0, r[SS_ITEMS];
    bool bad = false;
#pragma unroll
    for (int j0 = 0; j0 < SS_ITEMS; j0 += 4) {
        const uint32_t i0 = base + (uint32_t)t * SS_ITEMS + j0;
        uint4 u = make_uint4(0, 0, 0, 0);
        uint32_t lev[4] = {0, 0, 0, 0};
        if (i0 < R) u = philox(i0 >> 2, step, 0u, ctr3, k0, k1);
        if (VEC && i0 + 4 <= R) {
            const uint4 e4 = *reinterpret_cast<const uint4*>(ebin + i0);
            lev[0] = e4.x, lev[1] = e4.y, lev[2] = e4.z, lev[3] = e4.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j < R) lev[j] = ebin[i0 + j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t v = 0;
            if (i0 + j < R) {
                const uint32_t k = lev[j];
                if (k < bins) v = tab_n[k] + (pick(u, (uint32_t)j) < tab_F[k] ? 1u : 0u);
                else bad = true;
            }
            r[j0 + j] = v;
            sum += v;
        }
    }
#pragma unroll
    for (int j0 = 0; j0 < SS_ITEMS; j0 += 4) {  // after all loads: the compiler may not move them up
        const uint32_t i0 = base + (uint32_t)t * SS_ITEMS + j0;
        if (VEC && i0 + 4 <= R) {
            *reinterpret_cast<uint4*>(counts + i0) = make_uint4(r[j0], r[j0 + 1], r[j0 + 2], r[j0 + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j < R) counts[i0 + j] = r[j0 + j];
        }
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) s_warp[wid] = sum;
    const int any = __syncthreads_or(bad);
    if (t == 0) {
        uint32_t tot = 0;
#pragma unroll
        for (int w = 0; w < SS_THREADS / 32; ++w) tot += s_warp[w];
        s->tile[blockIdx.x] = ((unsigned long long)(any ? 1u : 0u) << 32) | tot;
    }
}

template <bool VEC>
__global__ void __launch_bounds__(SS_THREADS)
    k_static_offsets(const StaticScanScratch* s, const uint32_t* counts, uint32_t R,
                     uint32_t* offsets, uint32_t* total) {
    __shared__ uint32_t s_warp[SS_THREADS / 32], s_before[SS_THREADS / 32];
    chain_wait();
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const uint32_t tile = blockIdx.x, base = tile * SS_TILE;
    uint32_t r[SS_ITEMS];
    uint32_t sum = 0;
#pragma unroll
    for (int j0 = 0; j0 < SS_ITEMS; j0 += 4) {
        const uint32_t i0 = base + (uint32_t)t * SS_ITEMS + j0;
        if (VEC && i0 + 4 <= R) {
            const uint4 c4 = *reinterpret_cast<const uint4*>(counts + i0);
            r[j0] = c4.x, r[j0 + 1] = c4.y, r[j0 + 2] = c4.z, r[j0 + 3] = c4.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) r[j0 + j] = i0 + j < R ? counts[i0 + j] : 0u;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) sum += r[j0 + j];
    }
    // the tiles before this one, and whether any up to it saw a bad level
    uint32_t ahead = 0;
    bool bad = false;
    for (uint32_t k = t; k <= tile; k += SS_THREADS) {
        const unsigned long long v = s->tile[k];
        if (k < tile) ahead += (uint32_t)v;
        bad |= (v >> 32) != 0;
    }
    ahead = __reduce_add_sync(0xffffffffu, ahead);
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[wid] = incl;
    if (lane == 0) s_before[wid] = ahead;
    const int any = __syncthreads_or(bad);
    uint32_t o = incl - sum;
#pragma unroll
    for (int w = 0; w < SS_THREADS / 32; ++w) {
        o += s_before[w];
        if (w < wid) o += s_warp[w];
    }
#pragma unroll
    for (int j0 = 0; j0 < SS_ITEMS; j0 += 4) {
        const uint32_t i0 = base + (uint32_t)t * SS_ITEMS + j0;
        uint32_t oo[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            oo[j] = o;
            o += r[j0 + j];
        }
        if (VEC && i0 + 4 <= R) {
            *reinterpret_cast<uint4*>(offsets + i0) = make_uint4(oo[0], oo[1], oo[2], oo[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j < R) offsets[i0 + j] = oo[j];
        }
        if (i0 < R && R - 1 - i0 < 4) *total = any ? 0xffffffffu : o;  // the last replica's group
    }
}

// Device address of the scratch in the current context.  Host code may not use
// the symbol itself as a pointer: on the host it only names the array.  The
// address belongs to the context that loaded the module, so it is cached per
// context, keyed by the driver's context id, which is unique for the life of
// the process: a caller running in its own (non-primary) context, or a
// primary context re-created after cudaDeviceReset, gets a fresh lookup.
// The two driver calls are reached through the runtime's entry-point query,
// so the library does not link libcuda itself.
typedef int (*CtxGetCurrentFn)(void** ctx);
typedef int (*CtxGetIdFn)(void* ctx, unsigned long long* id);

struct ScratchCacheEntry {
    unsigned long long ctx_id;
    void* addr;
};
constexpr int SCRATCH_CACHE = 16;
std::mutex g_mu;
ScratchCacheEntry g_cache[SCRATCH_CACHE];
int g_cache_used = 0, g_cache_next = 0;
CtxGetCurrentFn g_ctx_get_current = nullptr;
CtxGetIdFn g_ctx_get_id = nullptr;

cudaError_t current_context_id(unsigned long long* id) {
    if (!g_ctx_get_current || !g_ctx_get_id) {
        void* f0 = nullptr;
        void* f1 = nullptr;
        cudaDriverEntryPointQueryResult q0, q1;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f0, 12000,
                                                         cudaEnableDefault, &q0);
        if (e != cudaSuccess || q0 != cudaDriverEntryPointSuccess || !f0)
            return e != cudaSuccess ? e : cudaErrorNotSupported;
        e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f1, 12000, cudaEnableDefault, &q1);
        if (e != cudaSuccess || q1 != cudaDriverEntryPointSuccess || !f1)
            return e != cudaSuccess ? e : cudaErrorNotSupported;
        g_ctx_get_current = reinterpret_cast<CtxGetCurrentFn>(f0);
        g_ctx_get_id = reinterpret_cast<CtxGetIdFn>(f1);
    }
    void* ctx = nullptr;
    if (g_ctx_get_current(&ctx) != 0 || !ctx) return cudaErrorDeviceUninitialized;
    if (g_ctx_get_id(ctx, id) != 0) return cudaErrorDeviceUninitialized;
    return cudaSuccess;
}

cudaError_t scratch_address(void** out) {
    std::lock_guard<std::mutex> lock(g_mu);
    unsigned long long id = 0;
    cudaError_t e = current_context_id(&id);
    if (e == cudaErrorDeviceUninitialized) {
        // no context is current yet: the symbol lookup makes the runtime bind
        // the device's primary context, after which the id can be read
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_scan_scratch);
        if (e != cudaSuccess) return e;
        e = current_context_id(&id);
    }
    if (e != cudaSuccess) return e;
    for (int i = 0; i < g_cache_used; ++i) {
        if (g_cache[i].ctx_id == id) {
            *out = g_cache[i].addr;
            return cudaSuccess;
        }
    }
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_scan_scratch);
    if (e != cudaSuccess) return e;
    int slot;
    if (g_cache_used < SCRATCH_CACHE) {
        slot = g_cache_used++;
    } else {  // evict the oldest entry
        slot = g_cache_next;
        g_cache_next = (g_cache_next + 1) % SCRATCH_CACHE;
    }
    g_cache[slot].ctx_id = id;
    g_cache[slot].addr = p;
    *out = p;
    return cudaSuccess;
}

}  // namespace
}  // namespace pa

extern "C" int pa_copy_counts_scan_noalloc(const uint32_t* d_ebin, int64_t R,
                                           const uint32_t* d_tab_n, const uint32_t* d_tab_F,
                                           int64_t bins, uint64_t seed, int32_t step,
                                           int32_t instance_id, uint32_t* d_counts,
                                           uint32_t* d_offsets, uint32_t* d_total,
                                           void* stream) {
    if (R < 0 || R > PA_NOALLOC_MAX_REPLICAS) return PA_ERR_INVALID_ARG;
    if (bins < 1 || bins > 0xffffffffll || step < 0 || instance_id < 0 ||
        instance_id >= (1 << 28))
        return PA_ERR_INVALID_ARG;
    if (!d_total || (R > 0 && (!d_ebin || !d_tab_n || !d_tab_F || !d_counts || !d_offsets)))
        return PA_ERR_INVALID_ARG;
    void* addr = nullptr;
    if (pa::scratch_address(&addr) != cudaSuccess) return PA_ERR_CUDA;
    auto* s = static_cast<pa::StaticScanScratch*>(addr);
    cudaStream_t st = (cudaStream_t)stream;
    if (R == 0) return cudaMemsetAsync(d_total, 0, 4, st) == cudaSuccess ? PA_OK : PA_ERR_CUDA;
    const uint32_t tiles = (uint32_t)((R + pa::SS_TILE - 1) / pa::SS_TILE);
    const uint32_t ctr3 = (pa::TAG_RESAMPLE << 28) | (uint32_t)instance_id;
    const bool vec = (((uintptr_t)d_ebin | (uintptr_t)d_counts | (uintptr_t)d_offsets) & 15u) == 0;
    const void* count = vec ? (const void*)pa::k_static_counts<true> : (const void*)pa::k_static_counts<false>;
    const void* scan = vec ? (const void*)pa::k_static_offsets<true> : (const void*)pa::k_static_offsets<false>;
    uint32_t r = (uint32_t)R, nb = (uint32_t)bins, st32 = (uint32_t)step, c3 = ctr3;
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    void* cargs[] = {&s, &d_ebin, &r, &d_tab_n, &d_tab_F, &nb, &st32, &c3, &k0, &k1, &d_counts};
    void* sargs[] = {&s, &d_counts, &r, &d_offsets, &d_total};
    if (pa::launch_chained(count, dim3(tiles), dim3(pa::SS_THREADS), 0, st, cargs) != cudaSuccess ||
        pa::launch_chained(scan, dim3(tiles), dim3(pa::SS_THREADS), 0, st, sargs) != cudaSuccess)
        return PA_ERR_CUDA;
    return PA_OK;
}
