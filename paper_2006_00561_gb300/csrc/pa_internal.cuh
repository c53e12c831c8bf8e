// pa_internal.cuh -- device-side data of one population-annealing run and the
// launchers the host engine (pa_engine.cu) calls.  Every array lives in the
// caller's workspace; the kernels read the run's scalars (population size,
// step index, buffer parity, sweep counter) from device memory, so a step can
// be enqueued or replayed from a CUDA graph without any host round trip.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/pa.h"

namespace pa {

// Counter tags: top four bits of Philox counter word 3 (low 28 bits: instance).
constexpr uint32_t TAG_INIT = 1u;
constexpr uint32_t TAG_SWEEP = 2u;
constexpr uint32_t TAG_RESAMPLE = 3u;
constexpr uint32_t TAG_COUPLING = 4u;
constexpr uint32_t TAG_POISSON = 5u;
constexpr uint32_t TAG_MULTINOMIAL = 6u;
constexpr int P1_MAX = 16;  // entries of the Poisson(1) inversion table

// Sticky status bits of DevState::status.
constexpr uint32_t ST_CAPACITY = 1u;
constexpr uint32_t ST_TIMEOUT = 2u;
constexpr uint32_t ST_EMPTY = 4u;
constexpr uint32_t ST_DONE = 8u;
constexpr uint32_t ST_INVARIANT = 16u;

// Scalars of a run, in device memory (first 256 bytes of the workspace).
struct DevState {
    uint32_t step;          // current beta index i
    uint32_t R;             // current population size
    uint32_t R_prev;        // population entering the last resample
    uint32_t epoch;         // bumped by every reweight; tags lookback descriptors
    uint32_t tile_counter;  // dynamic tile ids of the resample kernel
    uint32_t status;        // sticky ST_* bits
    uint32_t cur;           // population buffer holding the current replicas
    uint32_t src;           // buffer the last resample read from
    uint32_t sweep_base;    // global index of the next Metropolis sweep
    uint32_t active;        // 1 if the reweight of this step succeeded
    uint32_t kref;          // lowest occupied energy level at the last reweight
    uint32_t negbonds;      // number of J = -1 bonds (U mod 2 = negbonds mod 2)
    double lnQ, lnZ, S;
    unsigned long long sweeps_done;
    unsigned long long tau_done;  // CTAs of the running multi-CTA reweight that are done
    unsigned long long sources;   // replicas with a copy count > 0, summed over all resamples
    uint32_t over_n;              // copies left to k_spread: entries of RunDev::srcmap2
    uint32_t pad;
};
// Results of a reweight that shares its launch with the observables of the step
// before, until the last block moves them to DevState (second half of its slot).
struct TauNext {
    double lnQ, lnZ, S;
    uint32_t kref;
};
static_assert(sizeof(DevState) <= 128 && sizeof(TauNext) <= 128, "DevState's slot is 256 bytes");

// Per-step record, same layout as pa_obs.
static_assert(sizeof(pa_obs) == 104 && offsetof(pa_obs, sumM2) - offsetof(pa_obs, sumE) == 24 &&
                  offsetof(pa_obs, chi) - offsetof(pa_obs, e) == 24,
              "pa_obs layout (the sums and the averages are four in a row)");

// Everything a kernel needs, passed by value.
struct RunDev {
    DevState* st;
    uint8_t* spins[2];          // population buffers, cap_alloc * stride bytes each
    uint32_t* ebin[2];          // energy level k = U >> 1 per replica
    int32_t* mag[2];            // magnetisation per replica
    uint32_t* counts;           // copy counts of the last resample
    uint32_t* offsets;          // exclusive scan of the counts
    uint32_t* srcmap;           // [cap] source replica of every slot the last resample filled
    uint32_t* srcmap2;          // [cap] the same after a redistribution permuted the slots;
                                // in a whole resample the list of k_spread
    unsigned long long* accum;  // [2] = sum |M|, sum M^2 of the running measurement
    uint32_t* hist;             // [bins] energy histogram of the running measurement
    uint32_t* tab_n;            // [bins] floor(tau_k)
    uint32_t* tab_F;            // [bins] floor(frac(tau_k) * 2^32)
    const uint32_t* thr;        // [(K+1)*4]: T0, T1, T2 (clamped to u32), bit c of [3] = T_c is 2^32
    const double* dtab;         // [ndist * bins] Eq. 3 weights
    const uint32_t* dsel;       // [K+1] weight table of step i
    const double* beta;         // [K+1]
    const double* dbeta;        // [K+1] beta_i - beta_{i-1} (negative when heating)
    unsigned long long* desc;   // [tiles] lookback descriptors
    unsigned long long* mn_cum;   // multinomial: [cap] cumulative fixed-point weights C_i
    unsigned long long* mn_tiles; // multinomial: [tiles + 1] tile prefixes, then the total
    pa_obs* obs;                // [K+1] per-step records
    uint32_t* jpk;              // packed couplings [dim][nwords] (bit set: J = -1), PMJ only
    int8_t* j8;                 // int8 couplings [N][dim], PMJ only
    uint64_t seed, coupling_seed;
    uint32_t instance;          // instance id (< 2^28)
    int32_t dim, L, layout, model, K;
    int64_t N, bins;
    uint32_t stride;            // bytes per replica (multiple of 16)
    uint32_t nwords;            // packed: 32-bit words per replica
    uint32_t cap;               // logical capacity
    uint32_t cap_alloc;         // slots in each buffer
    uint32_t R0;
    uint32_t tiles;             // descriptors available
    uint32_t slice_lg;          // log2 of the CTAs that share a resample tile (resample_slices)
    uint32_t rk0[10], rk1[10];  // Philox round keys of `seed` (key + r * Weyl constant)
    uint32_t one;               // the value 1, opaque to the compiler (multiply-add tests)
    int32_t theta;              // sweeps per annealing step
    int32_t init;               // PA_INIT_RANDOM | PA_INIT_GROUND
    int32_t resample;           // PA_RESAMPLE_NEAREST | PA_RESAMPLE_POISSON
    uint32_t p1_len;            // entries of p1
    uint32_t p1[P1_MAX];        // Poisson(1) thresholds floor(2^32 P(X <= m))
    // Slots the plain sweep kernels visit: [slot_lo, min(R, slot_hi)).  0 and
    // 0xffffffff (the whole population) except in the launches of a
    // streamed step, whose bounds are multiples of 32.
    uint32_t slot_lo, slot_hi;
    uint32_t debug;  // PA_DEBUG_* test hooks, 0 in normal operation
    // the resample clears the histogram and the magnetisation sums for the sweep
    // that follows it (whole steps; a lone resample leaves them)
    uint32_t clear_hist;
    uint32_t spread;  // replicas may get many copies: k_spread shares them out (many_copies)
};

// A batch of runs stepped together (pa_batch_* in include/pa.h).  Arrays in
// the batch workspace; counters are cleared by the batched reweight kernel at
// the start of every step.
struct BatchDev {
    const RunDev* runs;          // [nruns]
    uint32_t nruns;
    int64_t max_bins;            // energy levels of the run with the most
    const uint32_t* tile_base;   // [nruns + 1] prefix sums of each run's slices of tiles
    uint32_t total_tiles;        // slices of all tiles
    uint32_t any_spread;         // some run's RunDev::spread is set
    uint32_t any_poisson;        // some run resamples by the Poisson rule
    uint32_t any_multinomial;    // some run resamples by multinomial draws
    uint32_t* counters;          // [0]: resample tiles, [1 + c]: sweep chunks of class c
    uint32_t ncounters;
};

// One (layout, dim, L, model) class of a batch: the runs one sweep kernel
// instantiation serves.  Global slot g of the class lies in run run_ids[j]
// when slot_base[j] <= g < slot_base[j + 1] (capacities rounded up to 32, so
// a chunk of `chunk` slots never straddles two runs).
struct BatchSweepArgs {
    const RunDev* runs;
    const uint32_t* run_ids;     // [n]
    const uint32_t* slot_base;   // [n + 1]
    uint32_t n;
    uint32_t total_slots;
    uint32_t* counter;           // chunk counter of this class
    uint32_t chunk;              // slots per claim: 1, 2, 4, 8, 16 or 32
};

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two 32x32
// multiplies whose high halves are xored with the other words and the key;
// the key advances by the two Weyl constants after every round.
__device__ __forceinline__ uint4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                        uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t a = c0, b = c2;
        const uint32_t hiA = __umulhi(0xD2511F53u, a), loA = 0xD2511F53u * a;
        const uint32_t hiB = __umulhi(0xCD9E8D57u, b), loB = 0xCD9E8D57u * b;
        c0 = hiB ^ c1 ^ k0;
        c1 = loB;
        c2 = hiA ^ c3 ^ k1;
        c3 = loA;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return make_uint4(c0, c1, c2, c3);
}

__device__ __forceinline__ uint32_t pick(const uint4& v, uint32_t j) {
    return j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w;
}

// Programmatic dependent launch along a step's chain of kernels (reweight ->
// resample -> sweep -> observables -> the next reweight): a kernel's blocks
// become resident as its predecessor's last blocks leave, and wait here, before
// they touch memory, until all of its writes are visible.  Every block of every
// kernel of the chain passes here first, so "the predecessor has finished" holds
// for all earlier ones too.  A plain launch passes at once.  On GB300 a step of
// 1000 replicas at L = 16 took 39.1 us by single launches and 31.3 us so, all else
// equal.
// What the predecessors write is not read-only for such a kernel's lifetime, which
// starts before the wait: its pointers carry no __restrict__, and it takes plain or
// __ldcg loads, never __ldg (a compiler may move invariant loads above the wait).
// Letting the successor in at the start of a kernel (launch_dependents) fills
// SMs with waiting blocks that keep out the sweep's: up to 78 us instead of 34 for
// 4099 spin glasses of L = 6.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
inline cudaError_t launch_chained(const void* fn, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                  void** args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

// Descriptors of a single-pass scan: flag (aggregate or prefix) << 62 | epoch
// << 32 | value.
constexpr unsigned long long DESC_AGG = 1ull;
constexpr unsigned long long DESC_PREFIX = 2ull;
constexpr unsigned LOOKBACK_SPIN_LIMIT = 1u << 22;

__device__ __forceinline__ void st_release(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long desc_make(unsigned long long flag, uint32_t epoch,
                                                         uint32_t value) {
    return (flag << 62) | ((unsigned long long)(epoch & 0x3fffffffu) << 32) | value;
}

// Decoupled lookback of tile `tile` > 0, by all NW warps of a CTA: the sum of
// the counts of all tiles before it.  Warp w watches the 32 predecessors tile -
// 1 - 32 w - lane; as soon as a prefix is among them and every nearer one has
// published its aggregate the warp's sum is known, without a prefix when all
// 32 aggregates are there, and the CTA's window of 32 NW tiles moves on.  The
// wait is a chain of L2 round trips (about 0.7 us each), as long as the number
// of windows between a tile and the nearest prefix.  Bounded:
// after LOOKBACK_SPIN_LIMIT polls without progress it returns what it has and
// ok = false.  All threads return the same values; sm is free for reuse only
// after a further barrier.
template <int NW>
struct LookSmem {
    uint32_t sum[2][NW], found[2][NW];
};
template <int NW>
__device__ __forceinline__ uint32_t lookback(const unsigned long long* desc, uint32_t tile,
                                             uint32_t epoch, LookSmem<NW>& sm, bool& ok) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t tag = epoch & 0x3fffffffu;
    uint32_t excl = 0;
    ok = true;
    int ph = 0;
    for (int64_t top = (int64_t)tile - 1;; top -= 32 * NW, ph ^= 1) {
        const int64_t p = top - 32 * wid - lane;
        unsigned spins = 0;
        for (;;) {
            unsigned long long v = desc_make(DESC_PREFIX, epoch, 0);  // before tile 0: nothing
            if (p >= 0) v = ld_acquire(desc + p);
            const bool ready = (v >> 62) != 0 && ((uint32_t)(v >> 32) & 0x3fffffffu) == tag;
            const unsigned have = __ballot_sync(0xffffffffu, ready);
            const unsigned pref = __ballot_sync(0xffffffffu, ready && (v >> 62) == DESC_PREFIX);
            // the lanes up to the nearest prefix are needed, all of them without one
            const unsigned need = pref ? (pref ^ (pref - 1u)) : 0xffffffffu;
            const bool late = (have & need) != need;
            if (!late || ++spins >= LOOKBACK_SPIN_LIMIT) {
                const uint32_t sum =
                    __reduce_add_sync(0xffffffffu, (need & have) >> lane & 1u ? (uint32_t)v : 0u);
                if (lane == 0) {
                    sm.sum[ph][wid] = sum;
                    sm.found[ph][wid] = late ? 2u : pref ? 1u : 0u;
                }
                break;
            }
            if (spins > 64) __nanosleep(64);
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            excl += sm.sum[ph][w];
            if (sm.found[ph][w] == 2u) ok = false;
            if (sm.found[ph][w]) return excl;
        }
    }
}

// ---- launchers (defined in the kernel translation units) ----------------
bool sweep_supported(int layout, int dim, int L);
cudaError_t launch_init(const RunDev& d, cudaStream_t s);
cudaError_t launch_sweep(const RunDev& d, int nsweeps, int grid, cudaStream_t s);
int sweep_grid(const RunDev& d);
cudaError_t launch_tau(const RunDev& d, cudaStream_t s);
// the observables of the step that has been swept, and the next step's reweight
cudaError_t launch_obs_tau(const RunDev& d, int nsweeps, cudaStream_t s);
cudaError_t launch_resample(const RunDev& d, cudaStream_t s);
// Redistribution between virtual GPUs (pa_resample_begin / pa_resample_finish):
// the counts and scan alone, then the gather into a permuted slot order.
// Post-exchange slots [dst[q], dst[q+1]) take the pre-exchange slots starting
// at src[q].
constexpr int MAX_SEGMENTS = 1024;
struct SegList {
    uint32_t n;
    uint32_t dst[MAX_SEGMENTS + 1];
    uint32_t src[MAX_SEGMENTS];
};
cudaError_t launch_resample_scan(const RunDev& d, cudaStream_t s);
cudaError_t launch_remap_gather(const RunDev& d, const SegList& segs, cudaStream_t s);
cudaError_t launch_multinomial(const RunDev& d, cudaStream_t s);
cudaError_t launch_obs(const RunDev& d, int nsweeps, cudaStream_t s);
// specialised 2D ferromagnet, L = 64 or 128, packed (pa_sweep_l64.cu)
bool l64_applies(const RunDev& d);
int l64_block_warps(const RunDev& d);
int l64_grid(const RunDev& d);
cudaError_t launch_sweep_l64(const RunDev& d, int nsweeps, int grid, cudaStream_t s);
// The register kernels' generator alone (pa_bench_philox).
int philox_rate_threads();
cudaError_t launch_philox_rate(uint64_t seed, uint32_t halfsweeps, uint32_t* out, cudaStream_t s);
// batched forms (one launch for every run of a batch, or of one class)
cudaError_t launch_tau_batched(const BatchDev& b, cudaStream_t s);
cudaError_t launch_resample_batched(const BatchDev& b, cudaStream_t s);
cudaError_t launch_obs_batched(const BatchDev& b, cudaStream_t s);
// sweep of one class; `warps` selects the block shape (an autotuned knob: 2, 4
// or 8 for the replica-sliced kernel; the register kernels have one shape),
// grid: one wave of resident blocks
cudaError_t launch_sweep_batched(const BatchSweepArgs& a, const RunDev& proto, int warps, int grid,
                                 cudaStream_t s);
int batched_sweep_grid(const RunDev& proto, int warps);
bool batched_warps_valid(const RunDev& proto, int warps);
// the shape of the replica-sliced classes of a batch of these runs
int batched_default_warps(const RunDev* runs, int n);
bool l64_batched_applies(const RunDev& proto);
cudaError_t launch_sweep_l64_batched(const BatchSweepArgs& a, const RunDev& proto, int grid,
                                     cudaStream_t s);
int l64_batched_grid(const RunDev& proto);

// Resample tiles: RS_ITEMS consecutive replicas per thread, RS_THREADS threads.
#ifndef PA_RS_ITEMS
#define PA_RS_ITEMS 8
#endif
constexpr int RS_THREADS = 256;
constexpr int RS_ITEMS = PA_RS_ITEMS;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
// log2 of the slices of a run's tiles, in a launch that resamples `total` bytes
// of spins.  One CTA gathers at about 30 GB/s whatever else runs, so the launch
// needs its bytes spread over as many CTAs as the GPU holds (152 x 4); where
// there are fewer tiles, or tiles of more bytes than that, several CTAs count the
// whole of a tile (a microsecond or two) and each gather its slice, of at least
// 32 replicas and `least` bytes.  In a batch the bytes matter, not the tiles: with one
// slice width for all, a tile of L = 128 (2 KB per replica) held the launch up.
constexpr uint32_t RS_CTAS = 608;
inline uint32_t resample_slices(uint64_t stride, uint64_t total, uint64_t least) {
    uint64_t target = total / RS_CTAS;
    if (target < least) target = least;
    uint32_t lg = 0;
    while (((uint32_t)RS_TILE >> (lg + 1)) >= 32 && ((uint64_t)RS_TILE >> lg) * stride > target) ++lg;
    return lg;
}

// A replica's copies are written by one CTA as long as they are few.  With beta
// steps of twice the inverse of the energy's standard deviation (sqrt(dim N) at
// beta = 0) and more a few replicas get hundreds of copies and then most of the
// population: the CTAs that hold them leave all copies beyond the first
// SPREAD_FROM, in entries of SPREAD_COPIES, to k_spread, which shares the entries
// out to all CTAs.  Such runs have kernels of their own: the code for it costs
// every resample about a microsecond.
constexpr uint32_t SPREAD_FROM = 16, SPREAD_COPIES = 64;
inline bool many_copies(double largest_dbeta, double bonds) {
    return largest_dbeta * largest_dbeta * bonds > 4.0;
}

}  // namespace pa
