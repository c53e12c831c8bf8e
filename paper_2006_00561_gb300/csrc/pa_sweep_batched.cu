// pa_sweep_batched.cu -- the batched replica-sliced sweep kernels
// (pa_sliced.cuh): one launch for the runs of a class.
#include "pa_sliced.cuh"

namespace pa {
namespace {

// Batched: 32-slot chunks claimed from the class's slot space (run capacities
// are rounded up to 32, so a chunk never straddles two runs).  The run of
// chunk slot g, and its first slot in the class.
__device__ __forceinline__ uint32_t run_of(const BatchSweepArgs& a, uint32_t g, uint32_t& base) {
    uint32_t lo = 0, hi = a.n;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a.slot_base[mid] <= g) lo = mid;
        else hi = mid;
    }
    base = a.slot_base[lo];
    return a.run_ids[lo];
}

// Blocks that the register budget leaves room for on an SM: with the round keys
// in registers the compiler takes up to 128 of them, and the SM then holds half
// the warps of the plain kernel.  us of a batched sweep on GB300 with room for 512,
// 640, 768, 1024 threads: 24 spin glasses of three sizes 887, 851, 873, 883; 12 of
// L = 8 729, 723, 737, 755; 12 of L = 10 1530, 1480, 1483, 1502; 12 runs of 2D L = 16 618, 649,
// 633, 635; L = 32 2356, 2406, 2359, 2380; a serving batch 1772, 1802, 1829, 1900.
template <int DIM, int L, int RSP>
__host__ __device__ constexpr int resident() {
    constexpr int n = (DIM == 3 ? 640 : 512) / Team<DIM, L, RSP>::TT;
    return n < 1 ? 1 : n;
}
// Each team claims a chunk at a time and stages its run's round keys and
// coupling patterns.
template <int DIM, int L, bool PMJ, int RSP>
__global__ void __launch_bounds__(Team<DIM, L, RSP>::TT, resident<DIM, L, RSP>())
    k_sweep_team_batched(BatchSweepArgs a) {
    extern __shared__ uint4 smem[];
    __shared__ uint32_t s_chunk;
    constexpr int SQ = s_quads<DIM, L>();
    uint32_t* sums = reinterpret_cast<uint32_t*>(smem + 64);
    uint32_t* keys = reinterpret_cast<uint32_t*>(smem + 80);
    uint32_t* S = reinterpret_cast<uint32_t*>(smem + 86);
    uint8_t* JS = reinterpret_cast<uint8_t*>(smem + 86 + SQ);
    uint32_t have = 0xffffffffu;
    unsigned long long* accum = nullptr;
    long long sAbsM = 0, sM2 = 0;
    for (;;) {
        __syncthreads();  // s_chunk, keys and JS of the previous chunk are read by no one any more
        if (threadIdx.x == 0) s_chunk = atomicAdd(a.counter, 1u);
        __syncthreads();
        const uint32_t g = s_chunk * 32u;
        if (g >= a.total_slots) break;
        uint32_t base;
        const uint32_t run = run_of(a, g, base);
        const RunDev& d = a.runs[run];
        if (run != have) {
            if (accum && threadIdx.x < 32) flush_mag(accum, sAbsM, sM2, threadIdx.x);
            have = run;
            accum = d.accum;
            if (threadIdx.x < 10) {
                keys[threadIdx.x] = d.rk0[threadIdx.x];
                keys[10 + threadIdx.x] = d.rk1[threadIdx.x];
            }
            if constexpr (PMJ) couplings<DIM, L>(d, JS, threadIdx.x, Team<DIM, L, RSP>::TT);
            __syncthreads();
        }
        const SweepCtx x = sweep_ctx(d);
        const uint32_t b0 = g - base;
        if (b0 < x.R) {
            KeyRegs K;
#pragma unroll
            for (int r = 0; r < 10; ++r) {
                K.rk0[r] = keys[r];
                K.rk1[r] = keys[10 + r];
            }
            team_chunk<DIM, L, PMJ, RSP, 8>(d, x, b0, d.theta, S, smem, sums, JS, K, sAbsM, sM2);
        }
    }
    if (accum && threadIdx.x < 32) flush_mag(accum, sAbsM, sM2, threadIdx.x);
}

template <int DIM, int L, bool PMJ>
KInfo pick_batched(bool four) {
    constexpr int smem = (86 + s_quads<DIM, L>() + j_quads<DIM, L, PMJ>()) * 16;
    if constexpr (!always_four<DIM, L>())
        if (!four)
            return {(const void*)k_sweep_team_batched<DIM, L, PMJ, 1>, Team<DIM, L, 1>::TT, smem, 32};
    return {(const void*)k_sweep_team_batched<DIM, L, PMJ, 4>, Team<DIM, L, 4>::TT, smem, 32};
}

KInfo find_batched(int dim, int L, bool pmj, bool four) {
#define PA_CASE(D_, L_) \
    if (dim == D_ && L == L_) \
        return pmj ? pick_batched<D_, L_, true>(four) : pick_batched<D_, L_, false>(four);
    PA_SIZES(PA_CASE)
#undef PA_CASE
    return {nullptr, 0, 0, 0};
}

// The shape of a batched class: 8 "warps per block" are four lanes per group, 2
// and 4 one lane.
KInfo batched_kernel(const RunDev& d, int warps) {
    return find_batched(d.dim, d.L, d.model == PA_MODEL_PMJ, warps == 8);
}

}  // namespace

bool batched_warps_valid(const RunDev& proto, int warps) {
    return l64_batched_applies(proto) || warps == 2 || warps == 4 || warps == 8;
}

int batched_default_warps(const RunDev* runs, int n) {
    int64_t warps = 0;
    for (int i = 0; i < n; ++i) warps += one_lane_warps(runs[i]);
    return warps < FOUR_BELOW ? 8 : 4;
}

int batched_sweep_grid(const RunDev& proto, int warps) {
    if (l64_batched_applies(proto)) return l64_batched_grid(proto);
    return grid_for(batched_kernel(proto, warps), 0);
}

cudaError_t launch_sweep_batched(const BatchSweepArgs& a, const RunDev& proto, int warps, int grid,
                                 cudaStream_t s) {
    if (l64_batched_applies(proto)) return launch_sweep_l64_batched(a, proto, grid, s);
    const KInfo k = batched_kernel(proto, warps);
    if (!k.fn) return cudaErrorInvalidValue;
    BatchSweepArgs aa = a;
    void* args[] = {&aa};
    return cudaLaunchKernel(k.fn, dim3(grid), dim3(k.threads), args, (size_t)k.smem, s);
}

}  // namespace pa
