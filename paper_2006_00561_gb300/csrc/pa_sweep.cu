// pa_sweep.cu -- initial population, couplings, and the plain replica-sliced
// sweep kernels (pa_sliced.cuh) with the choice of their form.
#include <cmath>

#include "pa_sliced.cuh"

namespace pa {
namespace {

template <int DIM, int L, bool PMJ, int RSP, int RPQ>
__global__ void __launch_bounds__(Team<DIM, L, RSP>::TT)
    k_sweep_team(__grid_constant__ const RunDev d, int nsweeps) {
    extern __shared__ uint4 smem[];
    uint32_t* sums = reinterpret_cast<uint32_t*>(smem + 64);
    uint32_t* S = reinterpret_cast<uint32_t*>(smem + 80);
    uint8_t* JS = reinterpret_cast<uint8_t*>(smem + 80 + s_quads<DIM, L>());
    chain_wait();
    if constexpr (PMJ) couplings<DIM, L>(d, JS, threadIdx.x, Team<DIM, L, RSP>::TT);
    const SweepCtx x = sweep_ctx(d);
    const Keys K{d.rk0, d.rk1};
    long long sAbsM = 0, sM2 = 0;
    const uint32_t end = min(x.R, d.slot_hi);
    constexpr uint32_t C = 4u * RPQ;  // replicas of a chunk; slot_lo is a multiple of 32
    for (uint32_t ch = d.slot_lo / C + blockIdx.x; ch * C < end; ch += gridDim.x)
        team_chunk<DIM, L, PMJ, RSP, RPQ>(d, x, ch * C, nsweeps, S, smem, sums, JS, K, sAbsM, sM2);
    if (threadIdx.x < 32) flush_mag(d.accum, sAbsM, sM2, threadIdx.x);
}

// --------------------------------------------------------------------------
// Initial population (Sec. 2: uniform states at beta0 = 0, or the ground
// state for heating from near T = 0) and couplings.
// Site s of replica `slot` takes the top bit of word s & 3 of the Philox
// block (s >> 2, 0, slot, INIT | instance); set means spin -1.  Coupling of
// bond (s, d): top bit of word s & 3 of (s >> 2, d, 0, COUPLING | instance)
// under the coupling key; set means J = -1.
// --------------------------------------------------------------------------
// Packed rows of any even length: one thread per word and replica.
__global__ void k_init_packed(RunDev d, int NW) {
    const uint64_t gid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t total = (uint64_t)d.R0 * d.nwords;
    if (gid >= total) return;
    const uint32_t slot = (uint32_t)(gid / d.nwords);
    const uint32_t w = (uint32_t)(gid % d.nwords);
    const int r = (int)(w / NW), k = (int)(w % NW);
    const uint32_t ctr3 = (TAG_INIT << 28) | d.instance;
    const uint32_t k0 = (uint32_t)d.seed, k1 = (uint32_t)(d.seed >> 32);
    uint32_t bits = 0;
    int64_t cached = -1;
    uint4 u = make_uint4(0, 0, 0, 0);
    for (int b = 0; b < 32; ++b) {
        const int x = 32 * k + b;
        if (x >= d.L) break;
        const int64_t s = x + (int64_t)d.L * r;
        if ((s >> 2) != cached) {
            cached = s >> 2;
            u = philox((uint32_t)(s >> 2), 0u, slot, ctr3, k0, k1);
        }
        bits |= (pick(u, (uint32_t)(s & 3)) >> 31) << b;
    }
    reinterpret_cast<uint32_t*>(d.spins[0] + (size_t)slot * d.stride)[w] = bits;
}

// The same for rows that are whole Philox blocks (L a multiple of 4): a thread
// keeps one word of the replica, NB blocks, and walks over the replicas.  The
// block index enters word 0 and the slot word 2, so the products of rounds 1
// and 2 each belong to a block (held in registers over all replicas) or to a
// replica (two per word): a block costs 16 + 2 / NB multiplies instead of 20.
// Bound by them: the creation of a run of 2^21 replicas of L = 64, with its first
// measurement, takes 5.6 ms on GB300; with one thread per word and replica (a
// 64-bit division, and every product of every block) it took 13.6 ms.
template <int NB>
__global__ void __launch_bounds__(256) k_init_words(__grid_constant__ const RunDev d) {
    const uint32_t per = 256u / d.nwords;  // replicas of a block's pass (0: part of one)
    uint32_t w, first, step;
    if (per) {
        w = threadIdx.x % d.nwords;
        const uint32_t sub = threadIdx.x / d.nwords;
        if (sub >= per) return;
        first = blockIdx.x * per + sub;
        step = gridDim.x * per;
    } else {
        w = blockIdx.y * 256u + threadIdx.x;
        if (w >= d.nwords) return;
        first = blockIdx.x;
        step = gridDim.x;
    }
    const uint32_t ctr3 = (TAG_INIT << 28) | d.instance;
    uint32_t h2[NB], l2[NB], l1[NB];  // block halves: round 2 (high, low), round 1 (low)
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        uint32_t h1;
        mul_hilo(PM0, w * NB + (uint32_t)j, h1, l1[j]);
        mul_hilo(PM1, h1 ^ ctr3 ^ d.rk1[0], h2[j], l2[j]);
    }
    for (uint32_t slot = first; slot < d.R0; slot += step) {
        uint32_t hs, ls, hr, lr;  // replica halves
        mul_hilo(PM1, slot, hs, ls);            // round 1
        mul_hilo(PM0, hs ^ d.rk0[0], hr, lr);   // round 2
        uint32_t bits = 0;
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            uint32_t c0 = h2[j] ^ ls ^ d.rk0[1], c1 = l2[j], c2 = hr ^ l1[j] ^ d.rk1[1], c3 = lr;
#pragma unroll
            for (int r = 2; r < 10; ++r) {
                uint32_t hiA, loA, hiB, loB;
                mul_hilo(PM0, c0, hiA, loA);
                mul_hilo(PM1, c2, hiB, loB);
                c0 = hiB ^ c1 ^ d.rk0[r];
                c1 = loB;
                c2 = hiA ^ c3 ^ d.rk1[r];
                c3 = loA;
            }
            const uint32_t nib = (c0 >> 31) | (c1 >> 31) << 1 | (c2 >> 31) << 2 | (c3 >> 31) << 3;
            bits |= nib << (4 * j);
        }
        reinterpret_cast<uint32_t*>(d.spins[0] + (size_t)slot * d.stride)[w] = bits;
    }
}

__global__ void k_init_i8(RunDev d) {
    const uint64_t calls = (uint64_t)(d.N + 3) / 4;
    const uint64_t gid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (uint64_t)d.R0 * calls) return;
    const uint32_t slot = (uint32_t)(gid / calls);
    const uint32_t q = (uint32_t)(gid % calls);
    int8_t* dst = reinterpret_cast<int8_t*>(d.spins[0] + (size_t)slot * d.stride);
    if (d.init == PA_INIT_GROUND) {  // all spins +1
        for (int j = 0; j < 4; ++j) {
            const int64_t s = 4 * (int64_t)q + j;
            if (s < d.N) dst[s] = 1;
        }
        return;
    }
    const uint4 u = philox(q, 0u, slot, (TAG_INIT << 28) | d.instance, (uint32_t)d.seed,
                           (uint32_t)(d.seed >> 32));
    for (int j = 0; j < 4; ++j) {
        const int64_t s = 4 * (int64_t)q + j;
        if (s < d.N) dst[s] = (pick(u, (uint32_t)j) >> 31) ? (int8_t)-1 : (int8_t)1;
    }
}

__global__ void k_init_couplings(RunDev d, int NW) {
    const uint64_t gid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t ctr3 = (TAG_COUPLING << 28) | d.instance;
    const uint32_t k0 = (uint32_t)d.coupling_seed, k1 = (uint32_t)(d.coupling_seed >> 32);
    uint32_t neg = 0;
    if (d.layout == PA_LAYOUT_PACKED) {
        if (gid < (uint64_t)d.dim * d.nwords) {
            const int dd = (int)(gid / d.nwords);
            const uint32_t w = (uint32_t)(gid % d.nwords);
            const int r = (int)(w / NW), k = (int)(w % NW);
            uint32_t bits = 0;
            for (int b = 0; b < 32; ++b) {
                const int x = 32 * k + b;
                if (x >= d.L) break;
                const int64_t s = x + (int64_t)d.L * r;
                const uint4 u = philox((uint32_t)(s >> 2), (uint32_t)dd, 0u, ctr3, k0, k1);
                bits |= (pick(u, (uint32_t)(s & 3)) >> 31) << b;
            }
            d.jpk[gid] = bits;
            neg = __popc(bits);
        }
    } else {
        if (gid < (uint64_t)d.N * d.dim) {
            const int64_t s = (int64_t)(gid / d.dim);
            const int dd = (int)(gid % d.dim);
            const uint4 u = philox((uint32_t)(s >> 2), (uint32_t)dd, 0u, ctr3, k0, k1);
            const uint32_t bit = pick(u, (uint32_t)(s & 3)) >> 31;
            d.j8[gid] = bit ? (int8_t)-1 : (int8_t)1;
            neg = bit;
        }
    }
    neg = warp_sum_u32(neg);
    if ((threadIdx.x & 31) == 0 && neg) atomicAdd(&d.st->negbonds, neg);
}

// --------------------------------------------------------------------------
// dispatch
// --------------------------------------------------------------------------
// Forms of the plain kernel: one lane per group on chunks of 32 replicas, or
// four lanes on chunks of 32, 16 or 8.
enum Form { ONE_LANE, FOUR_32, FOUR_16, FOUR_8 };

template <int DIM, int L, bool PMJ>
KInfo pick_plain(Form f) {
    constexpr int smem = (80 + s_quads<DIM, L>() + j_quads<DIM, L, PMJ>()) * 16;
    constexpr int T4 = Team<DIM, L, 4>::TT;
    if constexpr (!always_four<DIM, L>())
        if (f == ONE_LANE)
            return {(const void*)k_sweep_team<DIM, L, PMJ, 1, 8>, Team<DIM, L, 1>::TT, smem, 32};
    if (f == FOUR_16) return {(const void*)k_sweep_team<DIM, L, PMJ, 4, 4>, T4, smem, 16};
    if (f == FOUR_8) return {(const void*)k_sweep_team<DIM, L, PMJ, 4, 2>, T4, smem, 8};
    return {(const void*)k_sweep_team<DIM, L, PMJ, 4, 8>, T4, smem, 32};
}

KInfo find_kernel(int dim, int L, bool pmj, Form f) {
#define PA_CASE(D_, L_) \
    if (dim == D_ && L == L_) \
        return pmj ? pick_plain<D_, L_, true>(f) : pick_plain<D_, L_, false>(f);
    PA_SIZES(PA_CASE)
#undef PA_CASE
    return {nullptr, 0, 0, 0};
}

// The population with room for its fluctuations (their variance is at most R0).
int64_t typical_population(const RunDev& d) {
    return (int64_t)d.R0 + (int64_t)(3.0 * std::sqrt((double)d.R0));
}

// One lane per group or four: four draw a group's 32 blocks in a quarter of
// the time, for more instructions.  One is the faster form once its warps (32
// groups of a chunk each) fill the GPU's 608 schedulers four deep.  Measured on
// GB300 (us per launch, one / four; warps of the one-lane form): 3D L = 8 96 / 86
// (1024), 2D L = 16 77 / 66 (938), 3D L = 10 158 / 158 (2048) and 971 / 1056 (16384), 2D L = 32
// 133 / 147 (18752), 3D L = 8 969 / 1079 (16384).
//
// Below that, chunks of 16 or 8 replicas bring more SMs to work where the
// chunks of 32 are fewer than the SMs, and a half-sweep is a shorter chain, for
// more work per replica (flips, barriers and group words serve fewer replicas).
// The time of a launch is about 8 us + k max(w, w0), w the warps of the chunks
// that share an SM, with k and w0 fitted to launches of theta = 10 on GB300; us per
// launch on chunks of 32 / 16 / 8, the taken form marked: 2D L = 16 1000 replicas 20.3 /
// 16.6 / 14.4*, 2500 20.4 / 18.4 / 17.5*, 5000 24.5 / 22.7* / 22.8, 10000 32.8* / 30.8 /
// 34.5; 3D L = 6 4099 22.8 / 20.2* / 24.4, 8000 28.9* / 32.5 / 36.7; 3D L = 10 1000 45.5 / 32.0 /
// 24.6*, 2000 45.8 / 32.1* / 39.5, 4096 46.2* / 53.4 / 71.6; 3D L = 16 1000 156 / 102 / 71*.
Form form_of(const RunDev& d, int sms) {
    if (one_lane_warps(d) >= FOUR_BELOW) return ONE_LANE;
    struct {
        Form f;
        int replicas;
        double k, w0;
    } const form[] = {{FOUR_32, 32, 2.2, 6.0}, {FOUR_16, 16, 1.45, 7.0}, {FOUR_8, 8, 0.95, 9.0}};
    const double team = (double)((d.N / 2 + 31) / 32);  // warps of a chunk: four lanes per group
    Form best = FOUR_32;
    double least = 1e30;
    for (const auto& f : form) {
        const int64_t chunks = (typical_population(d) + f.replicas - 1) / f.replicas;
        const double w = team * (double)((chunks + sms - 1) / sms);
        const double cost = f.k * (w > f.w0 ? w : f.w0);
        if (cost < least) {
            least = cost;
            best = f.f;
        }
    }
    return best;
}

int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return sms;
}

KInfo plain_kernel(const RunDev& d) {
    const int sms = sm_count();
    if (sms <= 0) return {nullptr, 0, 0, 0};
    return find_kernel(d.dim, d.L, d.model == PA_MODEL_PMJ, form_of(d, sms));
}

}  // namespace

bool sweep_supported(int layout, int dim, int L) {
    if (layout != PA_LAYOUT_INT8 && layout != PA_LAYOUT_PACKED) return false;
    return find_kernel(dim, L, false, FOUR_32).fn != nullptr;
}

int sweep_grid(const RunDev& d) {
    if (l64_applies(d)) return l64_grid(d);
    const KInfo k = plain_kernel(d);
    // blocks for the population as it usually is: blocks without a chunk would take
    // the places next to those with one
    return k.fn ? grid_for(k, (typical_population(d) + k.replicas - 1) / k.replicas) : 0;
}

cudaError_t launch_sweep(const RunDev& d, int nsweeps, int grid, cudaStream_t s) {
    if (l64_applies(d)) return launch_sweep_l64(d, nsweeps, grid, s);
    const KInfo k = plain_kernel(d);
    if (!k.fn) return cudaErrorInvalidValue;
    RunDev dd = d;
    int n = nsweeps;
    void* args[] = {&dd, &n};
    return launch_chained(k.fn, dim3(grid), dim3(k.threads), (size_t)k.smem, s, args);
}

// --------------------------------------------------------------------------
// dispatch
// --------------------------------------------------------------------------
cudaError_t launch_init(const RunDev& d, cudaStream_t s) {
    const int NW = (d.L + 31) / 32;
    if (d.model == PA_MODEL_PMJ) {
        const uint64_t n = d.layout == PA_LAYOUT_PACKED ? (uint64_t)d.dim * d.nwords
                                                        : (uint64_t)d.N * d.dim;
        k_init_couplings<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(d, NW);
    }
    if (d.layout == PA_LAYOUT_PACKED && d.init == PA_INIT_GROUND) {  // all spins +1
        const cudaError_t e = cudaMemsetAsync(d.spins[0], 0, (size_t)d.R0 * d.stride, s);
        if (e != cudaSuccess) return e;
    } else if (d.layout == PA_LAYOUT_PACKED && d.L % 4 == 0) {
        // about eight blocks of 256 threads per SM
        const uint32_t per = 256u / d.nwords, parts = per ? 1u : (d.nwords + 255u) / 256u;
        const uint32_t passes = per ? (d.R0 + per - 1) / per : d.R0, most = 1216u / parts;
        const dim3 grid(passes < most ? passes : most, parts);
        switch (d.L < 32 ? d.L / 4 : 8) {
            case 1: k_init_words<1><<<grid, 256, 0, s>>>(d); break;
            case 2: k_init_words<2><<<grid, 256, 0, s>>>(d); break;
            case 3: k_init_words<3><<<grid, 256, 0, s>>>(d); break;
            case 4: k_init_words<4><<<grid, 256, 0, s>>>(d); break;
            default: k_init_words<8><<<grid, 256, 0, s>>>(d); break;
        }
    } else if (d.layout == PA_LAYOUT_PACKED) {
        const uint64_t n = (uint64_t)d.R0 * d.nwords;
        k_init_packed<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(d, NW);
    } else {
        const uint64_t n = (uint64_t)d.R0 * ((d.N + 3) / 4);
        k_init_i8<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(d);
    }
    return cudaGetLastError();
}

}  // namespace pa
