// pa_resample.cu -- reweighting and resampling of the population (Sec. 2,
// Eq. 3 and Eq. 4) and the per-step observables (Sec. 2, Eq. 5).
//
//  k_tau       up to 33 CTAs: the energy histogram H of the population at beta_{i-1}
//              gives kref (lowest occupied level when cooling, highest when
//              heating), S = sum_k H_k D[|k - kref|] with D[j] =
//              exp(-|beta_i - beta_{i-1}| 4 j), Q = S exp(-dbeta E(kref)) / R
//              (Eq. 3) and the per-level weights tau_k = R0 D[|k - kref|] / S
//              (Eq. 4, renormalised to R0), kept as n_k = floor(tau_k),
//              F_k = floor(frac(tau_k) 2^32).
//  k_poisson_counts, k_mn_tile_sums, k_mn_cum, k_mn_draw
//              the copy counts of the Poisson and multinomial rules, ahead of the
//              scan.
//  k_resample  one pass over the population, one tile of RS_TILE replicas per
//              CTA (or per group of CTAs that share its gather): copy counts r_j = n_k + [u_j < F_k] (nearest-integer rule),
//              a single-pass exclusive scan with decoupled lookback across
//              tiles, and the gather of r_j exact copies of replica j into slots
//              o_j .. o_j + r_j - 1 of the other population buffer.
//  k_spread    in runs whose beta steps leave replicas with many copies: the
//              copies that k_resample's CTAs have left, shared out to all CTAs.
//  k_obs       one CTA: exact integer sums over the histogram and the
//              magnetisation accumulators, then the FP64 averages.
//  k_obs_tau   in a row of steps: k_obs of a step beside k_tau of the next.
//  k_gather, k_remap  the copies in the slot order of a redistribution.
//
// Floating point: IEEE double with explicit _rn intrinsics (no contraction),
// summed in a fixed order, so the tables are the same bits as any other
// implementation of the same order; log() only feeds ln Q, never a decision.
#include "pa_internal.cuh"

namespace pa {
namespace {

// The batched kernels stage a run's descriptor in shared memory (PA_RS_STAGE
// = 1): read from global memory, its fields could alias the kernel's own
// global stores, so the compiler would reload them after every store.
#ifndef PA_RS_STAGE
#define PA_RS_STAGE 1
#endif
static_assert(sizeof(RunDev) % 4 == 0, "RunDev is copied in 32-bit words");

// Copies *src into the shared descriptor dst with all threads of the CTA; the
// caller synchronises before reading it.
__device__ __forceinline__ void stage_run(const RunDev* src, RunDev& dst) {
    const uint32_t* from = reinterpret_cast<const uint32_t*>(src);
    uint32_t* to = reinterpret_cast<uint32_t*>(&dst);
    for (uint32_t w = threadIdx.x; w < sizeof(RunDev) / 4; w += blockDim.x) to[w] = from[w];
}

// Calls f(k, H_k) for the occupied levels of the thread's share of the
// histogram (four consecutive levels of every 4 * 256), eight 16-byte loads at a
// time before their conditions.
template <typename F>
__device__ __forceinline__ void each_level(const uint32_t* hist, uint32_t bins, F&& f) {
    const uint4* h4 = reinterpret_cast<const uint4*>(hist);  // 16-byte aligned
    const uint32_t quads = bins >> 2;
    const uint32_t kt = 4 * quads + threadIdx.x;
    const uint32_t tail = kt < bins ? hist[kt] : 0u;
    for (uint32_t q0 = threadIdx.x; q0 < quads; q0 += 8 * 256) {
        uint4 h[8];
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j) {
            const uint32_t q = q0 + 256 * j;
            h[j] = q < quads ? h4[q] : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j) {
            if ((h[j].x | h[j].y | h[j].z | h[j].w) == 0u) continue;
            const uint32_t k = 4 * (q0 + 256 * j);
            if (h[j].x) f(k, h[j].x);
            if (h[j].y) f(k + 1, h[j].y);
            if (h[j].z) f(k + 2, h[j].z);
            if (h[j].w) f(k + 3, h[j].w);
        }
    }
    if (tail) f(kt, tail);
}

// Reweight of one run by nblk 256-thread CTAs.  Every CTA finds kref and S
// itself (the same fixed order, so the same bits) and writes the tau entries
// of its share of the levels; the last CTA to finish, when every CTA has read
// the step index and R, advances the run's scalars.  Returns whether this CTA
// is the one that was last to read the histogram.
//
// Bound: an FP64 operation takes some 140 cycles on GB300 and a division 1450, so
// the time is the chain of FP64 operations.  Hence the products H_k D are
// formed by all threads ahead of the chunks' sums, levels without replicas add
// nothing (x + 0 * D is x, exactly) and are skipped, one warp alone adds up the
// chunk sums, levels whose tau is below 2^-33 get (0, 0) without a division, n and
// F are cut from the bits of tau, and the logarithms run in a warp of their own
// beside the divisions.  us, timed by events around the launch, with FP64 work on
// every level -> so: 13.4 -> 10.3 (257 levels), 25 -> 12.2 (4097), 44 -> 17 (16385); a batch
// of 28 runs with up to 16385 levels 87 -> 24.
constexpr uint32_t TAU_LEVELS = 128;  // levels per CTA and pass
// Levels whose products a CTA holds at a time (any more are added in further
// passes over the occupied range).
constexpr uint32_t TAU_HELD = 2048;

// floor(x) and floor(2^32 frac(x)) of x >= 0 (exact: both are bits of x);
// floor saturates at 2^32 - 1.
__device__ __forceinline__ void split32(double x, uint32_t& n, uint32_t& F) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(bits >> 52) - 1023;  // x >= 0: no sign
    const unsigned long long m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;  // x = m 2^(e - 52)
    n = F = 0;
    if (e >= 32) {
        if (e == 1024 && m != 0x10000000000000ull) return;  // not a number: (0, 0)
        n = 0xffffffffu;
        if (e < 52) F = (uint32_t)(((m << (e + 12)) >> 32));
    } else if (e >= 0) {
        n = (uint32_t)(m >> (52 - e));
        F = (uint32_t)((m << (e + 12)) >> 32);
    } else if (e >= -32) {
        F = (uint32_t)(m >> (20 - e));
    }
}
// CTAs of a run at most: 33, 65 and 130 ran alike on GB300 (14.7 us at 4097
// levels, 24 us at 16385, before the products were formed by all threads).
#ifndef PA_TAU_CTAS
#define PA_TAU_CTAS 33
#endif
constexpr uint32_t TAU_CTAS = PA_TAU_CTAS;
__device__ __forceinline__ TauNext* tau_next(const RunDev& d) {
    return reinterpret_cast<TauNext*>(reinterpret_cast<uint8_t*>(d.st) + 128);
}

// The run's scalars after the reweight of step i, by one thread, once every block
// has read the old ones.
__device__ __forceinline__ void tau_advance(DevState* st, uint32_t i, uint32_t R, uint32_t cur,
                                            uint32_t epoch, uint32_t kref) {
    st->tau_done = 0;
    st->kref = kref;
    st->step = i;
    st->R_prev = R;
    st->epoch = epoch + 1;
    st->tile_counter = 0;
    st->over_n = 0;
    st->src = cur;
    st->cur = cur ^ 1u;
    st->active = 1;
}
__device__ __forceinline__ void tau_advance_next(const RunDev& d, uint32_t i, uint32_t R, uint32_t cur,
                                                 uint32_t epoch) {
    const TauNext* nx = tau_next(d);
    DevState* st = d.st;
    st->lnQ = __ldcg(&nx->lnQ);
    st->lnZ = __ldcg(&nx->lnZ);
    st->S = __ldcg(&nx->S);
    tau_advance(st, i, R, cur, epoch, __ldcg(&nx->kref));
}

// WITH_OBS: one more block of the launch takes the observables of the step
// before, which read ln Q and ln Z: the new ones wait in TauNext.
template <bool WITH_OBS>
__device__ __forceinline__ bool tau_run(const RunDev& d, uint32_t blk, uint32_t nblk) {
    DevState* st = d.st;
    __shared__ double s_prod[TAU_HELD];
    __shared__ double s_part[8];
    __shared__ double s_S;
    __shared__ uint32_t s_min[8], s_max[8];
    __shared__ unsigned long long s_sum;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const uint32_t i = st->step + 1;
    const uint32_t R = st->R, cur = st->cur, epoch = st->epoch, negbonds = st->negbonds;
    const double lnZ = st->lnZ;
    const uint32_t bins = (uint32_t)d.bins;
    if (i > (uint32_t)d.K || R == 0) {
        if (t == 0 && blk == 0) {
            st->active = 0;
            atomicOr(&st->status, i > (uint32_t)d.K ? ST_DONE : ST_EMPTY);
        }
        return blk == 0;
    }
    const double db = d.dbeta[i];
    const double* D = d.dtab + (size_t)d.dsel[i] * bins;
    // reference level: lowest occupied when cooling, highest when heating
    const bool heating = db < 0.0;
    if (t == 0) s_sum = 0;
    uint32_t kmin = 0xffffffffu, kmax = 0u;
    unsigned long long hs = 0;
    each_level(d.hist, bins, [&](uint32_t k, uint32_t h) {
        kmin = min(kmin, k);
        kmax = max(kmax, k);
        hs += h;
    });
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) {
        s_min[wid] = kmin;
        s_max[wid] = kmax;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        kmin = min(kmin, s_min[w]);
        kmax = max(kmax, s_max[w]);
    }
    const uint32_t kref = heating ? kmax : kmin;
    const bool logs = blk == nblk - 1;  // this CTA also takes ln Q and the check of sum H
    if (logs && hs) atomicAdd(&s_sum, hs);
    // S in the fixed order: 256 contiguous chunks summed left to right, then a
    // pairwise tree over the chunk sums; level k weighs D[|k - kref|].
    const uint32_t ch = (bins + 255) / 256;
    const uint32_t k_lo = max(t * ch, kmin), k_hi = min(min((t + 1) * ch, bins), kmax + 1u);
    double acc = 0.0;
    for (uint32_t b0 = kmin; b0 <= kmax; b0 += TAU_HELD) {  // kmin > kmax: no replicas
        const uint32_t b1 = min(b0 + TAU_HELD, kmax + 1u);
        for (uint32_t k = b0 + t; k < b1; k += 256) {
            const uint32_t h = d.hist[k];
            s_prod[k - b0] = h ? __dmul_rn((double)h, D[heating ? kref - k : k - kref]) : -1.0;
        }
        __syncthreads();
        const uint32_t lo = max(k_lo, b0), hi = min(k_hi, b1);
        for (uint32_t k = lo; k < hi; ++k) {
            const double p = s_prod[k - b0];
            if (__double_as_longlong(p) >= 0) acc = __dadd_rn(acc, p);
        }
        __syncthreads();
    }
    if (__any_sync(0xffffffffu, __double_as_longlong(acc) != 0)) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) acc = __dadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, o));
    }
    if (lane == 0) s_part[wid] = acc;
    __syncthreads();
    if (wid == 0) {
        double v = s_part[lane & 7];
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (lane == 0) s_S = v;
    }
    __syncthreads();
    const double S = s_S;
    if (wid < 4) {
        const double R0d = (double)d.R0;
        const long long least =  // 2^-34 S: tau < 2^-33 (positive doubles order like their bits)
            __double_as_longlong(__dmul_rn(S, 5.8207660913467407e-11));
        for (uint32_t k = blk * TAU_LEVELS + t; k < bins; k += nblk * TAU_LEVELS) {
            uint32_t n = 0, F = 0;
            const int64_t j = heating ? (int64_t)kref - (int64_t)k : (int64_t)k - (int64_t)kref;
            if (j >= 0) {
                const double w = __dmul_rn(R0d, D[j]);
                if (__double_as_longlong(w) >= least) split32(__ddiv_rn(w, S), n, F);
            }
            d.tab_n[k] = n;
            d.tab_F[k] = F;
        }
    } else if (logs && wid == 4) {
        const double ln = log(lane == 1 ? (double)R : S);  // both logarithms at once
        const double lnR = __shfl_sync(0xffffffffu, ln, 1);
        if (lane == 0) {
            if (s_sum != (unsigned long long)R) atomicOr(&st->status, ST_INVARIANT);
            const long long Eref =
                2 * (2 * (long long)kref + (long long)(negbonds & 1u)) - (long long)d.dim * d.N;
            const double lnQ = __dsub_rn(__dsub_rn(ln, lnR), __dmul_rn(db, (double)Eref));
            if constexpr (WITH_OBS) {
                *tau_next(d) = TauNext{lnQ, __dadd_rn(lnZ, lnQ), S, kref};
            } else {
                st->lnQ = lnQ;
                st->lnZ = __dadd_rn(lnZ, lnQ);
                st->S = S;
            }
        }
    }
    const uint32_t arrivals = nblk + (WITH_OBS ? 1u : 0u);
    if (arrivals > 1) {
        __shared__ bool s_last;
        __syncthreads();
        if (t == 0) {
            __threadfence();
            s_last = atomicAdd(&st->tau_done, 1ull) == (unsigned long long)(arrivals - 1);
            if (WITH_OBS) __threadfence();
        }
        __syncthreads();
        if (!s_last) return false;
    }
    if (t == 0) {
        if constexpr (WITH_OBS) tau_advance_next(d, i, R, cur, epoch);
        else tau_advance(st, i, R, cur, epoch, kref);
    }
    return true;
}

__global__ void __launch_bounds__(256) k_tau(__grid_constant__ const RunDev d) {
    chain_wait();
    tau_run<false>(d, blockIdx.x, gridDim.x);
}

// CTAs of a run's reweight: one per TAU_LEVELS levels, at most TAU_CTAS.
__host__ __device__ inline uint32_t tau_ctas(int64_t bins) {
    const int64_t per = (bins + TAU_LEVELS - 1) / TAU_LEVELS;
    return per < 1 ? 1u : per < (int64_t)TAU_CTAS ? (uint32_t)per : TAU_CTAS;
}

// Batched reweight: column r of the grid handles run r, whose last CTA then clears
// the run's histogram and magnetisation sums for the coming sweep (the
// reweight is their last reader); the first CTA clears the batch's work
// counters.
__global__ void __launch_bounds__(256) k_tau_batched(BatchDev b) {
    if (blockIdx.x == 0 && blockIdx.y == 0)
        for (uint32_t c = threadIdx.x; c < b.ncounters; c += 256) b.counters[c] = 0u;
    const uint32_t nblk = tau_ctas(b.runs[blockIdx.x].bins);
    if (blockIdx.y >= nblk) return;
    __shared__ RunDev s_d;
    stage_run(&b.runs[blockIdx.x], s_d);
    __syncthreads();
    const RunDev& d = s_d;
    if (!tau_run<false>(d, blockIdx.y, nblk)) return;
    __syncthreads();
    for (uint32_t k = threadIdx.x; k < (uint32_t)d.bins; k += blockDim.x) d.hist[k] = 0u;
    if (threadIdx.x < 2) d.accum[threadIdx.x] = 0ull;
}

// The gather walks only the tile's surviving replicas (count > 0), listed in
// order, so that every 16-byte item a thread takes has a load behind it.
struct ResampleSmem {
    // survivor j of this CTA's slice: tile index, count, first slot
    uint32_t surv[RS_TILE], r[RS_TILE], o[RS_TILE];
    uint32_t warp_nz[RS_THREADS / 32];  // survivors of each warp
    uint32_t warp[RS_THREADS / 32];
    uint32_t tile;
    LookSmem<RS_THREADS / 32> look;
};

// 16-byte loads in flight per thread in the gather, within the 64 registers of
// four CTAs per SM (only the data stays in registers between the loads and the
// stores).  Measured on GB300, us per launch: 2^21 replicas of 512 bytes 346 (4),
// 347 (6), 348 (8; 12 at 3 CTAs per SM 365; 4 at 5 CTAs 367); 24 spin-glass runs
// of 2^15..2^16 in one launch 112 (4), 117 (6), 122 (8).  346 us are 6.1 TB/s over the
// exact bytes, 0.90 of the measured copy peak: HBM bounds it.
#ifndef PA_RS_GU
#define PA_RS_GU 4
#endif

// Poisson(tau_k) copy count of replica i (Sec. 2), tau_k = n + F / 2^32: the
// event count of a unit-rate Poisson process on [0, tau_k].  The fractional
// interval contributes a Poisson(1) count thinned with keep probability
// F / 2^32, each unit interval a Poisson(1) count, every one drawn by
// inversion against the 32-bit thresholds p1.  Uniforms: words of the Philox
// blocks (i, step, b, POISSON|id), b = 0, 1, ..., consumed in that order.
// A level with n above the capacity overflows whatever the draw: its count is
// then n itself, which the capacity check rejects, instead of n draws.
__device__ __noinline__ uint32_t poisson_count(const RunDev& d, uint32_t i, uint32_t step,
                                               uint32_t n, uint32_t F) {
    if (n > d.cap) return n;
    const uint32_t ctr3 = (TAG_POISSON << 28) | d.instance;
    const uint32_t k0 = (uint32_t)d.seed, k1 = (uint32_t)(d.seed >> 32);
    uint4 blk = philox(i, step, 0u, ctr3, k0, k1);
    uint32_t b = 1, w = 0;
    auto next = [&]() -> uint32_t {
        if (w == 4) {
            blk = philox(i, step, b, ctr3, k0, k1);
            ++b;
            w = 0;
        }
        return pick(blk, w++);
    };
    auto unit = [&]() -> uint32_t {
        const uint32_t u = next();
        uint32_t m = 0;
        while (m < d.p1_len && u >= d.p1[m]) ++m;
        return m;
    };
    uint32_t count = 0;
    const uint32_t events = unit();
    for (uint32_t e = 0; e < events; ++e) count += next() < F ? 1u : 0u;
    for (uint32_t j = 0; j < n; ++j) count += unit();
    return count;
}

// Poisson copy counts, one replica per thread: a draw is two or three Philox
// blocks and a table walk one after the other, so they run over the whole GPU
// ahead of the scan instead of eight after another in a tile's threads.  The
// Poisson resample of 2^21 replicas (L = 64) takes 333 us with it on GB300 against
// 407 with the draws inside the scan kernel, at 89 registers.
__device__ __forceinline__ void poisson_counts(const RunDev& d, uint32_t first, uint32_t stride,
                                               uint32_t end) {
    const uint32_t step = d.st->step;
    const uint32_t* eb = d.ebin[d.st->src];
    for (uint32_t i = first; i < end; i += stride) {
        const uint32_t k = eb[i];
        d.counts[i] = poisson_count(d, i, step, d.tab_n[k], d.tab_F[k]);
    }
}

__global__ void __launch_bounds__(256) k_poisson_counts(__grid_constant__ const RunDev d) {
    chain_wait();
    if (!d.st->active) return;
    poisson_counts(d, blockIdx.x * 256u + threadIdx.x, gridDim.x * 256u, d.st->R_prev);
}

// Batched: CTA g takes slice g of the batch, if its run is on the rule.
__global__ void __launch_bounds__(RS_THREADS) k_poisson_counts_batched(BatchDev b) {
    __shared__ RunDev s_d;
    const uint32_t g = blockIdx.x;
    uint32_t lo = 0, hi = b.nruns;  // tile_base[lo] <= g < tile_base[hi]
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (b.tile_base[mid] <= g) lo = mid;
        else hi = mid;
    }
    if (b.runs[lo].resample != PA_RESAMPLE_POISSON || !b.runs[lo].st->active) return;
    stage_run(&b.runs[lo], s_d);
    __syncthreads();
    const uint32_t width = (uint32_t)RS_TILE >> s_d.slice_lg;
    const uint32_t base = (g - b.tile_base[lo]) * width, R = s_d.st->R_prev;
    if (base < R) poisson_counts(s_d, base + threadIdx.x, RS_THREADS, min(R, base + width));
}

// Entries of k_spread: {source replica, first slot, copies}, at most
// SPREAD_COPIES copies each.  Copies beyond the capacity are dropped here as they
// are everywhere; what is left fits the list (one entry per 17 copies at least).
__device__ __forceinline__ void leave_copies(const RunDev& d, uint32_t src, uint32_t dst, uint32_t n) {
    if (dst >= d.cap) return;
    n = min(n, d.cap - dst);
    const uint32_t m = (n + SPREAD_COPIES - 1) / SPREAD_COPIES, room = d.cap_alloc / 3u;
    const uint32_t e0 = atomicAdd(&d.st->over_n, m);
    for (uint32_t e = 0; e < m && e0 + e < room; ++e) {
        uint32_t* at = d.srcmap2 + 3 * (size_t)(e0 + e);
        at[0] = src;
        at[1] = dst + e * SPREAD_COPIES;
        at[2] = min(SPREAD_COPIES, n - e * SPREAD_COPIES);
    }
}

// The copies that the resample's CTAs have left: blk of nblk CTAs takes entries
// blk, blk + nblk, ...  Measured on GB300: the batched resample of a serving batch
// (163 000 replicas, beta steps up to seven standard deviations of the energy at L =
// 128) takes 35 us with it and 115 without, when one CTA wrote thousands of copies of a
// replica.
__device__ __forceinline__ void spread_run(const RunDev& d, uint32_t blk, uint32_t nblk) {
    const DevState* st = d.st;
    const uint32_t n = min(st->over_n, d.cap_alloc / 3u), src = st->src;
    const uint32_t CH = d.stride >> 4;
    for (uint32_t e = blk; e < n; e += nblk) {
        const uint32_t* at = d.srcmap2 + 3 * (size_t)e;
        const uint32_t rep = at[0], dst = at[1], copies = at[2];
        const uint4* from = reinterpret_cast<const uint4*>(d.spins[src]) + (size_t)rep * CH;
        uint4* to = reinterpret_cast<uint4*>(d.spins[src ^ 1u]) + (size_t)dst * CH;
        for (uint32_t it = threadIdx.x; it < copies * CH; it += 256) __stcs(to + it, __ldcg(from + it % CH));
        const uint32_t level = d.ebin[src][rep];
        const int32_t mag = d.mag[src][rep];
        for (uint32_t k = threadIdx.x; k < copies; k += 256) {
            d.ebin[src ^ 1u][dst + k] = level;
            d.mag[src ^ 1u][dst + k] = mag;
        }
    }
}

__global__ void __launch_bounds__(256) k_spread(__grid_constant__ const RunDev d) {
    chain_wait();
    if (d.st->active) spread_run(d, blockIdx.x, gridDim.x);
}

// Batched: column r of the grid serves run r.
__global__ void __launch_bounds__(256) k_spread_batched(BatchDev b) {
    const RunDev& d = b.runs[blockIdx.x];
    if (d.st->active && d.st->over_n) spread_run(d, blockIdx.y, gridDim.y);
}

// RULE 0 compiles the nearest-integer rule alone (the register budget of the
// HBM-bound default path); 2 takes the counts that the Poisson or multinomial
// draws have left in d.counts; 3 chooses between the two per run (batches).
//
// Counts, scan and gather of tile `tile` of one run (all threads of the CTA), or
// its slice of them.  SPLIT = false: the tile also gathers its replicas' spins.
// SPLIT = true: the tile writes, for each slot it fills, the index of the
// source replica (srcmap) with the copied energy level and magnetisation, and
// k_gather copies the spins afterwards over the whole new population (the
// redistribution's form).  SPREAD: copies beyond SPREAD_FROM are left to k_spread.
template <int RULE, bool SPLIT, bool SPREAD>
__device__ __forceinline__ void resample_tile(const RunDev& d, uint32_t tile, uint32_t slice,
                                              ResampleSmem& sm) {
    DevState* st = d.st;
    uint32_t* s_warp = sm.warp;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const uint32_t R = st->R_prev, epoch = st->epoch, src = st->src, step = st->step;
    const uint32_t base = tile * RS_TILE;
    // every CTA of a tile counts all of it; this one keeps slice [lo, hi)
    const uint32_t width = (uint32_t)RS_TILE >> d.slice_lg;
    const uint32_t lo = base + slice * width;
    if (lo >= R) return;
    const uint32_t end = min(R, base + (uint32_t)RS_TILE), hi = min(R, lo + width);
    // copy counts, RS_ITEMS consecutive replicas per thread
    const uint32_t* eb = d.ebin[src];
    const uint32_t ctr3 = (TAG_RESAMPLE << 28) | d.instance;
    const uint32_t k0 = (uint32_t)d.seed, k1 = (uint32_t)(d.seed >> 32);
    uint32_t r[RS_ITEMS];
    uint32_t sum = 0;
    const bool drawn = RULE == 2 || (RULE == 3 && d.resample != PA_RESAMPLE_NEAREST);
    if (drawn) {
#pragma unroll
        for (int j = 0; j < RS_ITEMS; ++j) {
            const uint32_t i = base + (uint32_t)t * RS_ITEMS + j;
            const uint32_t v = i < end ? d.counts[i] : 0u;
            r[j] = v;
            sum += v;
        }
    } else
#pragma unroll
    for (int j0 = 0; j0 < RS_ITEMS; j0 += 4) {
        const uint32_t i0 = base + (uint32_t)t * RS_ITEMS + j0;
        uint4 u = make_uint4(0, 0, 0, 0);
        uint32_t lev[4] = {0, 0, 0, 0};
        if (i0 < end) u = philox(i0 >> 2, step, 0u, ctr3, k0, k1);
        if (i0 + 4 <= end) {  // i0 is a multiple of 4: one 16-byte load
            const uint4 e4 = *reinterpret_cast<const uint4*>(eb + i0);
            lev[0] = e4.x, lev[1] = e4.y, lev[2] = e4.z, lev[3] = e4.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j < end) lev[j] = eb[i0 + j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t v = 0;
            if (i0 + j < end) {
                const uint32_t k = lev[j];
                v = d.tab_n[k] + (pick(u, (uint32_t)j) < d.tab_F[k] ? 1u : 0u);
            }
            r[j0 + j] = v;
            sum += v;
        }
    }
    const uint32_t i_first = base + (uint32_t)t * RS_ITEMS;
    const bool mine = i_first >= lo && i_first < hi;  // a slice holds whole threads
    // block-wide exclusive scan of the per-thread sums
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[wid] = incl;
    // and of the per-thread survivor counts
    uint32_t nz = 0;
#pragma unroll
    for (int j = 0; j < RS_ITEMS; ++j) nz += r[j] ? 1u : 0u;
    if (!mine) nz = 0;
    uint32_t nzi = nz;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, nzi, o);
        if (lane >= o) nzi += y;
    }
    if (lane == 31) sm.warp_nz[wid] = nzi;
    __syncthreads();
    uint32_t before = 0, total = 0;  // counts of the warps before this one, of the tile
    uint32_t before_nz = 0, nsurv = 0;
#pragma unroll
    for (int w = 0; w < RS_THREADS / 32; ++w) {
        if (w == wid) before = total;
        total += s_warp[w];
        if (w == wid) before_nz = nsurv;
        nsurv += sm.warp_nz[w];
    }
    uint32_t excl = 0;
    if (tile == 0) {
        // the test hook withholds tile 0's prefix, so that the bounded waits of
        // the tiles after it run out (PA_DEBUG_WITHHOLD_PREFIX)
        if (t == 0 && slice == 0 && !(d.debug & PA_DEBUG_WITHHOLD_PREFIX))
            st_release(&d.desc[0], desc_make(DESC_PREFIX, epoch, total));
    } else {
        // slice 0 speaks for the tile: it is claimed first
        if (t == 0 && slice == 0) st_release(&d.desc[tile], desc_make(DESC_AGG, epoch, total));
        bool ok;
        excl = lookback(d.desc, tile, epoch, sm.look, ok);
        if (t == 0) {
            if (!ok) atomicOr(&st->status, ST_TIMEOUT);
            if (slice == 0) st_release(&d.desc[tile], desc_make(DESC_PREFIX, epoch, excl + total));
        }
    }
    uint32_t o = excl + before + (incl - sum);
    uint32_t p = before_nz + (nzi - nz);
    if (mine)
#pragma unroll
    for (int j0 = 0; j0 < RS_ITEMS; j0 += 4) {
        const uint32_t li0 = (uint32_t)t * RS_ITEMS + j0;
        const uint32_t i0 = base + li0;
        uint32_t oo[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            oo[j] = o;
            o += r[j0 + j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t c = r[j0 + j];
            if (c) {  // 0 beyond R
                if (SPREAD && c > SPREAD_FROM) {
                    leave_copies(d, i0 + j, oo[j] + SPREAD_FROM, c - SPREAD_FROM);
                    c = SPREAD_FROM;
                }
                sm.surv[p] = li0 + j;
                sm.r[p] = c;
                sm.o[p++] = oo[j];
            }
        }
        if (i0 + 4 <= end) {  // i0 is a multiple of 4: 16-byte stores
            const uint4 r4 = make_uint4(r[j0], r[j0 + 1], r[j0 + 2], r[j0 + 3]);
            const uint4 o4 = make_uint4(oo[0], oo[1], oo[2], oo[3]);
            if (!drawn) *reinterpret_cast<uint4*>(d.counts + i0) = r4;
            *reinterpret_cast<uint4*>(d.offsets + i0) = o4;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (i0 + j < end) {
                    if (!drawn) d.counts[i0 + j] = r[j0 + j];
                    d.offsets[i0 + j] = oo[j];
                }
            }
        }
        if (i0 < R && R - 1 - i0 < 4) {  // the population's last replica
            if (o > d.cap) atomicOr(&st->status, ST_CAPACITY);
            if (o == 0) atomicOr(&st->status, ST_EMPTY);
            st->R = o > d.cap ? d.cap : o;
        }
    }
    __syncthreads();
    if (t == 0) atomicAdd(&st->sources, (unsigned long long)nsurv);

    // gather: 16-byte chunks, consecutive threads on consecutive chunks; GU
    // independent loads in flight per thread before their stores, whose
    // survivor is looked up again (shared memory) rather than kept in registers
    if (!SPLIT) {
        constexpr int GU = PA_RS_GU;
        const uint32_t CH = d.stride >> 4;
        // it / CH for it < RS_TILE * CH: the product with ceil(2^32 / CH) is exact
        // while it * CH < 2^32 (CH <= 1024)
        const uint32_t recip = CH > 1 ? 0xffffffffu / CH + 1u : 0u;
        const uint4* srcp = reinterpret_cast<const uint4*>(d.spins[src]) + (size_t)base * CH;
        uint4* dstp = reinterpret_cast<uint4*>(d.spins[src ^ 1u]);
        const uint32_t items = nsurv * CH;
        for (uint32_t it0 = t; it0 < items; it0 += RS_THREADS * GU) {
            uint4 v[GU];
#pragma unroll
            for (int u = 0; u < GU; ++u) {
                const uint32_t it = it0 + (uint32_t)u * RS_THREADS;
                if (it < items) {
                    const uint32_t jl = recip ? __umulhi(it, recip) : it;
                    v[u] = __ldcg(srcp + (size_t)sm.surv[jl] * CH + (it - jl * CH));
                }
            }
#pragma unroll
            for (int u = 0; u < GU; ++u) {
                const uint32_t it = it0 + (uint32_t)u * RS_THREADS;
                if (it < items) {
                    const uint32_t jl = recip ? __umulhi(it, recip) : it;
                    const uint32_t rr = sm.r[jl], d0 = sm.o[jl], c = it - jl * CH;
                    for (uint32_t k = 0; k < rr; ++k) {
                        const uint32_t dst = d0 + k;
                        if (dst < d.cap) __stcs(dstp + (size_t)dst * CH + c, v[u]);
                    }
                }
            }
        }
    }
    const uint32_t* esrc = d.ebin[src] + base;
    const int32_t* msrc = d.mag[src] + base;
    uint32_t* edst = d.ebin[src ^ 1u];
    int32_t* mdst = d.mag[src ^ 1u];
    for (uint32_t jl = t; jl < nsurv; jl += RS_THREADS) {
        const uint32_t li = sm.surv[jl], rr = sm.r[jl], d0 = sm.o[jl];
        const uint32_t e = esrc[li];
        const int32_t m = msrc[li];
        for (uint32_t k = 0; k < rr; ++k) {
            const uint32_t dst = d0 + k;
            if (dst < d.cap) {
                edst[dst] = e;
                mdst[dst] = m;
                if (SPLIT) d.srcmap[dst] = base + li;
            }
        }
    }
}

// Persistent: one wave of CTAs, each claiming slices of tiles until none is
// left.  Claims come in increasing order, so a tile's lookback only waits on
// tiles whose first slice is already claimed by a running CTA.  Measured on
// GB300 (us per launch, one CTA per tile and a lookback by one thread -> slices
// and the block-wide lookback): 20480 replicas at L = 64 (12 tiles) 77 -> 13.7,
// 5001 at L = 128 (4 tiles) 243 -> 14.9, 150001 at L = 32 (77 tiles) 38 -> 20,
// 1000 at L = 16 29 -> 8.5, 2^21 at L = 64 (1036 tiles, no slices) 362 -> 346.
// Resident CTAs per SM the register budget is sized for.
#ifndef PA_RS_MINB
#define PA_RS_MINB 4
#endif
template <int RULE, bool SPLIT, bool SPREAD>
__global__ void __launch_bounds__(RS_THREADS, PA_RS_MINB) k_resample(__grid_constant__ const RunDev d) {
    __shared__ ResampleSmem sm;
    chain_wait();
    if (threadIdx.x == 0) sm.tile = atomicAdd(&d.st->tile_counter, 1u);
    const bool active = d.st->active != 0;
    const uint32_t R = d.st->R_prev;
    if (d.clear_hist) {  // the reweight was their last reader
        uint32_t* acc = reinterpret_cast<uint32_t*>(d.accum);  // accum, then the histogram
        for (uint32_t k = blockIdx.x * RS_THREADS + threadIdx.x; k < 4u + (uint32_t)d.bins;
             k += gridDim.x * RS_THREADS)
            acc[k] = 0u;
    }
    if (!active) return;
    // with a CTA for every slice each claims one and none has to look for more
    const bool single = gridDim.x >= ((R + (uint32_t)RS_TILE - 1) / (uint32_t)RS_TILE) << d.slice_lg;
    __syncthreads();
    for (;;) {
        const uint32_t id = sm.tile, tile = id >> d.slice_lg;
        if (tile >= (R + (uint32_t)RS_TILE - 1) / (uint32_t)RS_TILE) break;
        resample_tile<RULE, SPLIT, SPREAD>(d, tile, id & ((1u << d.slice_lg) - 1u), sm);
        if (single) break;
        __syncthreads();  // sm is reused by the next tile
        if (threadIdx.x == 0) sm.tile = atomicAdd(&d.st->tile_counter, 1u);
        __syncthreads();
    }
}

// Gather of the new population (the plain form's second kernel): slot j of
// the other buffer receives the spins of replica srcmap[j], for every slot j <
// R_i, in 16-byte chunks.  Work item t is chunk t % CH of slot t / CH, so the
// stores of consecutive threads are consecutive and the loads of one slot's
// chunks are one contiguous source replica; a source with r copies is read
// by r neighbouring slots at nearly the same time, so its later reads hit
// L2.  Every thread keeps GA_U loads in flight: the map words first, then the
// data they point to, then the streaming stores.  Persistent: one wave of
// resident CTAs strides over all R_i * CH chunks.
#ifndef PA_GA_U
#define PA_GA_U 8
#endif
#ifndef PA_GA_MINB
#define PA_GA_MINB 3
#endif
constexpr int GA_THREADS = 256;
constexpr int GA_U = PA_GA_U;

// EM = true (the redistribution's gather) also copies every slot's energy
// level and magnetisation from the source replica.
template <bool EM>
__global__ void __launch_bounds__(GA_THREADS, PA_GA_MINB) k_gather(RunDev d) {
    const DevState* st = d.st;
    if (!st->active) return;
    const uint32_t Rn = st->R;  // clamped to the capacity by the scan
    const uint32_t src = st->src;
    const uint32_t CH = d.stride >> 4;
    const uint32_t last = d.cap_alloc - 1;
    const uint4* __restrict__ sp = reinterpret_cast<const uint4*>(d.spins[src]);
    uint4* __restrict__ dp = reinterpret_cast<uint4*>(d.spins[src ^ 1u]);
    const uint32_t* __restrict__ map = d.srcmap;
    if ((CH & 31u) == 0) {
        // a replica is a whole number of warp rows (L = 64: one 512-byte row
        // of 32 chunks): each warp takes groups of 32 consecutive slots, reads
        // their 32 map words in one coalesced load, and then copies GA_U
        // replicas at a time, lane l moving chunks l, l + 32, ... of each
        const uint32_t lane = threadIdx.x & 31u;
        const uint32_t rows = CH >> 5;
        const uint32_t nwarps = gridDim.x * (GA_THREADS / 32);
        for (uint32_t g = blockIdx.x * (GA_THREADS / 32) + (threadIdx.x >> 5); g * 32u < Rn;
             g += nwarps) {
            const uint32_t slot0 = g * 32u;
            const uint32_t nslot = min(32u, Rn - slot0);
            const uint32_t mine = lane < nslot ? min(__ldg(map + slot0 + lane), last) : 0u;
            for (uint32_t row = 0; row < rows; ++row) {
                const uint32_t c = row * 32u + lane;
                for (uint32_t k0 = 0; k0 < nslot; k0 += GA_U) {
                    uint4 v[GA_U];
#pragma unroll
                    for (int u = 0; u < GA_U; ++u) {
                        const uint32_t sidx = __shfl_sync(0xffffffffu, mine, (k0 + u) & 31u);
                        if (k0 + u < nslot) v[u] = __ldg(sp + (size_t)sidx * CH + c);
                    }
#pragma unroll
                    for (int u = 0; u < GA_U; ++u)
                        if (k0 + u < nslot) __stcs(dp + (size_t)(slot0 + k0 + u) * CH + c, v[u]);
                }
            }
        }
    } else {
        const unsigned long long items = (unsigned long long)Rn * CH;
        const unsigned long long nth = (unsigned long long)gridDim.x * GA_THREADS;
        const bool pow2 = (CH & (CH - 1)) == 0;
        const int shift = __ffs(CH) - 1;
        for (unsigned long long it0 = (unsigned long long)blockIdx.x * GA_THREADS + threadIdx.x;
             it0 < items; it0 += nth * GA_U) {
            uint32_t sidx[GA_U], c[GA_U];
#pragma unroll
            for (int u = 0; u < GA_U; ++u) {
                const unsigned long long it = it0 + (unsigned long long)u * nth;
                sidx[u] = 0;
                c[u] = 0;
                if (it < items) {
                    const uint32_t slot = pow2 ? (uint32_t)(it >> shift) : (uint32_t)(it / CH);
                    c[u] = (uint32_t)(it - (unsigned long long)slot * CH);
                    sidx[u] = min(__ldg(map + slot), last);  // a slot never holds more than cap_alloc
                }
            }
            uint4 v[GA_U];
#pragma unroll
            for (int u = 0; u < GA_U; ++u) {
                const unsigned long long it = it0 + (unsigned long long)u * nth;
                if (it < items) v[u] = __ldg(sp + (size_t)sidx[u] * CH + c[u]);
            }
#pragma unroll
            for (int u = 0; u < GA_U; ++u) {
                const unsigned long long it = it0 + (unsigned long long)u * nth;
                if (it < items) __stcs(dp + it, v[u]);
            }
        }
    }
    if (EM) {
        const uint32_t* es = d.ebin[src];
        const int32_t* ms = d.mag[src];
        uint32_t* ed = d.ebin[src ^ 1u];
        int32_t* md = d.mag[src ^ 1u];
        for (uint32_t j = blockIdx.x * GA_THREADS + threadIdx.x; j < Rn; j += gridDim.x * GA_THREADS) {
            const uint32_t i = min(map[j], last);
            ed[j] = es[i];
            md[j] = ms[i];
        }
    }
}

// Slot permutation of a redistribution: post-exchange slot j in segment q
// (dst[q] <= j < dst[q+1]) takes the source of pre-exchange slot
// src[q] + j - dst[q].
__global__ void __launch_bounds__(256) k_remap(RunDev d, const __grid_constant__ SegList segs) {
    const DevState* st = d.st;
    if (!st->active) return;
    const uint32_t Rn = st->R;
    const uint32_t last = d.cap_alloc - 1;
    for (uint32_t j = blockIdx.x * 256 + threadIdx.x; j < Rn; j += gridDim.x * 256) {
        uint32_t lo = 0, hi = segs.n;  // dst[lo] <= j < dst[hi]
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (segs.dst[mid] <= j) lo = mid;
            else hi = mid;
        }
        const uint32_t pre = min(segs.src[lo] + (j - segs.dst[lo]), last);
        d.srcmap2[j] = d.srcmap[pre];
    }
}

// Batched: global tile ids are claimed in increasing order; run r owns ids
// tile_base[r] .. tile_base[r+1]-1, so within a run tiles are claimed in order
// and the lookback only ever waits on tiles already running.
template <int RULE, bool SPREAD>
__global__ void __launch_bounds__(RS_THREADS, PA_RS_MINB) k_resample_batched(BatchDev b) {
    __shared__ ResampleSmem sm;
    __shared__ uint32_t s_run;
#if PA_RS_STAGE
    __shared__ RunDev s_d;
    uint32_t have = 0xffffffffu;
#endif
    for (;;) {
        if (threadIdx.x == 0) {
            const uint32_t g = atomicAdd(&b.counters[0], 1u);
            if (g >= b.total_tiles) {
                s_run = 0xffffffffu;
            } else {
                uint32_t lo = 0, hi = b.nruns;  // tile_base[lo] <= g < tile_base[hi]
                while (hi - lo > 1) {
                    const uint32_t mid = (lo + hi) >> 1;
                    if (b.tile_base[mid] <= g) lo = mid;
                    else hi = mid;
                }
                s_run = lo;
                sm.tile = g - b.tile_base[lo];
            }
        }
        __syncthreads();
        if (s_run == 0xffffffffu) break;
#if PA_RS_STAGE
        if (s_run != have) {
            stage_run(&b.runs[s_run], s_d);
            have = s_run;
            __syncthreads();
        }
        const RunDev& d = s_d;
#else
        const RunDev& d = b.runs[s_run];
#endif
        if (d.st->active)
            resample_tile<RULE, false, SPREAD>(d, sm.tile >> d.slice_lg, sm.tile & ((1u << d.slice_lg) - 1u), sm);
        __syncthreads();
    }
}

__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The record of the measured step: integer sums over the histogram by the CTA,
// then the averages, one per lane of a warp (an FP64 division takes some 1450
// cycles on GB300: two of them one after the other instead of eight).  Loads
// that depend on nothing come first.  us, timed by events: 10.0 -> 8.3 (4097
// levels), 12.6 -> 8.3 (16385).
__device__ __forceinline__ void obs_run(const RunDev& d, int nsweeps) {
    DevState* st = d.st;
    __shared__ long long s_part[3][8];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const uint32_t step = st->step, R = st->R, negbonds = st->negbonds, base = st->sweep_base;
    const unsigned long long done = st->sweeps_done;
    const double lnQ = st->lnQ, lnZ = st->lnZ;
    const long long mags = lane == 2 || lane == 3 ? (long long)d.accum[lane - 2] : 0ll;
    const long long dimN = (long long)d.dim * d.N;
    const long long E0 = 2 * (long long)(negbonds & 1u) - dimN;  // energy of level 0
    long long cnt = 0, sE = 0, sE2 = 0;
    each_level(d.hist, (uint32_t)d.bins, [&](uint32_t k, uint32_t h) {
        const long long E = E0 + 4 * (long long)k;
        const long long hE = (long long)h * E;
        cnt += h;
        sE += hE;
        sE2 += hE * E;
    });
    const double beta = d.beta[step];
    cnt = warp_sum_ll(cnt);
    sE = warp_sum_ll(sE);
    sE2 = warp_sum_ll(sE2);
    if (lane == 0) {
        s_part[0][wid] = cnt;
        s_part[1][wid] = sE;
        s_part[2][wid] = sE2;
    }
    __syncthreads();
    if (wid != 0) return;
    long long p0 = 0, p1 = 0, p2 = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        p0 += s_part[0][w];
        p1 += s_part[1][w];
        p2 += s_part[2][w];
    }
    // lanes 0..3: sum E, sum E^2, sum |M|, sum M^2 and their averages
    const long long sum = lane == 0 ? p1 : lane == 1 ? p2 : mags;
    const double mean = __ddiv_rn((double)sum, (double)R);
    const double mE = __shfl_sync(0xffffffffu, mean, 0), mE2 = __shfl_sync(0xffffffffu, mean, 1);
    const double mA = __shfl_sync(0xffffffffu, mean, 2), mM2 = __shfl_sync(0xffffffffu, mean, 3);
    // lanes 0..3: e, cv, m_abs, chi
    const double sq = lane == 1 ? mE : mA, sq2 = lane == 1 ? mE2 : mM2;
    const double var = __dsub_rn(sq2, __dmul_rn(sq, sq));
    const double fac = lane == 1 ? __dmul_rn(beta, beta) : beta;
    const double num = lane == 0 ? mE : lane == 2 ? mA : __dmul_rn(fac, var);
    const double avg = __ddiv_rn(num, (double)d.N);
    pa_obs* o = d.obs + step;
    if (lane < 4) {
        (&o->sumE)[lane] = sum;
        (&o->e)[lane] = avg;
    }
    if (lane == 0) {
        if (p0 != (long long)R) atomicOr(&st->status, ST_INVARIANT);
        o->step = step;
        o->R = R;
        o->beta = beta;
        o->lnQ = lnQ;
        o->lnZ = lnZ;
        st->sweep_base = base + (uint32_t)nsweeps;
        st->sweeps_done = done + (unsigned long long)nsweeps;
    }
}

__global__ void __launch_bounds__(256) k_obs(__grid_constant__ const RunDev d, int nsweeps) {
    chain_wait();
    obs_run(d, nsweeps);
}

// The observables of the swept step (last block) beside the reweight of the
// next (the others): neither waits for the other's result, and the chain of a
// step in a run of steps is a kernel shorter.  us per step on GB300: 1000 replicas at
// L = 16 22.9 -> 20.9, 4099 x 3D L = 6 31.1 -> 28.8, 20480 x L = 64 (theta = 1) 75.2 -> 72.8.
__global__ void __launch_bounds__(256) k_obs_tau(__grid_constant__ const RunDev d, int nsweeps) {
    chain_wait();
    if (blockIdx.x + 1 < gridDim.x) {
        tau_run<true>(d, blockIdx.x, gridDim.x - 1);
        return;
    }
    DevState* st = d.st;
    const uint32_t i = st->step + 1, R = st->R, cur = st->cur, epoch = st->epoch;
    obs_run(d, nsweeps);
    if (threadIdx.x >= 32) return;
    __syncwarp();
    if (threadIdx.x == 0 && i <= (uint32_t)d.K && R != 0) {
        __threadfence();
        if (atomicAdd(&st->tau_done, 1ull) == (unsigned long long)(gridDim.x - 1)) {
            __threadfence();
            tau_advance_next(d, i, R, cur, epoch);
        }
    }
}

__global__ void __launch_bounds__(256) k_obs_batched(BatchDev b) {
#if PA_RS_STAGE
    __shared__ RunDev s_d;
    stage_run(&b.runs[blockIdx.x], s_d);
    __syncthreads();
    const RunDev& d = s_d;
#else
    const RunDev& d = b.runs[blockIdx.x];
#endif
    obs_run(d, d.theta);
}

}  // namespace

cudaError_t launch_tau(const RunDev& d, cudaStream_t s) {
    RunDev dd = d;
    void* args[] = {&dd};
    return launch_chained((const void*)k_tau, dim3(tau_ctas(d.bins)), dim3(256), 0, s, args);
}

cudaError_t launch_obs_tau(const RunDev& d, int nsweeps, cudaStream_t s) {
    RunDev dd = d;
    void* args[] = {&dd, &nsweeps};
    return launch_chained((const void*)k_obs_tau, dim3(tau_ctas(d.bins) + 1), dim3(256), 0, s, args);
}

// One wave of resident CTAs (capped by the number of tiles), looked up once
// per device and kernel.
static int resample_wave(const void* fn, int which, uint32_t tiles) {
    static int cache[64][12];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int wave = cache[dev][which];
    if (wave <= 0) {
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, RS_THREADS, 0) != cudaSuccess)
            return 0;
        wave = sms * (per_sm < 1 ? 1 : per_sm);
        cache[dev][which] = wave;
    }
    return (int)((int64_t)tiles < wave ? (int64_t)tiles : wave);
}

// PA_RS_SPLIT = 1: the plain resample is two kernels, counts + scan (with the
// slot -> source map, levels and magnetisations) and then k_gather over the
// whole new population; 0 (the default): one kernel that gathers tile by
// tile.  Measured on GB300 at 2^21 replicas, L = 64, same bits, before that gather
// kept only data in registers (0.346 ms since): one kernel 0.366 ms with 4 loads in
// flight per thread (0.361 ms with 6); two kernels 0.374 ms (16 loads in flight per thread, 2 CTAs of
// 256 per SM), 0.380 ms (4 loads, 4 CTAs), 0.385 ms (8 loads, 3 CTAs).  The split
// form serves the redistribution's gather (pa_resample_finish), whose slot
// order is only known after the host has read the scan.
#ifndef PA_RS_SPLIT
#define PA_RS_SPLIT 0
#endif
constexpr bool RS_SPLIT = PA_RS_SPLIT != 0;

static int gather_grid() {
    static int cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (cache[dev] <= 0) {
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)k_gather<false>,
                                                          GA_THREADS, 0) != cudaSuccess)
            return 0;
        cache[dev] = sms * (per_sm < 1 ? 1 : per_sm);
    }
    return cache[dev];
}

// CTAs of a grid-stride pass over `n` replicas, 256 threads each.
static int flat_grid(uint64_t n) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    const uint64_t want = (n + 255u) / 256u, cap = (uint64_t)sms * 8u;
    return (int)(want < cap ? (want ? want : 1u) : cap);
}

template <bool SPLIT>
static cudaError_t launch_counts_scan(const RunDev& d, cudaStream_t s) {
    RunDev dd = d;
    void* args[] = {&dd};
    if (d.resample == PA_RESAMPLE_POISSON) {
        const int g = flat_grid(d.cap);
        if (g <= 0) return cudaErrorInvalidValue;
        const cudaError_t e = launch_chained((const void*)k_poisson_counts, dim3(g), dim3(256), 0, s, args);
        if (e != cudaSuccess) return e;
    }
    const bool drawn = d.resample != PA_RESAMPLE_NEAREST;
    const bool spread = !SPLIT && d.spread;
    const void* fn = drawn ? (spread ? (const void*)k_resample<2, SPLIT, !SPLIT>
                                     : (const void*)k_resample<2, SPLIT, false>)
                           : (spread ? (const void*)k_resample<0, SPLIT, !SPLIT>
                                     : (const void*)k_resample<0, SPLIT, false>);
    // cache slots: 0 and 4 the one-kernel forms (2 and 3 with k_spread), 7 and 9
    // the split forms
    const int grid = resample_wave(fn, SPLIT ? (drawn ? 9 : 7) : spread ? (drawn ? 3 : 2) : (drawn ? 4 : 0),
                                   d.tiles << d.slice_lg);
    if (grid <= 0) return cudaErrorInvalidValue;
    return launch_chained(fn, dim3(grid), dim3(RS_THREADS), 0, s, args);
}

cudaError_t launch_resample(const RunDev& d, cudaStream_t s) {
    cudaError_t e = launch_counts_scan<RS_SPLIT>(d, s);
    if (e == cudaSuccess && !RS_SPLIT && d.spread) {
        RunDev dd = d;
        void* args[] = {&dd};
        e = launch_chained((const void*)k_spread, dim3(RS_CTAS), dim3(256), 0, s, args);
    }
    if (e != cudaSuccess || !RS_SPLIT) return e;
    const int g = gather_grid();
    if (g <= 0) return cudaErrorInvalidValue;
    k_gather<false><<<g, GA_THREADS, 0, s>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_resample_scan(const RunDev& d, cudaStream_t s) {
    return launch_counts_scan<true>(d, s);
}

cudaError_t launch_remap_gather(const RunDev& d, const SegList& segs, cudaStream_t s) {
    const int g = gather_grid();
    if (g <= 0) return cudaErrorInvalidValue;
    k_remap<<<g, 256, 0, s>>>(d, segs);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    RunDev dm = d;
    dm.srcmap = d.srcmap2;
    k_gather<true><<<g, GA_THREADS, 0, s>>>(dm);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Multinomial resampling: the copy counts of all replicas come from R0
// independent draws.  Replica i weighs t_i = n_k 2^32 + F_k (k = its level);
// C_i = t_0 + ... + t_i are exact 64-bit integers, built by a two-pass scan over
// tiles of RS_TILE replicas (tile sums, then the prefix of each tile).  Draw j: v = words 2(j & 1) (low) and 2(j & 1) + 1 (high)
// of Philox block (j >> 1, step, 0, MULTINOMIAL|id), x = floor(v C_{R-1} /
// 2^64), one copy (atomic add) to the first replica with C_i > x.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long mn_weight(const RunDev& d, uint32_t k) {
    return ((unsigned long long)d.tab_n[k] << 32) + (unsigned long long)d.tab_F[k];
}

__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long v, unsigned long long* sw) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) sw[wid] = v;
    __syncthreads();
    unsigned long long tot = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += sw[w];
    __syncthreads();
    return tot;
}

__global__ void __launch_bounds__(RS_THREADS) k_mn_tile_sums(__grid_constant__ const RunDev d) {
    __shared__ unsigned long long sw[RS_THREADS / 32];
    chain_wait();
    const DevState* st = d.st;
    if (!st->active) return;
    const uint32_t R = st->R_prev, src = st->src;
    const uint32_t ntiles = (R + RS_TILE - 1) / RS_TILE;
    const uint32_t* eb = d.ebin[src];
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        unsigned long long part = 0;
        for (uint32_t j = threadIdx.x; j < (uint32_t)RS_TILE; j += RS_THREADS) {
            const uint32_t i = tile * RS_TILE + j;
            if (i < R) part += mn_weight(d, eb[i]);
        }
        const unsigned long long tot = block_sum_u64(part, sw);
        if (threadIdx.x == 0) d.mn_tiles[tile] = tot;
    }
}

// C_i per replica (inclusive), and the copy counts cleared for the draws.  A CTA
// adds up the sums of the tiles before its own itself (a few independent loads a
// thread), from its last tile on, so that it reads each sum once however many tiles
// it takes: the loads grow with the tiles, not with their square.  The resample of 2^26
// replicas of L = 4 (32768 tiles) takes 20.9 ms on GB300, 21.1 with the sums from the
// first tile on.  mn_tiles[ntiles] = the total.
__global__ void __launch_bounds__(RS_THREADS) k_mn_cum(__grid_constant__ const RunDev d) {
    __shared__ unsigned long long sw[RS_THREADS / 32];
    chain_wait();
    const DevState* st = d.st;
    if (!st->active) return;
    const uint32_t R = st->R_prev, src = st->src;
    const uint32_t ntiles = (R + RS_TILE - 1) / RS_TILE;
    const uint32_t* eb = d.ebin[src];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long prefix = 0;  // of the tiles before `summed`
    uint32_t summed = 0;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const uint32_t i0 = tile * RS_TILE + threadIdx.x * RS_ITEMS;
        unsigned long long w[RS_ITEMS], part = 0;
#pragma unroll
        for (int j = 0; j < RS_ITEMS; ++j) {
            w[j] = i0 + j < R ? mn_weight(d, eb[i0 + j]) : 0ull;
            part += w[j];
        }
        unsigned long long incl = part;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        unsigned long long ahead = 0;
        for (uint32_t k = summed + threadIdx.x; k < tile; k += RS_THREADS) ahead += d.mn_tiles[k];
        prefix += block_sum_u64(ahead, sw);
        summed = tile;
        unsigned long long before = prefix;
        if (lane == 31) sw[wid] = incl;
        __syncthreads();
        if (tile == ntiles - 1 && threadIdx.x == 0) {
            unsigned long long all = before;
            for (int k = 0; k < RS_THREADS / 32; ++k) all += sw[k];
            d.mn_tiles[ntiles] = all;
        }
        for (int k = 0; k < wid; ++k) before += sw[k];
        unsigned long long run = before + incl - part;
#pragma unroll
        for (int j = 0; j < RS_ITEMS; ++j) {
            if (i0 + j < R) {
                run += w[j];
                d.mn_cum[i0 + j] = run;
                d.counts[i0 + j] = 0u;
            }
        }
        __syncthreads();
    }
}

constexpr uint32_t MN_TOP = 1024;
__global__ void __launch_bounds__(256) k_mn_draw(__grid_constant__ const RunDev d) {
    chain_wait();
    const DevState* st = d.st;
    if (!st->active) return;
    const uint32_t R = st->R_prev, step = st->step;
    const uint32_t ntiles = (R + RS_TILE - 1) / RS_TILE;
    const unsigned long long total = d.mn_tiles[ntiles];
    if (total == 0ull) return;
    // the cumulative weight at the end of every `span` replicas, so that the first
    // steps of a search stay in shared memory: 150001 replicas take 18 steps of an L2
    // round trip each otherwise (a step of the run 165.9 -> 164.4 us on GB300)
    __shared__ unsigned long long s_top[MN_TOP];
    const uint32_t span = (ntiles + MN_TOP - 1) / MN_TOP * (uint32_t)RS_TILE;
    const uint32_t tops = (R + span - 1) / span;
    const bool staged = tops > 8;  // fewer cost more to stage than they save
    for (uint32_t e = threadIdx.x; staged && e < tops; e += blockDim.x)
        s_top[e] = d.mn_cum[min((uint64_t)(e + 1) * span, (uint64_t)R) - 1];
    __syncthreads();
    const uint32_t ctr3 = (TAG_MULTINOMIAL << 28) | d.instance;
    const uint32_t k0 = (uint32_t)d.seed, k1 = (uint32_t)(d.seed >> 32);
    const uint32_t pairs = (d.R0 + 1u) / 2u;
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < pairs;
         p += gridDim.x * blockDim.x) {
        const uint4 u = philox(p, step, 0u, ctr3, k0, k1);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t j = 2u * p + (uint32_t)e;
            if (j >= d.R0) break;
            const unsigned long long v = e == 0 ? (((unsigned long long)u.y << 32) | u.x)
                                                : (((unsigned long long)u.w << 32) | u.z);
            const unsigned long long x = __umul64hi(v, total);
            uint32_t t0 = 0, t1 = staged ? tops - 1 : 0;  // first top with C > x
            while (t0 < t1) {
                const uint32_t mid = (t0 + t1) / 2;
                if (s_top[mid] > x) t1 = mid;
                else t0 = mid + 1;
            }
            uint32_t lo = t0 * span;  // first i with C_i > x
            uint32_t hi = staged ? (uint32_t)min((uint64_t)lo + span, (uint64_t)R) - 1 : R - 1;
            while (lo < hi) {
                const uint32_t mid = lo + (hi - lo) / 2;
                if (d.mn_cum[mid] > x) hi = mid;
                else lo = mid + 1;
            }
            atomicAdd(&d.counts[lo], 1u);
        }
    }
}

cudaError_t launch_multinomial(const RunDev& d, cudaStream_t s) {
    if (!d.mn_cum || !d.mn_tiles) return cudaErrorInvalidValue;
    const int wave = resample_wave((const void*)k_mn_cum, 5, d.tiles);
    if (wave <= 0) return cudaErrorInvalidValue;
    const int g = flat_grid((d.R0 + 1u) / 2u);
    if (g <= 0) return cudaErrorInvalidValue;
    RunDev dd = d;
    void* args[] = {&dd};
    const struct {
        const void* fn;
        int grid, threads;
    } pass[] = {{(const void*)k_mn_tile_sums, wave, RS_THREADS},
                {(const void*)k_mn_cum, wave, RS_THREADS},
                {(const void*)k_mn_draw, g, 256}};
    for (const auto& p : pass) {
        const cudaError_t e = launch_chained(p.fn, dim3(p.grid), dim3(p.threads), 0, s, args);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_obs(const RunDev& d, int nsweeps, cudaStream_t s) {
    RunDev dd = d;
    void* args[] = {&dd, &nsweeps};
    return launch_chained((const void*)k_obs, dim3(1), dim3(256), 0, s, args);
}

cudaError_t launch_tau_batched(const BatchDev& b, cudaStream_t s) {
    k_tau_batched<<<dim3(b.nruns, tau_ctas(b.max_bins)), 256, 0, s>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_resample_batched(const BatchDev& b, cudaStream_t s) {
    if (b.any_poisson) {
        k_poisson_counts_batched<<<b.total_tiles, RS_THREADS, 0, s>>>(b);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const bool drawn = b.any_poisson || b.any_multinomial;
    const void* fn = drawn ? (b.any_spread ? (const void*)k_resample_batched<3, true>
                                           : (const void*)k_resample_batched<3, false>)
                           : (b.any_spread ? (const void*)k_resample_batched<0, true>
                                           : (const void*)k_resample_batched<0, false>);
    const int grid = resample_wave(fn, b.any_spread ? (drawn ? 11 : 10) : (drawn ? 6 : 1), b.total_tiles);
    if (grid <= 0) return cudaErrorInvalidValue;
    BatchDev bb = b;
    void* args[] = {&bb};
    const cudaError_t e = cudaLaunchKernel(fn, dim3(grid), dim3(RS_THREADS), args, 0, s);
    if (e != cudaSuccess) return e;
    if (b.any_spread) k_spread_batched<<<dim3(b.nruns, 32), 256, 0, s>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_obs_batched(const BatchDev& b, cudaStream_t s) {
    k_obs_batched<<<b.nruns, 256, 0, s>>>(b);
    return cudaGetLastError();
}

}  // namespace pa
