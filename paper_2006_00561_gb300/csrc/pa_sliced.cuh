// pa_sliced.cuh -- the replica-sliced Metropolis sweep with its fused
// measurement (energy, magnetisation, energy histogram): every lattice and layout
// but the packed 2D L = 64 and 128 ones, whose register kernels are in
// pa_sweep_l64.cu.  The plain kernels are in pa_sweep.cu, the batched ones in
// pa_sweep_batched.cu.
//
// Model: Eq. 6 (H = -sum_<ij> J_ij s_i s_j over the bonds of a periodic L^dim
// lattice; J = +1 for the ferromagnet, +-1 for the Edwards-Anderson variant).
// Equilibration (Sec. 2, theta MCMC sweeps at the new temperature): one sweep
// updates the sites of colour 0 (even coordinate sum), then colour 1; sites of
// one colour have no bond between them, so they are updated together.  A site
// with c_u unsatisfied bonds has dE = 4 (dim - c_u); it flips if dE <= 0, or
// if its uniform u (word h & 3 of the Philox block with counter (2 g + colour,
// h >> 2, SWEEP | instance, slot), h = s >> 1, g = global sweep index) is below the
// threshold T(beta_i, dE) = floor(2^32 exp(-beta_i dE)).
//
// Replica-sliced: 32 replicas of one run, slots b0 .. b0 + 31 (a chunk), are
// kept in shared memory as one 32-bit word per lattice site whose bit r is the
// spin of replica b0 + r (set = -1).  All bit logic (bond states, the bit-sliced
// count of unsatisfied bonds, the energy classes, the flips) then runs on 32
// replicas at once, whatever L and the dimension.  A half-sweep of colour c is
// NGROUPS x 32 Philox blocks: group k holds the four colour-c sites with h in
// 4k .. 4k + 3, and replica r draws its block (2g + c, k, SWEEP | instance,
// b0 + r).  Every uniform is folded into carry chains, one per (site, class):
// acc = 2 acc + [u >= T_class], so replica r ends at bit r.  A site flips in
// replica r if its class has dE <= 0, or if bit r of the chain of its class is
// clear (u < T).
#pragma once

#include "pa_internal.cuh"

namespace pa {
namespace {

__device__ __forceinline__ uint32_t warp_sum_u32(uint32_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Histogram of the valid lanes' energy levels, with one atomic per distinct
// level (warp-aggregated: lanes holding the same level elect one).
__device__ __forceinline__ void hist_flush(uint32_t* hist, uint32_t level, bool valid, int lane) {
    const unsigned mask = __ballot_sync(0xffffffffu, valid);
    if (valid) {
        const unsigned peers = __match_any_sync(mask, level);
        if (lane == __ffs(peers) - 1) atomicAdd(&hist[level], (uint32_t)__popc(peers));
    }
}

// Per-run scalars of one sweep launch, read from the run's device state.
struct SweepCtx {
    uint32_t R, cur, g0, parity, T[3], full, ctag;
};

__device__ __forceinline__ SweepCtx sweep_ctx(const RunDev& d) {
    SweepCtx x;
    const DevState* st = d.st;
    const uint32_t step = st->step;
    x.R = st->R;
    x.cur = st->cur;
    x.g0 = st->sweep_base;
    x.parity = st->negbonds & 1u;
#pragma unroll
    for (int c = 0; c < 3; ++c) x.T[c] = d.thr[step * 4 + c];
    x.full = d.thr[step * 4 + 3];
    x.ctag = (TAG_SWEEP << 28) | d.instance;  // counter word 2 of the sweep
    return x;
}

__host__ __device__ constexpr int ceil_div(int a, int b) { return (a + b - 1) / b; }
__host__ __device__ constexpr int gcd(int a, int b) { return b ? gcd(b, a % b) : a; }
__host__ __device__ constexpr int bits_of(int v) { return v <= 1 ? 1 : 1 + bits_of(v >> 1); }

template <int DIM, int L>
struct Geo {
    static constexpr int N = DIM == 2 ? L * L : L * L * L;
    static constexpr int NROWS = DIM == 2 ? L : L * L;
    static constexpr int NGROUPS = N / 8;          // groups of four colour sites
    static constexpr int NCLS = DIM == 2 ? 2 : 3;  // classes with dE > 0
    // Site words: row r, column x at r LP + x.  The odd row pitch spreads the
    // sites of one column, and of groups eight sites apart, over the banks.
    static constexpr int LP = L + 1;
    static constexpr int NS = NROWS * LP;
    // Packed row words (ceil(L / 32) per row) and the transfer unit: UROWS row words
    // of a replica (a multiple of four: 16-byte loads) make UWORDS words of 32
    // consecutive sites.
    static constexpr int RW = NROWS * ceil_div(L, 32);
    static constexpr int UROWS = L >= 32 ? 4 : (32 / gcd(L, 32) > 4 ? 32 / gcd(L, 32) : 4);
    static constexpr int UWORDS = L >= 32 ? 4 : UROWS * L / 32;
    static constexpr int UNITS = ceil_div(RW, UROWS);
    static constexpr uint32_t ROWMASK = L >= 32 ? 0xffffffffu : ((1u << (L & 31)) - 1u);
    static_assert(N % 8 == 0 && RW % 4 == 0, "whole groups, whole 16-byte words");
    static constexpr int JWORDS = (NS + 3) / 4;  // coupling patterns, one byte per site word
};

template <int DIM, int L>
__device__ __forceinline__ int ix_of(int s) {  // site word of site s
    const int row = s / L;
    return row * Geo<DIM, L>::LP + (s - row * L);
}

// Transpose of a 32 x 32 bit matrix, row r in lane r: afterwards bit r of lane
// c is what bit c of lane r was.  Five exchanges, four instructions each;
// forming the 32 columns by ballots takes about 130 instructions.
__device__ __forceinline__ uint32_t transpose32(uint32_t v, int lane) {
#pragma unroll
    for (int k = 4; k >= 0; --k) {
        const int j = 1 << k;
        const uint32_t m = k == 4   ? 0x0000ffffu
                           : k == 3 ? 0x00ff00ffu
                           : k == 2 ? 0x0f0f0f0fu
                           : k == 1 ? 0x33333333u
                                    : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, v, j);
        v = (lane & j) ? ((v & ~m) | ((y >> j) & m)) : ((v & m) | ((y & m) << j));
    }
    return v;
}

// Population -> site words: unit u of the chunk, by one warp (lane r reads
// replica b0 + r).  Rows of another length than 32 are shifted together into
// words of 32 sites at compile-time offsets.
template <int DIM, int L>
__device__ __forceinline__ void load_unit(const uint8_t* src, bool i8, uint32_t stride, bool valid,
                                          uint32_t* S, int u, int lane) {
    using G = Geo<DIM, L>;
    uint32_t w[G::UWORDS];
    if (i8) {  // one byte per site, the sign bit is the spin
#pragma unroll
        for (int k = 0; k < G::UWORDS; ++k) {
            const uint32_t at = 32u * (uint32_t)(u * G::UWORDS + k);
            w[k] = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (valid && at + 16u * h < stride) {
                    const uint4 b = *reinterpret_cast<const uint4*>(src + at + 16u * h);
                    // the four sign bits of a word to bits 0..3: one product, no carries
                    auto nib = [](uint32_t x) { return (((x >> 7) & 0x01010101u) * 0x10204080u) >> 28; };
                    w[k] |= (nib(b.x) | nib(b.y) << 4 | nib(b.z) << 8 | nib(b.w) << 12) << (16 * h);
                }
            }
        }
    } else {
        uint32_t row[G::UROWS];
#pragma unroll
        for (int q = 0; q < G::UROWS; q += 4) {
            const int r = u * G::UROWS + q;
            uint4 b = make_uint4(0, 0, 0, 0);
            if (valid && r < G::RW) b = *reinterpret_cast<const uint4*>(src + 4 * (size_t)r);
            // a loaded population may have bits set beyond the row: they are not spins
            row[q] = b.x & G::ROWMASK, row[q + 1] = b.y & G::ROWMASK;
            row[q + 2] = b.z & G::ROWMASK, row[q + 3] = b.w & G::ROWMASK;
        }
        if constexpr (L >= 32) {
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = row[k];
        } else {
#pragma unroll
            for (int k = 0; k < G::UWORDS; ++k) w[k] = 0;
#pragma unroll
            for (int r = 0; r < G::UROWS; ++r) {
                const int o = r * L, k = o >> 5, sh = o & 31;
                w[k] |= row[r] << sh;
                if (sh + L > 32) w[k + 1] |= row[r] >> (32 - sh);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < G::UWORDS; ++k) {
        const int s = 32 * (u * G::UWORDS + k) + lane;
        const uint32_t t = transpose32(w[k], lane);
        if (s < G::N) S[ix_of<DIM, L>(s)] = t;
    }
}

// Site words -> population, the reverse of load_unit.  Bytes beyond the last
// site keep what they hold.
template <int DIM, int L>
__device__ __forceinline__ void store_unit(uint8_t* dst, bool i8, bool valid, const uint32_t* S,
                                           int u, int lane) {
    using G = Geo<DIM, L>;
    uint32_t w[G::UWORDS];
#pragma unroll
    for (int k = 0; k < G::UWORDS; ++k) {
        const int s = 32 * (u * G::UWORDS + k) + lane;
        w[k] = transpose32(s < G::N ? S[ix_of<DIM, L>(s)] : 0u, lane);
    }
    if (!valid) return;
    if (i8) {
#pragma unroll
        for (int k = 0; k < G::UWORDS; ++k) {
            const int at = 32 * (u * G::UWORDS + k);
            // four bits to four bytes of 0 / 1 (no carries), then to +1 / -1
            auto spins4 = [](uint32_t n) {
                return 0x01010101u | ((((n & 15u) * 0x00204081u) & 0x01010101u) * 0xfeu);
            };
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t b = w[k] >> (16 * h);
                const int s = at + 16 * h;
                if (s + 16 <= G::N) {
                    *reinterpret_cast<uint4*>(dst + s) = make_uint4(spins4(b), spins4(b >> 4),
                                                                    spins4(b >> 8), spins4(b >> 12));
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (s + 4 * q < G::N)
                            *reinterpret_cast<uint32_t*>(dst + s + 4 * q) = spins4(b >> (4 * q));
                }
            }
        }
        return;
    }
    uint32_t row[G::UROWS];
    if constexpr (L >= 32) {
#pragma unroll
        for (int k = 0; k < 4; ++k) row[k] = w[k];
    } else {
#pragma unroll
        for (int r = 0; r < G::UROWS; ++r) {
            const int o = r * L, k = o >> 5, sh = o & 31;
            uint32_t v = w[k] >> sh;
            if (sh + L > 32) v |= w[k + 1] << (32 - sh);
            row[r] = v & G::ROWMASK;
        }
    }
#pragma unroll
    for (int q = 0; q < G::UROWS; q += 4) {
        const int r = u * G::UROWS + q;
        if (r < G::RW)
            *reinterpret_cast<uint4*>(dst + 4 * (size_t)r) =
                make_uint4(row[q], row[q + 1], row[q + 2], row[q + 3]);
    }
}

// Site words of a site's neighbours in the order +x, -x, +y, -y (, +z, -z), periodic.
template <int DIM, int L>
__device__ __forceinline__ void nbrs_of(int row, int x, int (&nb)[2 * DIM]) {
    constexpr int LP = Geo<DIM, L>::LP;
    const int at = row * LP + x, y = DIM == 2 ? row : row % L;
    nb[0] = x == L - 1 ? at - (L - 1) : at + 1;
    nb[1] = x == 0 ? at + (L - 1) : at - 1;
    nb[2] = y == L - 1 ? at - (L - 1) * LP : at + LP;
    nb[3] = y == 0 ? at + (L - 1) * LP : at - LP;
    if constexpr (DIM == 3) {
        const int z = row / L;
        nb[4] = z == L - 1 ? at - (L - 1) * L * LP : at + L * LP;
        nb[5] = z == 0 ? at + (L - 1) * L * LP : at - L * LP;
    }
}

// acc = 2 acc + [u >= T]: the carry of u - T, shifted in with the add.
__device__ __forceinline__ uint32_t chain(uint32_t acc, uint32_t u, uint32_t T) {
    uint32_t out;
    asm("{\n\t.reg .u32 t;\n\tsub.cc.u32 t, %1, %2;\n\taddc.u32 %0, %3, %3;\n\t}"
        : "=r"(out) : "r"(u), "r"(T), "r"(acc));
    return out;
}

__device__ __forceinline__ void mul_hilo(uint32_t m, uint32_t a, uint32_t& hi, uint32_t& lo) {
    uint64_t p;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(m));
    hi = (uint32_t)(p >> 32);
    lo = (uint32_t)p;
}

// Bit-sliced counter of 32 replicas: adds word v into C[0..K-1].
template <int K>
__device__ __forceinline__ void count_in(uint32_t (&C)[K], uint32_t v) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t t = C[k] & v;
        C[k] ^= v;
        v = t;
    }
}

// Sum over the warp of the bit-sliced counters, for replica r = lane: the
// transposed plane k of lane r holds bit r of every lane, weighted 2^k.
template <int K>
__device__ __forceinline__ uint32_t count_out(const uint32_t (&C)[K], int lane) {
    uint32_t tot = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) tot += (uint32_t)__popc(transpose32(C[k], lane)) << k;
    return tot;
}

// Philox round keys: pointers into the kernel parameters (plain kernels, so
// that the xors take them as constant-bank operands) or registers (batched
// kernels, from a shared-memory copy of the chunk's run; read from there in
// every round they run 1-2 % slower).
struct Keys {
    const uint32_t* rk0;
    const uint32_t* rk1;
};
struct KeyRegs {
    uint32_t rk0[10], rk1[10];
};

// Philox4x32-10 of the blocks (c0, k, ctag, slot) of a half-sweep, c0 = 2 g +
// colour: round 1 multiplies only words that all of them share (the group index
// k enters word 1 and the slot word 3, both by xors); round 2 multiplies one
// group word and one replica word, round 3 again one of each.  The replica
// words depend only on the chunk and the half-sweep, so they are formed once
// per replica into a table of 32 entries (replica_words) that every group
// reads; the group words once per group and thread: a block costs 14 of
// Philox's 20 multiplies.  With the table no thread has to hold several groups
// to share the replica products, so a thread needs 46 to 60 registers and 32
// warps fit an SM, where the form without it ran fastest with four groups per
// lane, one warp per chunk, at 126 to 212 registers.
constexpr uint32_t PM0 = 0xD2511F53u, PM1 = 0xCD9E8D57u;

struct HalfSweep {
    uint32_t y0s, y1;   // round 1 of ctag: word 0 before the xor with k, word 1
    uint32_t y2s, y3k;  // round 1 of c0: word 2 before the xor with the slot, word 3 ^ key
};

template <typename KT>
__device__ __forceinline__ HalfSweep half_sweep(const KT& K, uint32_t ctag, uint32_t c0) {
    HalfSweep h;
    uint32_t hi, lo;
    mul_hilo(PM1, ctag, hi, lo);
    h.y0s = hi ^ K.rk0[0];
    h.y1 = lo ^ K.rk0[1];
    mul_hilo(PM0, c0, hi, lo);
    h.y2s = hi ^ K.rk1[0];
    h.y3k = lo ^ K.rk1[1];
    return h;
}

// Table place of replica r: the eight replicas of a quarter of the chunk are
// four apart, so that four lanes on the same replica of each quarter read one
// 64-byte span.
__device__ __forceinline__ int rt_place(int r) { return (r & 7) * 4 + (r >> 3); }

// {round-2 word 1, round-3 word 2 before the xor, round-3 word 3} of a slot.
template <typename KT>
__device__ __forceinline__ uint4 replica_words(const KT& K, const HalfSweep& h, uint32_t slot) {
    uint32_t h2, z1, h3, l3;
    mul_hilo(PM1, h.y2s ^ slot, h2, z1);  // round 2, replica half
    mul_hilo(PM0, h2 ^ h.y1, h3, l3);     // round 3, replica half
    return make_uint4(z1, h3, l3, 0u);
}

struct GroupWords {
    uint32_t w0, w1, w2;  // round-3 words 0 and 2 before the xor with the replica's, word 1
};

template <typename KT>
__device__ __forceinline__ GroupWords group_words(const KT& K, const HalfSweep& h, uint32_t k) {
    GroupWords g;
    uint32_t hi, lo, z2;
    mul_hilo(PM0, h.y0s ^ k, hi, lo);  // round 2, group half
    z2 = hi ^ h.y3k;
    g.w2 = lo ^ K.rk1[2];
    mul_hilo(PM1, z2, hi, lo);         // round 3, group half
    g.w0 = hi ^ K.rk0[2];
    g.w1 = lo;
    return g;
}

// Draws RL replicas' blocks of a group (the RL of quarter q of the chunk, or all
// of it if RL = 32), highest replica first, and folds their uniforms into the
// chains of the group's four sites.
// Replicas unrolled together, measured on GB300 (attempts/ns at 2, 4, 8, 16): 3D
// +-J L = 10 1257, 1349, 1370, 1369; L = 8 1401, 1385, 1425, 1358; 2D L = 32 1623, 1589,
// 1695, 1658; L = 64 (bytes) 1584, 1591, 1616, 1559.
#ifndef PA_RS_UNROLL
#define PA_RS_UNROLL 8
#endif
constexpr int RS_UNROLL = PA_RS_UNROLL;
template <int NC, int RL, typename KT>
__device__ __forceinline__ void draw(const KT& K, const GroupWords& g, const uint4* rt, int q,
                                     const uint32_t (&T)[3], uint32_t (&acc)[4][NC]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[i][c] = 0u;
#pragma unroll RS_UNROLL
    for (int r = RL - 1; r >= 0; --r) {
        const uint4 e = rt[RL == 32 ? rt_place(r) : r * 4 + q];
        uint32_t c0 = g.w0 ^ e.x, c1 = g.w1, c2 = g.w2 ^ e.y, c3 = e.z;
#pragma unroll
        for (int rr = 3; rr < 10; ++rr) {
            uint32_t hiA, loA, hiB, loB;
            mul_hilo(PM0, c0, hiA, loA);
            mul_hilo(PM1, c2, hiB, loB);
            c0 = hiB ^ c1 ^ K.rk0[rr];
            c1 = loB;
            c2 = hiA ^ c3 ^ K.rk1[rr];
            c3 = loA;
        }
        const uint32_t w[4] = {c0, c1, c2, c3};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[i][c] = chain(acc[i][c], w[i], T[c]);
    }
}

// Flips the colour-c site of pair h in the 32 replicas: counts their
// unsatisfied bonds bit-sliced and combines the classes with the chains.
template <int DIM, int L, bool PMJ>
__device__ __forceinline__ void flip_site(uint32_t* S, const uint8_t* JS, int h, int c,
                                          const uint32_t (&acc)[Geo<DIM, L>::NCLS], uint32_t full) {
    const int row = h / (L / 2), m = h - row * (L / 2);
    const int par = DIM == 2 ? (row & 1) : ((row % L + row / L) & 1);
    const int x = 2 * m + ((c + par) & 1);
    int nb[2 * DIM];
    nbrs_of<DIM, L>(row, x, nb);
    const int at = row * Geo<DIM, L>::LP + x;
    const uint32_t W = S[at];
    uint32_t v[2 * DIM];
    const uint32_t jp = PMJ ? (uint32_t)JS[at] : 0u;
#pragma unroll
    for (int d = 0; d < 2 * DIM; ++d) {
        const uint32_t jm = PMJ ? (0u - ((jp >> d) & 1u)) : 0u;
        v[d] = W ^ S[nb[d]] ^ jm;
    }
    uint32_t a[Geo<DIM, L>::NCLS];  // replicas whose uniform is below the class's threshold
#pragma unroll
    for (int k = 0; k < Geo<DIM, L>::NCLS; ++k) a[k] = ~acc[k] | (0u - ((full >> k) & 1u));
    const uint32_t s1 = v[0] ^ v[1] ^ v[2], k1 = (v[0] & v[1]) | (v[2] & (v[0] ^ v[1]));
    uint32_t flip;
    if constexpr (DIM == 2) {
        const uint32_t b0 = s1 ^ v[3], k2 = s1 & v[3];
        const uint32_t b1 = k1 ^ k2, b2 = k1 & k2;
        const uint32_t hi = b1 | b2;  // c_u >= 2: dE <= 0; 1: dE = 4; 0: dE = 8
        flip = hi | (b0 & a[0]) | (~b0 & a[1]);
    } else {
        const uint32_t s2 = v[3] ^ v[4] ^ v[5], k2 = (v[3] & v[4]) | (v[5] & (v[3] ^ v[4]));
        const uint32_t b0 = s1 ^ s2, k3 = s1 & s2;
        const uint32_t b1 = k1 ^ k2 ^ k3, b2 = (k1 & k2) | (k3 & (k1 ^ k2));
        // c_u >= 3: dE <= 0; 2: dE = 4; 1: dE = 8; 0: dE = 12
        flip = b2 | (b1 & (b0 | a[0])) | (~b1 & ((b0 & a[1]) | (~b0 & a[2])));
    }
    S[at] = W ^ flip;
}

// Coupling pattern of every site, bit d of JS = J(s, dir d) is -1, dirs in the
// order of nbrs_of; threads first, first + step, ...
template <int DIM, int L>
__device__ __forceinline__ void couplings(const RunDev& d, uint8_t* JS, int first, int step) {
    using G = Geo<DIM, L>;
    constexpr int NW = ceil_div(L, 32);
    const bool i8 = d.layout == PA_LAYOUT_INT8;
    const int nw = (int)d.nwords;
    for (int s = first; s < G::N; s += step) {
        const int row = s / L, x = s - row * L;
        int nb[2 * DIM];
        nbrs_of<DIM, L>(row, x, nb);
        uint32_t jp = 0;
#pragma unroll
        for (int dd = 0; dd < DIM; ++dd) {
            const int nr = nb[2 * dd + 1] / G::LP, nx = nb[2 * dd + 1] - nr * G::LP;
            // bond (s, +d) and bond (s - e_d, +d)
            if (i8) {
                jp |= (d.j8[s * DIM + dd] < 0 ? 1u : 0u) << (2 * dd);
                jp |= (d.j8[(nr * L + nx) * DIM + dd] < 0 ? 1u : 0u) << (2 * dd + 1);
            } else {
                const uint32_t* j = d.jpk + dd * nw;
                jp |= ((j[row * NW + x / 32] >> (x % 32)) & 1u) << (2 * dd);
                jp |= ((j[nr * NW + nx / 32] >> (nx % 32)) & 1u) << (2 * dd + 1);
            }
        }
        JS[row * G::LP + x] = (uint8_t)jp;
    }
}

// Measurement of the threads' sites (first, first + TT, ...): unsatisfied bonds
// (s, +d) and spins down of the 32 replicas, summed over the warp for replica
// r = lane.
template <int DIM, int L, bool PMJ, int TT>
__device__ __forceinline__ void measure(const uint32_t* S, const uint8_t* JS, int first, int lane,
                                        uint32_t& U, uint32_t& down) {
    using G = Geo<DIM, L>;
    constexpr int SPT = ceil_div(G::N, TT);  // sites per thread
    uint32_t CU[bits_of(DIM * SPT)] = {}, CM[bits_of(SPT)] = {};
    for (int s = first; s < G::N; s += TT) {
        const int row = s / L, x = s - row * L;
        int nb[2 * DIM];
        nbrs_of<DIM, L>(row, x, nb);
        const int at = row * G::LP + x;
        const uint32_t W = S[at];
        const uint32_t jp = PMJ ? (uint32_t)JS[at] : 0u;
        count_in(CM, W);
#pragma unroll
        for (int dd = 0; dd < DIM; ++dd) {
            const uint32_t jm = PMJ ? (0u - ((jp >> (2 * dd)) & 1u)) : 0u;
            count_in(CU, W ^ S[nb[2 * dd]] ^ jm);
        }
    }
    U = count_out(CU, lane);
    down = count_out(CM, lane);
}

// Level, magnetisation and histogram of the chunk's replicas (one warp, one
// replica per valid lane), and the magnetisation sums.
template <int N>
__device__ __forceinline__ void record(const RunDev& d, const SweepCtx& x, uint32_t slot, bool valid,
                                       uint32_t U, uint32_t down, int lane, long long& sAbsM,
                                       long long& sM2) {
    const int M = N - 2 * (int)down;
    if (valid) {
        d.ebin[x.cur][slot] = U >> 1;
        d.mag[x.cur][slot] = M;
        if ((U & 1u) != x.parity) atomicOr(&d.st->status, ST_INVARIANT);
        sAbsM += (long long)(M < 0 ? -M : M);
        sM2 += (long long)M * M;
    }
    hist_flush(d.hist, U >> 1, valid, lane);
}

// Adds the lanes' magnetisation sums to the run's (one warp) and clears them.
__device__ __forceinline__ void flush_mag(unsigned long long* accum, long long& sAbsM, long long& sM2,
                                          int lane) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sAbsM += __shfl_xor_sync(0xffffffffu, sAbsM, o);
        sM2 += __shfl_xor_sync(0xffffffffu, sM2, o);
    }
    if (lane == 0 && (sAbsM | sM2)) {
        atomicAdd(&accum[0], (unsigned long long)sAbsM);
        atomicAdd(&accum[1], (unsigned long long)sM2);
    }
    sAbsM = sM2 = 0;
}

// --------------------------------------------------------------------------
// The bound is integer issue: 14 multiplies of two FMA-heavy slots each, 8 or 12
// two-instruction tests and some 16 xors per block of four attempts.  Measured
// on GB300, attempts/ns, one warp per chunk (packed) or per replica (bytes) ->
// teams: 3D +-J L = 10 1174 -> 1370 (2^17 replicas), L = 8 1117 -> 1425 (2^18), L = 6 963
// -> 1106, L = 12 890 -> 1221, L = 16 1035 -> 1348, 2D L = 32 1466 -> 1695, L = 16 1352 ->
// 1633, L = 8 345 -> 1449; bytes: 2D L = 64 364 -> 1616, L = 128 220 -> 938 (3000
// replicas).  Small populations, us per sweep launch of theta = 10: 1024 x 3D L = 10
// 218 -> 45, 4099 x L = 6 74 -> 21, 1000 x 2D L = 16 (bytes) 26 -> 21; theta = 1: 150001 x 2D L =
// 32 229 -> 127.
//
// A team of TT threads (one CTA) per chunk.  RSP = 1: thread t takes group t, t
// + TT, ... of all 32 replicas; RSP = 4: threads 4k .. 4k + 3 share group k, each
// drawing the blocks of the RPQ = 8 replicas of a quarter of the chunk.  Their
// chains hold one byte each of the four sites' words; two exchanges transpose the
// bytes, and thread 4k + i flips site i.  With RPQ = 4 or 2 a chunk has 16 or 8
// replicas, which take the low bits of each byte.
// --------------------------------------------------------------------------
template <int DIM, int L, int RSP>
struct Team {
    static constexpr int TASKS = Geo<DIM, L>::NGROUPS * RSP;
    static constexpr int PASSES = ceil_div(TASKS, RSP == 1 && TASKS <= 1024 ? 512 : 1024);
    static constexpr int TT = ceil_div(ceil_div(TASKS, PASSES), 32) * 32;
    static constexpr int NW = TT / 32;
};

// Byte j of lane 4k + i <- byte i of lane 4k + j.
__device__ __forceinline__ uint32_t bytes4x4(uint32_t v, int lane) {
    const uint32_t y = __shfl_xor_sync(0xffffffffu, v, 2);
    v = __byte_perm(v, y, (lane & 2) ? 0x3276 : 0x5410);
    const uint32_t z = __shfl_xor_sync(0xffffffffu, v, 1);
    return __byte_perm(v, z, (lane & 1) ? 0x3715 : 0x6240);
}

template <int DIM, int L, bool PMJ, int RSP, int RPQ, typename KT>
__device__ __forceinline__ void team_chunk(const RunDev& d, const SweepCtx& x, uint32_t b0,
                                           int nsweeps, uint32_t* S, uint4* RT, uint32_t* sums,
                                           const uint8_t* JS, const KT& K, long long& sAbsM,
                                           long long& sM2) {
    using G = Geo<DIM, L>;
    using TM = Team<DIM, L, RSP>;
    static_assert(RPQ == 8 || RSP == 4, "only four lanes per group take part of the chunk's bits");
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    // bit (and lane) 8 q + r is replica r of quarter q; r < RPQ
    const uint32_t slot = b0 + (uint32_t)(RPQ == 8 ? lane : (lane >> 3) * RPQ + (lane & 7));
    const bool valid = (RPQ == 8 || (lane & 7) < RPQ) && slot < x.R;
    const bool i8 = d.layout == PA_LAYOUT_INT8;
    uint8_t* rep = d.spins[x.cur] + (size_t)slot * d.stride;
#pragma unroll 1
    for (int u = wid; u < G::UNITS; u += TM::NW) load_unit<DIM, L>(rep, i8, d.stride, valid, S, u, lane);
    HalfSweep h = half_sweep(K, x.ctag, 2u * x.g0);
    if (wid == 0) {
        RT[rt_place(lane)] = replica_words(K, h, slot);
        sums[lane] = sums[32 + lane] = 0u;
    }
    __syncthreads();
    for (int hs = 0; hs < 2 * nsweeps; ++hs) {
        const uint4* rt = RT + 32 * (hs & 1);
#pragma unroll 1
        for (int p = 0; p < TM::PASSES; ++p) {
            const int task = t + p * TM::TT, k = task / RSP;
            if (RSP == 1 && task >= TM::TASKS) break;
            uint32_t acc[4][G::NCLS];
            const GroupWords g = group_words(K, h, (uint32_t)k);
            draw<G::NCLS, RSP == 1 ? 32 : RPQ>(K, g, rt, task % RSP, x.T, acc);
            if constexpr (RSP == 1) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    flip_site<DIM, L, PMJ>(S, JS, 4 * k + i, hs & 1, acc[i], x.full);
            } else {
                uint32_t mine[G::NCLS];
#pragma unroll
                for (int c = 0; c < G::NCLS; ++c) {
                    const uint32_t lo = __byte_perm(acc[0][c], acc[1][c], 0x0040);
                    const uint32_t hi = __byte_perm(acc[2][c], acc[3][c], 0x0040);
                    mine[c] = bytes4x4(__byte_perm(lo, hi, 0x5410), lane);
                }
                if (task < TM::TASKS) flip_site<DIM, L, PMJ>(S, JS, task, hs & 1, mine, x.full);
            }
        }
        // the next half-sweep's table goes to the other half of RT
        h = half_sweep(K, x.ctag, 2u * x.g0 + (uint32_t)hs + 1u);
        if (wid == 0) RT[32 * ((hs & 1) ^ 1) + rt_place(lane)] = replica_words(K, h, slot);
        __syncthreads();
    }
    uint32_t U, down;
    measure<DIM, L, PMJ, TM::TT>(S, JS, t, lane, U, down);
    if constexpr (TM::NW > 1) {
        atomicAdd(&sums[lane], U);
        atomicAdd(&sums[32 + lane], down);
    }
    if (nsweeps > 0)
#pragma unroll 1
        for (int u = wid; u < G::UNITS; u += TM::NW) store_unit<DIM, L>(rep, i8, valid, S, u, lane);
    __syncthreads();
    if (wid == 0) {
        if constexpr (TM::NW > 1) {
            U = sums[lane];
            down = sums[32 + lane];
        }
        record<G::N>(d, x, slot, valid, U, down, lane, sAbsM, sM2);
        __syncwarp();
    }
    // warp 0 alone writes sums and RT before the next chunk's first barrier, and
    // every warp is past its last read of S here
}

// Shared memory: RT entries, then 32-bit words.  Sizes in 16-byte units.
template <int DIM, int L>
__host__ __device__ constexpr int s_quads() {
    return ceil_div(Geo<DIM, L>::NS, 4);
}
template <int DIM, int L, bool PMJ>
__host__ __device__ constexpr int j_quads() {
    return PMJ ? ceil_div(Geo<DIM, L>::JWORDS, 4) : 0;
}

// --------------------------------------------------------------------------
// Host side of both forms
// --------------------------------------------------------------------------
struct KInfo {
    const void* fn;
    int threads;
    int smem;
    int replicas;  // of a chunk
};

// Lanes that share a group: 1 or 4 (RSP of team_chunk).  A lattice of fewer
// than 32 groups fills a warp only with 4, and a team of 7 warps (3D L = 12)
// loads one of the SM's four schedulers with one warp where the others have
// two: 1089 attempts/ns against 1207 with 4 (27 warps).
template <int DIM, int L>
constexpr bool always_four() {
    return Geo<DIM, L>::NGROUPS < 32 || (Team<DIM, L, 1>::NW > 4 && Team<DIM, L, 1>::NW % 4);
}

#define PA_SIZES(X) X(2, 4) X(2, 8) X(2, 16) X(2, 32) X(2, 64) X(2, 128) \
    X(3, 2) X(3, 4) X(3, 6) X(3, 8) X(3, 10) X(3, 12) X(3, 16)

inline int grid_for(const KInfo& k, int64_t need_blocks) {
    if (!k.fn) return 0;
    if (cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem) !=
        cudaSuccess)
        return 0;
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, k.threads, k.smem) != cudaSuccess)
        return 0;
    if (per_sm < 1) return 0;
    const int64_t full = (int64_t)sms * per_sm;
    if (need_blocks > 0 && need_blocks < full) return (int)need_blocks;
    return (int)full;
}

// One-lane warps (32 groups of a chunk) of the run's population, and the number
// of them from which one lane per group is the faster form.
constexpr int64_t FOUR_BELOW = 2432;
inline int64_t one_lane_warps(const RunDev& d) {
    return ((int64_t)d.R0 + 31) / 32 * ((d.N / 8 + 31) / 32);
}

}  // namespace
}  // namespace pa
