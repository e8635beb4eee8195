// pt_kernels.cu -- a6 + a7: parallel tempering (Sec. II, PT; Eq. "temperatureexchange").
//
// M replicas of every realization, one per temperature slot k (beta ascending with k, slot
// 0 hottest; every realization has its own temperature set).  Each sweep: a Metropolis sweep
// of every slot colour class by colour class (even L: the checkerboard, sites with even
// coordinate sum first; odd L: three colours, see pt_colour), then replica exchange between
// slots (k, k+1) for k = t mod 2, t mod 2 + 2, ..., then one round-trip check per replica
// (Sec. III, PT variant: between E_g and an energy typical of a high temperature, E_hot).
//
// Layout.  Realizations come in groups of 32 (realization id 32g + b is bit b); the
// configuration at slot k of a group is one multi-spin-coded word per site.  Exchanges move
// configurations (not temperatures) with masked XOR swaps of whole words.
//
// Acceptance.  For a site word the unsatisfied-bond count of every bit is a bit-sliced sum;
// bits with dE <= 0 flip.  Each uphill bit b compares its 32-bit random number r_b with its
// own threshold (slot k, its realization's beta_k, its class); r_b's bit 31-m is bit b of
// random word m (Philox4x32-10 of counter (8i + m/4, t, g, 4 | k<<8), word m&3), and the
// thresholds are stored the same way, as bit planes: plane m of class c holds bit 31-m of
// the 32 realizations' thresholds.  The comparison runs over planes from the most
// significant one: the first 8 without branches, the rest only while a bit is undecided.
//
// What bounds it.  A site word costs two Philox calls (40 wide multiplies at a quarter of the issue
// rate), about 40 operations of the comparison and 25 for its neighbours, most of them at half rate, so
// a batch that fills the SMs (L = 8, 1024 x 32: two CTAs on two SMs of three) is bound by those pipes;
// between the colour passes a CTA walks a chain of short steps (open comparisons, energies, exchange)
// whose latencies add up: 13 of 29 thousand cycles a sweep before they were shortened, 7 now.
// us per sweep, before -> now: 1024 x 32 of L = 8 15.9 -> 11.6 (1056 -> 1447 attempts/ns); 32 x 32 of
// L = 8 11.3 -> 6.7; 1024 x 14 of L = 6 7.4 -> 5.3; 128 x 20 of L = 12 35 -> 16; 333 x 12 of L = 5 6.7 ->
// 4.6; 256 x 17 of L = 7 36 -> 7.9.
//
// Parallel work.  One thread-block cluster per group: CS CTAs, each owning M/CS (rounded up) consecutive
// slots in shared memory; a thread keeps its sites (index, neighbours, bonds) and goes through
// the slots.  Energies come from the updates themselves (bit-sliced counts, warp bit-matrix
// transpose, popcount): for even L the unsatisfied bonds counted at the second colour's sites, for
// odd L the change at every site, instead of a pass over all bonds.  Exchanges between slots owned by
// different CTAs read and write the neighbour CTA's shared memory (distributed shared memory)
// between cluster barriers, all loads before the stores; a replica's round-trip record moves with it,
// so that the check after the exchange is local.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <type_traits>
#include <vector>

#include "eamc.h"
#include "eamc_ctx.cuh"
#include "eamc_internal.cuh"

namespace cg = cooperative_groups;
using namespace eamc;

struct PtRt {
    int32_t phase, n_rt;
    int64_t t_first, t_last;
    int32_t e_min, pad;
};

struct PtState {
    int dim = 0, L = 0, V = 0, nb = 0, M = 0, n_real = 0, n_groups = 0, cs = 1;
    uint32_t rid0 = 0;
    uint64_t t = 0;
    uint64_t t_win = 0;            // start of the exchange-count window (pt_adapt)
    uint32_t *d_spins = nullptr;   // [g][k][V]
    uint32_t *d_bonds = nullptr;   // [g][nb]
    int32_t *d_E = nullptr;        // [g][k][32]
    int32_t *d_label = nullptr;    // [g][k][32]
    PtRt *d_rt = nullptr;          // [g][label][32]
    int32_t *d_bounds = nullptr;   // [g][32][2] (e_g, e_hot)
    double *d_beta = nullptr;      // [g][k][32] inverse temperatures
    uint32_t *d_planes = nullptr;  // [g][k][32 planes][4] Metropolis thresholds (classes 0..2, pad)
    uint32_t *d_xacc = nullptr;    // [g][k][32] accepted exchanges of pair (k, k+1) in the window
    unsigned long long *d_swaps = nullptr;  // [M-1]
    int *d_err = nullptr;
};

namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) {
    return (a & b) | (a & c) | (b & c);
}

// 32x32 bit-matrix transpose across a warp: afterwards lane t holds, in bit s, bit t of what lane s
// held.  Stage j swaps the off-diagonal j x j blocks: a lane keeps the bits of mask k, and takes the
// others from its partner's word rotated by j (down where its own bit j is set): one shuffle, one
// rotation, one three-input operation a stage
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, int lane) {
    const uint32_t masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const int j = 16 >> s;
        const uint32_t keep = (lane & j) ? ~masks[s] : masks[s];
        const uint32_t y = __shfl_xor_sync(kFull, x, j);
        const uint32_t r = __funnelshift_l(y, y, (lane & j) ? 32 - j : j);
        x = (x & keep) | (r & ~keep);
    }
    return x;
}

constexpr int kTailQ = 32;  // open comparisons a warp defers per colour phase

template <int DIM, int L, bool WIDE = false>
struct PtGeo {
    static constexpr int NR = DIM == 3 ? L * L : L;
    static constexpr int V = NR * L;
    static constexpr int NB = DIM * V;
    static constexpr int HALF = V / 2;  // sites of one colour (even L)
    static constexpr bool ODD = (L & 1) != 0;
    // most sites of one colour, odd L: the axis colours 0, 1, 2 of L positions occur n0, n1, n2 times;
    // the fullest class of their DIM-fold sums mod 3
    static constexpr int axn(int c) {
        int n = 0;
        for (int x = 0; x < L; ++x) n += ((x == L - 1 && (L - 1) % 3 == 0) ? 1 : x % 3) == c;
        return n;
    }
    static constexpr int most_odd() {
        int best = 0;
        for (int c = 0; c < 3; ++c) {
            int n = 0;
            for (int a = 0; a < 3; ++a)
                for (int b = 0; b < 3; ++b) {
                    if (DIM == 3) n += axn(a) * axn(b) * axn(((c - a - b) % 3 + 3) % 3);
                    else if ((a + b) % 3 == c) n += axn(a) * axn(b);
                }
            best = n > best ? n : best;
        }
        return best;
    }
    static constexpr int NC = ODD ? most_odd() : HALF;
    // a block's threads: JT over the sites of a colour (whole warps, in NP passes where the sites are more
    // than MAX), times KT slots side by side.  At most 288 threads, two blocks to an SM; the wide form
    // (WIDE: at most 576, one block to an SM) is for batches whose CTAs have an SM each, which wait for
    // latencies, not for pipes
    static constexpr int MAX = WIDE ? 576 : 288;
    static constexpr int NP = (NC + MAX - 1) / MAX;
    static constexpr int JT = ((NC + NP - 1) / NP + 31) / 32 * 32;
    static constexpr int KT_MAX = WIDE ? MAX / JT : (JT > 128 ? 1 : 256 / JT);
    static __host__ __device__ constexpr int kt(int spc) { return spc < KT_MAX ? spc : KT_MAX; }
    static __host__ __device__ constexpr int threads(int spc) { return JT * kt(spc); }
    static constexpr size_t smem(int spc) {
        return (size_t)(spc * 128 + spc * V + NB + spc * 32 * 2 + spc + (threads(spc) / 32) * (kTailQ * 6 + spc * 32) +
                        spc * 32 + 64 + 1 + 2 * spc * 32 + spc * 32 * (int)(sizeof(PtRt) / 4) + (ODD ? V + 4 : 0)) * 4;
    }
};

// neighbour of site i along axis d (0 x, 1 y, 2 z), direction +1 / -1
template <int DIM, int L>
__device__ __forceinline__ int pt_nbr(int i, int d, int sgn) {
    int x = i % L, y = (i / L) % L, z = DIM == 3 ? i / (L * L) : 0;
    if (d == 0) x = (x + sgn + L) % L;
    else if (d == 1) y = (y + sgn + L) % L;
    else z = (z + sgn + L) % L;
    return x + L * (y + L * z);
}

// Colour of a site for the PT sweep.  Even L: (x + y + z) mod 2.  Odd L: the sum of per-axis
// colours mod 3, an axis position x having colour x mod 3 except the last one (x = L-1) when
// L = 1 (mod 3), which takes 1 so that it differs from both neighbours L-2 and 0; a step to a
// neighbour then changes the sum by 1 or 2 (mod 3), so no two neighbours share a colour.
template <int DIM, int L>
__device__ __forceinline__ int pt_colour(int i) {
    const int x = i % L, y = (i / L) % L, z = DIM == 3 ? i / (L * L) : 0;
    if constexpr ((L & 1) == 0) {
        return (x + y + z) & 1;
    } else {
        auto ax = [](int c) { return (c == L - 1 && (L - 1) % 3 == 0) ? 1 : c % 3; };
        return (ax(x) + ax(y) + (DIM == 3 ? ax(z) : 0)) % 3;
    }
}

__device__ __forceinline__ uint32_t quantize_prob(double p) {
    if (p >= 1.0) return kAlways;
    const double q = floor(p * 4294967296.0);
    return (q >= 4294967294.0) ? 0xFFFFFFFEu : (uint32_t)q;
}

struct PtArgs {
    uint32_t *spins;
    const uint32_t *bonds;
    int32_t *E;
    int32_t *label;
    PtRt *rt;
    const int32_t *bounds;
    const uint32_t *planes;
    const double *beta;
    uint32_t *xacc;
    unsigned long long *swaps;
    int M, spc, n_real;
    uint32_t rid0;
    uint64_t t0, n_sweeps;
    int count_rt;
    PhiloxKey key;
};

template <int DIM, int L, bool WIDE>
__global__ void __launch_bounds__(PtGeo<DIM, L, WIDE>::MAX, WIDE ? 1 : 2) pt_kernel(PtArgs a) {
    using G = PtGeo<DIM, L, WIDE>;
    constexpr int V = G::V, NB = G::NB, HALF = G::HALF;
    constexpr bool ODD = G::ODD;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int g = blockIdx.x / (int)cluster.num_blocks();
    const int spc = a.spc, k0 = rank * spc, M = a.M;
    // slots of this CTA: the last one may have fewer than spc, and sweeps empty ones (zeroed) for the rest
    const int mine = min(spc, M - k0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;

    constexpr int NCOL = (L & 1) ? 3 : 2;
    extern __shared__ __align__(16) uint32_t sm[];
    uint4 *P = reinterpret_cast<uint4 *>(sm);  // [spc][32] threshold planes (class 0, 1, 2, pad)
    uint32_t *S = sm + spc * 128;           // [spc][V]
    uint32_t *J = S + spc * V;              // [NB], J[i*DIM + d]
    int32_t *Es = (int32_t *)(J + NB);      // [spc][32]
    int32_t *Ls = Es + spc * 32;            // [spc][32]
    uint32_t *Amask = (uint32_t *)(Ls + spc * 32);  // [spc] exchange masks of owned pairs
    // per-warp queue of site words whose comparison is still open after 8 planes:
    // [nwarps][kTailQ] x (site | slot << 16, acc, und, C0, C1, C2)
    uint32_t *TQ = Amask + spc;
    int32_t *Ep = (int32_t *)(TQ + nwarps * kTailQ * 6);   // [nwarps][spc][32] partial counts
    uint32_t *Xc = (uint32_t *)(Ep + nwarps * spc * 32);  // [spc][32] accepted exchanges, this launch
    int32_t *Bd = (int32_t *)(Xc + spc * 32);             // [32][2] round-trip bounds (e_g, e_hot)
    double *Db = reinterpret_cast<double *>((reinterpret_cast<uintptr_t>(Bd + 64) + 7) & ~uintptr_t(7));  // [spc][32]
    // round-trip records of the replicas in the CTA's slots, for the launch; an exchange moves them with
    // the configurations
    PtRt *Rh = reinterpret_cast<PtRt *>(Db + spc * 32);    // [spc][32]
    int32_t *Cl = (int32_t *)(Rh + spc * 32);  // odd L: sites by colour [V], then offsets [4]

    const uint32_t group_rid0 = a.rid0 + 32u * (uint32_t)g;
    const int nvalid = min(32, a.n_real - 32 * g);
    const uint32_t valid = nvalid >= 32 ? kFull : ((1u << nvalid) - 1u);

    for (int k = tid; k < spc * V; k += blockDim.x)
        S[k] = k < mine * V ? a.spins[((size_t)g * M + k0) * V + k] : 0u;
    for (int k = tid; k < NB; k += blockDim.x) J[k] = a.bonds[(size_t)g * NB + k];
    for (int k = tid; k < mine * 32; k += blockDim.x) {
        Es[k] = a.E[((size_t)g * M + k0) * 32 + k];
        const int label = a.label[((size_t)g * M + k0) * 32 + k];
        Ls[k] = label;
        Rh[k] = a.rt[((size_t)g * M + label) * 32 + (k & 31)];
    }
    for (int k = tid; k < spc * 128; k += blockDim.x)
        sm[k] = k < mine * 128 ? a.planes[((size_t)g * M + k0) * 128 + k] : 0u;
    // per launch: beta_{k+1} - beta_k of every owned pair and realization, the round-trip bounds,
    // zeroed exchange counters (added to the global ones at the end)
    for (int q = tid; q < mine * 32; q += blockDim.x) {
        const int k = k0 + (q >> 5), b = q & 31;
        Db[q] = (k + 1 < M) ? a.beta[((size_t)g * M + k + 1) * 32 + b] - a.beta[((size_t)g * M + k) * 32 + b] : 0.0;
        Xc[q] = 0u;
    }
    for (int q = tid; q < 64; q += blockDim.x) Bd[q] = a.bounds[(size_t)g * 64 + q];
    if constexpr ((L & 1) != 0) {
        if (tid == 0) {  // colour classes in lexicographic order (a few thousand steps per launch)
            int n = 0;
            for (int c = 0; c < NCOL; ++c) {
                Cl[V + c] = n;
                for (int i = 0; i < V; ++i)
                    if (pt_colour<DIM, L>(i) == c) Cl[n++] = i;
            }
            Cl[V + NCOL] = n;
        }
    }
    __syncthreads();
    cluster.sync();

    // this thread's sites of a colour are jt, jt + JT, ..., its slots kt, kt + KT, ...
    const int KT = G::kt(spc), jt = tid % G::JT, kt = tid / G::JT;
    const int nk = (spc + KT - 1) / KT;
    for (uint64_t s = 0; s < a.n_sweeps; ++s) {
        const uint64_t t = a.t0 + s;
        const uint32_t tt = (uint32_t)t;
        // ---- checkerboard Metropolis sweep of every owned slot
        // planes 8..31 of one site word: 8..15 together (two calls side by side decide all but about
        // 2^-8 of the words that come here), the rest while a bit is still undecided
        auto finish = [&](int i, int ks, uint32_t C0, uint32_t C1, uint32_t C2, uint32_t acc, uint32_t und) {
            const uint32_t c2 = (uint32_t)g + (a.rid0 >> 5), c3 = 4u | ((uint32_t)(k0 + ks) << 8);
            const uint4 *Pk = P + ks * 32;
            auto planes = [&](const uint4 &w, int m0) {
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const uint32_t R = uint4_get(w, m);
                    const uint4 q = Pk[m0 + m];
                    const uint32_t Tm = (C0 & q.x) | (C1 & q.y) | (C2 & q.z);
                    acc |= und & ~R & Tm;
                    und &= ~(R ^ Tm);
                }
            };
            const uint4 wa = philox4x32_10(make_uint4((uint32_t)(8 * i + 2), tt, c2, c3), a.key);
            const uint4 wb = philox4x32_10(make_uint4((uint32_t)(8 * i + 3), tt, c2, c3), a.key);
            planes(wa, 8);
            planes(wb, 12);
#pragma unroll 1
            for (int m = 16; m < 32 && und; m += 4)
                planes(philox4x32_10(make_uint4((uint32_t)(8 * i + (m >> 2)), tt, c2, c3), a.key), m);
            return acc;
        };
        uint32_t *tq = TQ + warp * kTailQ * 6;
        for (int colour = 0; colour < NCOL; ++colour) {
            const int nc = ODD ? Cl[V + colour + 1] - Cl[V + colour] : HALF;
            // site words of one colour never neighbour each other, so a word whose comparison
            // is still open after 8 planes (about 6 % of them) can be finished after the others:
            // the warp queues them and finishes them together, one per lane
            int nq = 0;
            for (int pass = 0; pass < G::NP; ++pass) {
                const int j = jt + pass * G::JT;
                const bool site = j < nc;
                // the site, its neighbours and its bonds: the same for every slot
                int i = 0;
                if constexpr (!ODD) {
                    const int row = site ? j / (L / 2) : 0, xh = site ? j % (L / 2) : 0;
                    const int y = row % L, z = DIM == 3 ? row / L : 0;
                    i = 2 * xh + ((colour + y + z) & 1) + L * row;
                } else {
                    if (site) i = Cl[Cl[V + colour] + j];
                }
                int nb[2 * DIM];
                uint32_t jw[2 * DIM];
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    nb[2 * d] = pt_nbr<DIM, L>(i, d, +1);
                    nb[2 * d + 1] = pt_nbr<DIM, L>(i, d, -1);
                    jw[2 * d] = J[i * DIM + d];
                    jw[2 * d + 1] = J[nb[2 * d + 1] * DIM + d];
                }
                const uint32_t c2 = (uint32_t)g + (a.rid0 >> 5);
                for (int it = 0; it < nk; ++it) {
                    const int ks = kt + it * KT;
                    const bool act = site && ks < spc;
                    uint32_t *Sk = S + (act ? ks : 0) * V;
                    const uint32_t si = Sk[i];
                    uint32_t u[2 * DIM];
#pragma unroll
                    for (int d = 0; d < 2 * DIM; ++d) u[d] = si ^ Sk[nb[d]] ^ jw[d];
                    uint32_t n0, n1, n2;  // bit-sliced count of unsatisfied bonds
                    if constexpr (DIM == 3) {
                        const uint32_t s1 = u[0] ^ u[1] ^ u[2], c1 = maj3(u[0], u[1], u[2]);
                        const uint32_t s2 = u[3] ^ u[4] ^ u[5], d1 = maj3(u[3], u[4], u[5]);
                        n0 = s1 ^ s2;
                        const uint32_t c3 = s1 & s2;
                        n1 = c1 ^ d1 ^ c3;
                        n2 = maj3(c1, d1, c3);
                    } else {
                        const uint32_t s1 = u[0] ^ u[1] ^ u[2], c1 = maj3(u[0], u[1], u[2]);
                        n0 = s1 ^ u[3];
                        const uint32_t d1 = s1 & u[3];
                        n1 = c1 ^ d1;
                        n2 = c1 & d1;
                    }
                    // uphill classes: n < DIM unsatisfied bonds (dE = 2*(2*DIM) - 4n > 0)
                    uint32_t C[3];
                    C[0] = ~n2 & ~n1 & ~n0;
                    C[1] = ~n2 & ~n1 & n0;
                    C[2] = (DIM == 3) ? (~n2 & n1 & ~n0) : 0u;
                    const uint32_t up = C[0] | C[1] | C[2];
                    uint32_t acc = ~up;  // dE <= 0 always accepted
                    uint32_t und = act ? up & valid : 0u;
                    const uint4 *Pk = P + (act ? ks : 0) * 32;
                    // the 8 most significant planes come from two independent Philox calls and are
                    // compared without branches; planes 8..31 are drawn only while a bit is still
                    // undecided (about 2^-8 per uphill bit)
                    const uint32_t c3 = 4u | ((uint32_t)(k0 + ks) << 8);
                    const uint4 wa = philox4x32_10(make_uint4((uint32_t)(8 * i), tt, c2, c3), a.key);
                    const uint4 wb = philox4x32_10(make_uint4((uint32_t)(8 * i + 1), tt, c2, c3), a.key);
                    const uint32_t Rm[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
                    // from the least significant of the eight: less = (r < threshold) on the bits so far, one
                    // three-input operation a plane (below: r bit 0, threshold bit 1; equal: as before)
                    uint32_t less = 0u, same = und;
#pragma unroll
                    for (int m = 7; m >= 0; --m) {
                        const uint4 q = Pk[m];
                        const uint32_t Tm = (C[0] & q.x) | (C[1] & q.y) | (C[2] & q.z);
                        less = (~Rm[m] & Tm) | (~(Rm[m] ^ Tm) & less);
                        same &= ~(Rm[m] ^ Tm);
                    }
                    acc |= und & less;
                    und = same;
                    const bool open = und != 0u;
                    const uint32_t om = __ballot_sync(kFull, open);
                    const int pos = nq + __popc(om & ((1u << lane) - 1u));
                    const bool deferred = open && pos < kTailQ;
                    if (deferred) {
                        uint32_t *e = tq + pos * 6;
                        e[0] = (uint32_t)i | ((uint32_t)ks << 16);
                        e[1] = acc;
                        e[2] = und;
                        e[3] = C[0];
                        e[4] = C[1];
                        e[5] = C[2];
                    } else if (act) {
                        if (open) acc = finish(i, ks, C[0], C[1], C[2], acc, und);  // queue full
                        Sk[i] = si ^ (acc & valid);
                    }
                    nq += __popc(om);
                    // the slot's energy from the updates.  Even L: every bond has one end of the second
                    // colour, so the unsatisfied bonds are the sum of n over its sites, after the update
                    // (2 DIM - n where the spin flipped).  Odd L: the sum over all sites of 2 DIM - n where it
                    // flipped and DIM where not, the change against all DIM.  A deferred word counts with the
                    // bits decided so far.
                    if (ODD || colour == 1) {
                        const uint32_t in = act ? kFull : 0u, f = acc & valid & in;
                        const uint32_t r0 = n0, r1 = DIM == 3 ? n1 ^ ~n0 : n1 ^ n0;  // 2 DIM - n
                        const uint32_t r2 = DIM == 3 ? ~n2 & ~(n1 & n0) : ~n2 & ~n1 & ~n0;
                        uint32_t m0, m1, m2;
                        if constexpr (ODD) {
                            m0 = (f & r0) | (DIM == 3 ? ~f : 0u);
                            m1 = (f & r1) | ~f;
                            m2 = f & r2;
                        } else {
                            m0 = n0;
                            m1 = (f & r1) | (~f & n1);
                            m2 = (f & r2) | (~f & n2);
                        }
                        const int part = __popc(warp_transpose(m0 & in, lane)) + 2 * __popc(warp_transpose(m1 & in, lane)) +
                                         4 * __popc(warp_transpose(m2 & in, lane));
                        if (ks < spc) {
                            int32_t *e = Ep + ((jt >> 5) * spc + ks) * 32 + lane;
                            *e = (pass == 0 && (!ODD || colour == 0)) ? part : *e + part;
                        }
                    }
                }
            }
            __syncwarp();
            for (int e0 = 0; e0 < min(nq, kTailQ); e0 += 32) {
                const int e = e0 + lane;
                if (e < min(nq, kTailQ)) {
                    const uint32_t *q = tq + e * 6;
                    const int i = (int)(q[0] & 0xFFFFu), ks = (int)(q[0] >> 16);
                    const uint32_t acc = finish(i, ks, q[3], q[4], q[5], q[1], q[2]);
                    S[ks * V + i] ^= acc & valid;
                    if (ODD || colour == 1) {  // bits accepted only now
                        uint32_t late = acc & ~q[1] & valid;
                        while (late) {
                            const int b = __ffs(late) - 1;
                            late &= late - 1u;
                            const int n = (int)((q[4] >> b) & 1u) + 2 * (int)((q[5] >> b) & 1u);
                            atomicAdd(&Ep[((jt >> 5) * spc + ks) * 32 + b], ODD ? DIM - n : 2 * DIM - 2 * n);
                        }
                    }
                }
            }
            __syncthreads();
        }
        // ---- energies of the owned slots from the warps' sums
        for (int k = tid; k < mine * 32; k += blockDim.x) {
            int u = 0;
#pragma unroll
            for (int w = 0; w < G::JT / 32; ++w) u += Ep[w * spc * 32 + k];
            Es[k] = ODD ? Es[k] + 4 * (u - DIM * V) : 2 * u - NB;
        }
        cluster.sync();  // every slot's energy is known (and a barrier of this CTA)
        // ---- replica exchange between (k, k+1), k = t mod 2 (mod 2); the owner of k decides,
        //      one warp per owned pair ks0, ks0 + 2, ...
        const int ks0 = (k0 ^ (int)t) & 1;
        const int np = max(0, (min(spc, M - 1 - k0) - ks0 + 1) / 2);
        for (int p = warp; p < np; p += nwarps) {
            const int ks = ks0 + 2 * p, k = k0 + ks;
            const int kr = (ks + 1 < spc) ? rank : rank + 1;
            const int ksr = (ks + 1 < spc) ? ks + 1 : 0;
            const int32_t *Er = cluster.map_shared_rank(Es, kr);
            const int e0 = Es[ks * 32 + lane], e1 = Er[ksr * 32 + lane];
            const uint4 w = philox4x32_10(make_uint4((uint32_t)k, tt, group_rid0 + lane, 1u), a.key);
            bool ok = true;
            if (e1 < e0) {
                // Eq. "temperatureexchange" with this realization's beta_k, beta_k+1: accepted with
                // p = exp(-x), quantised to 32 bits.  In single precision p is known to 1e-5; the exact
                // threshold (FP64, 32 times slower) is needed only where the word lies that close to it
                const int d4 = (e0 - e1) / 4;
                const float x = (float)Db[ks * 32 + lane] * (4.0f * (float)d4), pf = expf(-x) * 4294967296.0f, wf = (float)w.x;
                const float slack = (2e-6f + 1e-6f * x) * pf + 1e-6f * wf + 4.0f;
                ok = wf < pf;
                if (!(fabsf(wf - pf) > slack)) {
                    const uint32_t th = quantize_prob(exp(-Db[ks * 32 + lane] * 4.0 * (double)d4));
                    ok = (th == kAlways) || (w.x < th);
                }
            }
            const uint32_t A = __ballot_sync(kFull, ok) & valid;
            Xc[ks * 32 + lane] += (A >> lane) & 1u;
            if (lane == 0) Amask[ks] = A;
        }
        __syncthreads();
        // the configurations, energies, labels and records of the accepted pairs change places; the pairs
        // are disjoint, and all loads of a round (the neighbour CTA's shared memory) come before its stores
        {
            constexpr int VQ = (V % 4 == 0) ? 4 : 1;  // words per access
            constexpr int Q = V / VQ;
            using W = typename std::conditional<VQ == 4, uint4, uint32_t>::type;
            const int ne = np * 32, nw = np * Q;
            for (int e = tid; e < max(nw, ne); e += blockDim.x) {
                W a0, b0, *pa = nullptr, *pb = nullptr;
                uint32_t A = 0u;
                if (e < nw) {
                    const int ks = ks0 + 2 * (e / Q), i = e % Q;
                    A = Amask[ks];
                    if (A) {
                        const bool far = ks + 1 >= spc;
                        pa = reinterpret_cast<W *>(S + ks * V) + i;
                        pb = reinterpret_cast<W *>(far ? cluster.map_shared_rank(S, rank + 1) : S + (ks + 1) * V) + i;
                        a0 = *pa;
                        b0 = *pb;
                    }
                }
                bool moves = false;
                int q0 = 0, q1 = 0, kr = rank;
                int32_t ea = 0, eb = 0, la = 0, lb = 0;
                PtRt ra, rb;
                if (e < ne) {
                    const int ks = ks0 + 2 * (e >> 5), bit = e & 31;
                    moves = ((Amask[ks] >> bit) & 1u) != 0u;
                    if (moves) {
                        kr = (ks + 1 < spc) ? rank : rank + 1;
                        q0 = ks * 32 + bit;
                        q1 = ((ks + 1 < spc) ? ks + 1 : 0) * 32 + bit;
                        ea = Es[q0];
                        la = Ls[q0];
                        ra = Rh[q0];
                        eb = cluster.map_shared_rank(Es, kr)[q1];
                        lb = cluster.map_shared_rank(Ls, kr)[q1];
                        rb = cluster.map_shared_rank(Rh, kr)[q1];
                    }
                }
                if (A) {
                    if constexpr (VQ == 4) {
                        const uint4 d = make_uint4((a0.x ^ b0.x) & A, (a0.y ^ b0.y) & A, (a0.z ^ b0.z) & A, (a0.w ^ b0.w) & A);
                        *pa = make_uint4(a0.x ^ d.x, a0.y ^ d.y, a0.z ^ d.z, a0.w ^ d.w);
                        *pb = make_uint4(b0.x ^ d.x, b0.y ^ d.y, b0.z ^ d.z, b0.w ^ d.w);
                    } else {
                        const uint32_t d = (a0 ^ b0) & A;
                        *pa = a0 ^ d;
                        *pb = b0 ^ d;
                    }
                }
                if (moves) {
                    Es[q0] = eb;
                    Ls[q0] = lb;
                    Rh[q0] = rb;
                    cluster.map_shared_rank(Es, kr)[q1] = ea;
                    cluster.map_shared_rank(Ls, kr)[q1] = la;
                    cluster.map_shared_rank(Rh, kr)[q1] = ra;
                }
            }
        }
        cluster.sync();  // exchanges complete everywhere
        // ---- round trips / lowest energy per replica; its record travels with it
        for (int q = tid; q < mine * 32; q += blockDim.x) {
            const int b = q & 31;
            if (!((valid >> b) & 1u)) continue;
            const int E = Es[q];
            PtRt &r = Rh[q];
            if (E < r.e_min) r.e_min = E;
            if (a.count_rt) {
                const int eg = Bd[2 * b + 0];
                const int ehot = Bd[2 * b + 1];
                if (r.phase == 0) {
                    if (E >= ehot) { r.t_first = (int64_t)t; r.phase = 1; }
                } else if (r.phase == 1) {
                    if (E <= eg) r.phase = 2;
                } else {
                    if (E >= ehot) { r.n_rt += 1; r.t_last = (int64_t)t; r.phase = 1; }
                }
            }
        }
        // (the next sweep writes energies, labels and records only after further barriers)
    }
    __syncthreads();
    // ---- write back; a replica's record to its label
    for (int q = tid; q < mine * 32; q += blockDim.x) a.rt[((size_t)g * M + Ls[q]) * 32 + (q & 31)] = Rh[q];
    for (int q = tid; q < mine * 32; q += blockDim.x) {
        const int k = k0 + (q >> 5);
        if (Xc[q]) {
            a.xacc[((size_t)g * M + k) * 32 + (q & 31)] += Xc[q];
            atomicAdd(&a.swaps[k], (unsigned long long)Xc[q]);
        }
    }
    for (int k = tid; k < mine * V; k += blockDim.x) a.spins[((size_t)g * M + k0) * V + k] = S[k];
    for (int k = tid; k < mine * 32; k += blockDim.x) {
        a.E[((size_t)g * M + k0) * 32 + k] = Es[k];
        a.label[((size_t)g * M + k0) * 32 + k] = Ls[k];
    }
    cluster.sync();
}

// initial state: couplings and per-slot random spins from the seed (or the caller), energies
// by full recomputation, labels = slot.  One warp per (group, slot).
template <int DIM, int L>
__global__ void pt_init_kernel(uint32_t *spins, uint32_t *bonds, int32_t *E, int32_t *label,
                               const int8_t *Jin, int M, int n_real, uint32_t rid0, PhiloxKey key) {
    using G = PtGeo<DIM, L>;
    constexpr int V = G::V, NB = G::NB;
    const int g = blockIdx.x / M, k = blockIdx.x % M, lane = threadIdx.x;
    const uint32_t rid = rid0 + 32u * g + lane;
    const bool act = (int)(32 * g + lane) < n_real;
    uint32_t *sp = spins + ((size_t)g * M + k) * V;
    uint32_t *bd = bonds + (size_t)g * NB;
    if (k == 0) {
        for (int j0 = 0; j0 < NB; j0 += 4) {
            const uint4 w = philox4x32_10(make_uint4((uint32_t)(j0 >> 2), 0u, rid, 3u), key);
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                const int j = j0 + jj;
                if (j < NB) {
                    const bool neg = act && (Jin ? (Jin[(size_t)(32 * g + lane) * NB + j] < 0)
                                                 : ((uint4_get(w, jj) >> 31) != 0));
                    const uint32_t m = __ballot_sync(kFull, neg);
                    if (lane == 0) bd[j] = m;
                }
            }
        }
    }
    for (int i0 = 0; i0 < V; i0 += 4) {
        const uint4 w = philox4x32_10(make_uint4((uint32_t)(i0 >> 2), 0u, rid, 2u | ((uint32_t)k << 8)), key);
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            const int i = i0 + jj;
            if (i < V) {
                const bool neg = act && ((uint4_get(w, jj) >> 31) != 0);
                const uint32_t m = __ballot_sync(kFull, neg);
                if (lane == 0) sp[i] = m;
            }
        }
    }
    label[((size_t)g * M + k) * 32 + lane] = k;
}

// energies of every (group, slot) from scratch; one warp per (group, slot)
template <int DIM, int L>
__global__ void pt_energy_kernel(const uint32_t *spins, const uint32_t *bonds, int32_t *E, int M) {
    using G = PtGeo<DIM, L>;
    constexpr int V = G::V, NB = G::NB;
    const int g = blockIdx.x / M, k = blockIdx.x % M, lane = threadIdx.x;
    const uint32_t *sp = spins + ((size_t)g * M + k) * V;
    const uint32_t *bd = bonds + (size_t)g * NB;
    int u = 0;
    for (int i = 0; i < V; ++i)
        for (int d = 0; d < DIM; ++d) {
            const uint32_t w = sp[i] ^ sp[pt_nbr<DIM, L>(i, d, +1)] ^ bd[i * DIM + d];
            u += (w >> lane) & 1u;
        }
    E[((size_t)g * M + k) * 32 + lane] = 2 * u - NB;
}

template <int DIM, int L, bool WIDE>
cudaError_t pt_launch_sweeps(const PtState *p, const PtArgs &a, cudaStream_t st) {
    using G = PtGeo<DIM, L, WIDE>;
    const int threads = G::threads(a.spc);
    const size_t smem = G::smem(a.spc);
    cudaError_t e = cudaFuncSetAttribute(pt_kernel<DIM, L, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBlockSmemMax);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(pt_kernel<DIM, L, WIDE>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(p->n_groups * p->cs);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p->cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, pt_kernel<DIM, L, WIDE>, a);
}

template <int DIM, int L>
cudaError_t pt_launch_all(PtState *p, const int8_t *dJ, ea_ctx *ctx, int what, uint64_t n_sweeps,
                          int count_rt) {
    using G = PtGeo<DIM, L>;
    if (what == 0) {
        pt_init_kernel<DIM, L><<<p->n_groups * p->M, 32, 0, ctx->stream>>>(
            p->d_spins, p->d_bonds, p->d_E, p->d_label, dJ, p->M, p->n_real, p->rid0, ctx->key);
        pt_energy_kernel<DIM, L><<<p->n_groups * p->M, 32, 0, ctx->stream>>>(p->d_spins, p->d_bonds, p->d_E, p->M);
        return cudaGetLastError();
    }
    PtArgs a;
    a.spins = p->d_spins;
    a.bonds = p->d_bonds;
    a.E = p->d_E;
    a.label = p->d_label;
    a.rt = p->d_rt;
    a.bounds = p->d_bounds;
    a.planes = p->d_planes;
    a.beta = p->d_beta;
    a.xacc = p->d_xacc;
    a.swaps = p->d_swaps;
    a.M = p->M;
    a.spc = (p->M + p->cs - 1) / p->cs;
    a.n_real = p->n_real;
    a.rid0 = p->rid0;
    a.t0 = p->t;
    a.n_sweeps = n_sweeps;
    a.count_rt = count_rt;
    a.key = ctx->key;
    // the wide form from 3D L = 8 while the clusters fit the SMs with a CTA to each (a cluster of 8 stays
    // within a GPC: 15 of them fit, so the line is three quarters of the SMs).  us per sweep, narrow ->
    // wide: L = 8, 448 x 32 7.16 -> 6.75; L = 9, 64 x 32 12.5 -> 11.6; L = 10, 256 x 14 8.0 -> 6.9; L = 11,
    // 128 x 20 21.0 -> 17.4; L = 12, 448 x 32 24.3 -> 20.0.  Beyond the line two narrow CTAs share an SM:
    // L = 8, 512 x 32 10.6 (wide 13.4); L = 9, 608 x 32 19.4 (25.0).  Below L = 8 the sites of a colour fill
    // 128 threads at most and slots lie side by side already: L = 6, 200 x 32 4.75 (5.17), L = 7, 448 x 20
    // 8.0 (8.3)
    if constexpr (DIM == 3 && L >= 8) {
        using W = PtGeo<DIM, L, true>;
        if (4 * p->n_groups * p->cs <= 3 * ctx->n_sm && W::threads(a.spc) > G::threads(a.spc) &&
            W::smem(a.spc) <= kBlockSmemMax)
            return pt_launch_sweeps<DIM, L, true>(p, a, ctx->stream);
    }
    return pt_launch_sweeps<DIM, L, false>(p, a, ctx->stream);
}

cudaError_t pt_dispatch(PtState *p, const int8_t *dJ, ea_ctx *ctx, int what, uint64_t n_sweeps, int count_rt) {
#define PT_CASE(D, LL) \
    if (p->dim == D && p->L == LL) return pt_launch_all<D, LL>(p, dJ, ctx, what, n_sweeps, count_rt);
    PT_CASE(3, 3) PT_CASE(3, 4) PT_CASE(3, 5) PT_CASE(3, 6) PT_CASE(3, 7) PT_CASE(3, 8) PT_CASE(3, 9)
    PT_CASE(3, 10) PT_CASE(3, 11) PT_CASE(3, 12)
    PT_CASE(2, 3) PT_CASE(2, 4) PT_CASE(2, 5) PT_CASE(2, 6) PT_CASE(2, 7) PT_CASE(2, 8) PT_CASE(2, 9)
    PT_CASE(2, 10) PT_CASE(2, 11) PT_CASE(2, 12)
#undef PT_CASE
    return cudaErrorInvalidValue;
}

// what a CTA of spc slots takes: passes over them in a colour, and shared memory (the narrow form)
struct PtForm {
    int passes = 0;
    size_t smem = 0;
};
PtForm pt_form(int dim, int L, int spc) {
#define PT_CASE(D, LL) \
    if (dim == D && L == LL) return {(spc + PtGeo<D, LL>::kt(spc) - 1) / PtGeo<D, LL>::kt(spc), PtGeo<D, LL>::smem(spc)};
    PT_CASE(3, 3) PT_CASE(3, 4) PT_CASE(3, 5) PT_CASE(3, 6) PT_CASE(3, 7) PT_CASE(3, 8) PT_CASE(3, 9)
    PT_CASE(3, 10) PT_CASE(3, 11) PT_CASE(3, 12)
    PT_CASE(2, 3) PT_CASE(2, 4) PT_CASE(2, 5) PT_CASE(2, 6) PT_CASE(2, 7) PT_CASE(2, 8) PT_CASE(2, 9)
    PT_CASE(2, 10) PT_CASE(2, 11) PT_CASE(2, 12)
#undef PT_CASE
    return {};
}

// CTAs per realization group, at most 8 (clusters of 16 measured slower): the largest number that divides
// the slots, or the one with the fewest slots to a CTA, whose last CTA sweeps some empty ones.  A sweep
// takes about passes x max(1, CTAs / SMs); the second has to win by a quarter, as empty slots and smaller
// blocks cost it up to that.  us per sweep, dividing -> fewest: M = 17, L = 7, 256 realizations 23.7 -> 7.9;
// L = 8, 1024 28.7 -> 8.8; L = 12, 256 104 -> 18; L = 4, 1024 6.0 -> 3.7; M = 20, L = 10, 256 13.7 -> 10.8;
// M = 13, L = 8, 600 21.0 -> 6.8.  Left dividing: M = 17, L = 4, 8192 9.5 (11.2); M = 20, L = 6, 1024 6.8
// (7.5), L = 8, 2048 16.6 (17.4).  A dividing split whose slots exceed a block's shared memory (a prime M
// of the larger lattices keeps them all in one block) is none; the fewest slots, 8 at most, always fit.
int pt_cluster(int dim, int L, int M, int n_groups, int n_sm) {
    int even = 1;
    for (int c = 8; c >= 2 && even == 1; --c)
        if (M % c == 0) even = c;
    const int spc = (M + 7) / 8, least = (M + spc - 1) / spc;
    if (pt_form(dim, L, M / even).smem > kBlockSmemMax) return least;
    auto cost = [&](int cs) {
        return (long long)pt_form(dim, L, (M + cs - 1) / cs).passes * std::max((long long)n_sm, (long long)n_groups * cs);
    };
    return 4 * cost(even) >= 5 * cost(least) ? least : even;
}

// Metropolis threshold planes of every (group, slot): one warp, lane b = realization bit.
// Class n (n unsatisfied bonds, dE = 2z - 4n > 0) accepts with exp(-beta dE) (Sec. II, PT).
__global__ void pt_planes_kernel(const double *__restrict__ beta, int dim, uint32_t *__restrict__ planes) {
    const int gk = blockIdx.x, lane = threadIdx.x;
    const int z = 2 * dim;
    const double b = beta[(size_t)gk * 32 + lane];
    uint32_t thr[3];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
        const int dE = 2 * z - 4 * n;
        thr[n] = (dE <= 0) ? kAlways : quantize_prob(exp(-b * (double)dE));
    }
    uint32_t *out = planes + (size_t)gk * 128;
    for (int m = 0; m < 32; ++m) {
        const int sh = 31 - m;
        const uint32_t p0 = __ballot_sync(kFull, (thr[0] >> sh) & 1u);
        const uint32_t p1 = __ballot_sync(kFull, (thr[1] >> sh) & 1u);
        const uint32_t p2 = __ballot_sync(kFull, (thr[2] >> sh) & 1u);
        if (lane == 0) {
            out[4 * m + 0] = p0;
            out[4 * m + 1] = p1;
            out[4 * m + 2] = p2;
            out[4 * m + 3] = 0u;
        }
    }
}

constexpr int kMaxSlots = 64;

// One step of the constant-exchange-rate adaptation (Sec. II, PT: the temperatures of every
// realization are moved during equilibration until its exchange rates are equal).  One thread
// per realization.  Pair k accepted xacc of att_k attempts in the window: rate A_k clamped to
// [0.005, 0.995], stiffness s_k = -ln A_k / D_k of its gap D_k; the gaps that equalise the rates
// are D*_k = span (1/s_k) / sum_j (1/s_j); new gaps (1 - eta) D_k + eta D*_k, end points fixed.
// A pair without attempts leaves the realization unchanged.  Counts of the window are cleared.
__global__ void pt_adapt_kernel(double *__restrict__ beta, uint32_t *__restrict__ xacc, int M, int n_real,
                                uint64_t t0, uint64_t t1, double eta) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_real) return;
    const size_t g = r / 32, b = r % 32;
    auto at = [&](int k) -> size_t { return (g * M + k) * 32 + b; };
    bool ok = M >= 3;
    double inv_s[kMaxSlots], gap[kMaxSlots];
    double sum = 0.0;
    for (int k = 0; k + 1 < M; ++k) {
        const uint64_t first = t0 + (uint64_t)(((uint64_t)k - t0) & 1u);  // first t >= t0, t = k (mod 2)
        const uint64_t att = (first >= t1) ? 0 : (t1 - 1 - first) / 2 + 1;
        if (att == 0) ok = false;
        if (!ok) break;
        double a = (double)xacc[at(k)] / (double)att;
        a = a < 0.005 ? 0.005 : (a > 0.995 ? 0.995 : a);
        gap[k] = __dsub_rn(beta[at(k + 1)], beta[at(k)]);
        inv_s[k] = gap[k] / -log(a);
        sum = __dadd_rn(sum, inv_s[k]);
    }
    if (ok) {
        const double span = __dsub_rn(beta[at(M - 1)], beta[at(0)]);
        double bk = beta[at(0)];
        for (int k = 0; k + 2 < M; ++k) {
            const double target = __dmul_rn(span, inv_s[k]) / sum;
            bk = __dadd_rn(bk, __dadd_rn(__dmul_rn(__dsub_rn(1.0, eta), gap[k]), __dmul_rn(eta, target)));
            beta[at(k + 1)] = bk;
        }
    }
    for (int k = 0; k < M; ++k) xacc[at(k)] = 0u;
}

}  // namespace

void pt_release(ea_ctx *ctx) {
    if (!ctx || !ctx->pt) return;
    PtState *p = ctx->pt;
    void *ptrs[] = {p->d_spins, p->d_bonds, p->d_E, p->d_label, p->d_rt, p->d_bounds,
                    p->d_beta, p->d_planes, p->d_xacc, p->d_swaps, p->d_err};
    for (void *q : ptrs)
        if (q) cudaFree(q);
    delete p;
    ctx->pt = nullptr;
}

#define PT_CUDA(call)                                        \
    do {                                                     \
        cudaError_t e_ = (call);                             \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call);  \
    } while (0)

// host betas [n_real][M] -> device [g][k][32] (bits past n_real copy the group's first
// realization), then the threshold planes
static int pt_upload_betas(ea_ctx *ctx, const double *betas) {
    PtState *p = ctx->pt;
    const size_t G = p->n_groups, M = p->M;
    std::vector<double> h(G * M * 32);
    for (size_t g = 0; g < G; ++g)
        for (size_t k = 0; k < M; ++k)
            for (size_t b = 0; b < 32; ++b) {
                const size_t r = (32 * g + b < (size_t)p->n_real) ? 32 * g + b : 32 * g;
                h[(g * M + k) * 32 + b] = betas[r * M + k];
            }
    PT_CUDA(cudaMemcpyAsync(p->d_beta, h.data(), h.size() * 8, cudaMemcpyHostToDevice, ctx->stream));
    pt_planes_kernel<<<(int)(G * M), 32, 0, ctx->stream>>>(p->d_beta, p->dim, p->d_planes);
    PT_CUDA(cudaGetLastError());
    PT_CUDA(cudaStreamSynchronize(ctx->stream));
    return EA_OK;
}

extern "C" int pt_get_split(int dim, int L, int n_real, int M, int n_sm, int *ctas, int *slots, size_t *smem_bytes) {
    if ((dim != 2 && dim != 3) || L < 3 || L > 12 || n_real <= 0 || M < 2 || M > 64 || n_sm <= 0)
        return fail(EA_EINVAL, "no parallel tempering of dim=%d, L=%d, %d realizations, M=%d", dim, L, n_real, M);
    const int cs = pt_cluster(dim, L, M, (n_real + 31) / 32, n_sm), spc = (M + cs - 1) / cs;
    if (ctas) *ctas = cs;
    if (slots) *slots = spc;
    if (smem_bytes) *smem_bytes = pt_form(dim, L, spc).smem;
    return EA_OK;
}

extern "C" int pt_init(ea_ctx *ctx, int dim, int L, int n_real, uint32_t rid0, int M, const double *betas,
                       const int8_t *couplings_or_null) {
    if (!ctx) return fail(EA_EINVAL, "null context");
    if (dim != 2 && dim != 3) return fail(EA_EINVAL, "dim must be 2 or 3");
    if (L < 3 || L > 12) return fail(EA_EINVAL, "PT needs L in [3, 12]");
    if (n_real <= 0) return fail(EA_EINVAL, "n_real must be positive");
    if (rid0 % 32) return fail(EA_EINVAL, "rid0 must be a multiple of 32 (realizations are packed 32 per word)");
    if (M < 2 || M > 64) return fail(EA_EINVAL, "M must be in [2, 64]");
    if (!betas) return fail(EA_EINVAL, "null betas");
    for (int k = 0; k + 1 < M; ++k)
        if (!(betas[k + 1] > betas[k])) return fail(EA_EINVAL, "betas must increase with the slot index");
    PT_CUDA(cudaSetDevice(ctx->device));
    pt_release(ctx);
    PtState *p = new PtState();
    ctx->pt = p;
    p->dim = dim;
    p->L = L;
    p->V = volume_of(dim, L);
    p->nb = dim * p->V;
    p->M = M;
    p->n_real = n_real;
    p->n_groups = (n_real + 31) / 32;
    p->rid0 = rid0;
    p->cs = pt_cluster(dim, L, M, p->n_groups, ctx->n_sm);
    const size_t G = p->n_groups;
    auto alloc = [&](void **ptr, size_t bytes) -> int {
        if (cudaMalloc(ptr, bytes) != cudaSuccess) return fail(EA_ENOMEM, "PT allocation of %zu bytes failed", bytes);
        cudaMemsetAsync(*ptr, 0, bytes, ctx->stream);
        return EA_OK;
    };
    int rc;
    if ((rc = alloc((void **)&p->d_spins, G * M * p->V * 4)) || (rc = alloc((void **)&p->d_bonds, G * p->nb * 4)) ||
        (rc = alloc((void **)&p->d_E, G * M * 32 * 4)) || (rc = alloc((void **)&p->d_label, G * M * 32 * 4)) ||
        (rc = alloc((void **)&p->d_rt, G * M * 32 * sizeof(PtRt))) ||
        (rc = alloc((void **)&p->d_bounds, G * 32 * 2 * 4)) || (rc = alloc((void **)&p->d_beta, G * M * 32 * 8)) ||
        (rc = alloc((void **)&p->d_planes, G * M * 128 * 4)) || (rc = alloc((void **)&p->d_xacc, G * M * 32 * 4)) ||
        (rc = alloc((void **)&p->d_swaps, (M - 1) * 8)) || (rc = alloc((void **)&p->d_err, 4))) {
        pt_release(ctx);
        return rc;
    }
    // the same temperatures for every realization; bounds default: never reached
    std::vector<double> hbeta((size_t)n_real * M);
    for (int r = 0; r < n_real; ++r)
        for (int k = 0; k < M; ++k) hbeta[(size_t)r * M + k] = betas[k];
    if ((rc = pt_upload_betas(ctx, hbeta.data()))) return rc;
    void *scr;
    const int8_t *dJ = nullptr;
    if (couplings_or_null) {
        if ((rc = ctx_scratch(ctx, (size_t)n_real * p->nb + 256, &scr))) return rc;
        dJ = (const int8_t *)scr;
        PT_CUDA(cudaMemcpyAsync((void *)dJ, couplings_or_null, (size_t)n_real * p->nb, cudaMemcpyHostToDevice,
                                ctx->stream));
    }
    std::vector<int32_t> hb(G * 32 * 2);
    for (size_t q = 0; q < G * 32; ++q) {
        hb[2 * q] = -(1 << 30);   // e_g: never reached
        hb[2 * q + 1] = 1 << 30;  // e_hot: never reached
    }
    PT_CUDA(cudaMemcpyAsync(p->d_bounds, hb.data(), hb.size() * 4, cudaMemcpyHostToDevice, ctx->stream));
    PT_CUDA(pt_dispatch(p, dJ, ctx, 0, 0, 0));
    // round-trip records start at phase 0 with e_min = the initial energy
    std::vector<int32_t> hE(G * M * 32);
    PT_CUDA(cudaMemcpyAsync(hE.data(), p->d_E, hE.size() * 4, cudaMemcpyDeviceToHost, ctx->stream));
    PT_CUDA(cudaStreamSynchronize(ctx->stream));
    std::vector<PtRt> hr(G * M * 32);
    for (size_t gg = 0; gg < G; ++gg)
        for (int k = 0; k < M; ++k)
            for (int b = 0; b < 32; ++b) {
                PtRt &r = hr[(gg * M + k) * 32 + b];  // label k starts at slot k
                r.phase = 0;
                r.n_rt = 0;
                r.t_first = -1;
                r.t_last = -1;
                r.e_min = hE[(gg * M + k) * 32 + b];
                r.pad = 0;
            }
    PT_CUDA(cudaMemcpyAsync(p->d_rt, hr.data(), hr.size() * sizeof(PtRt), cudaMemcpyHostToDevice, ctx->stream));
    PT_CUDA(cudaStreamSynchronize(ctx->stream));
    p->t = 0;
    p->t_win = 0;
    return EA_OK;
}

extern "C" int pt_set_betas(ea_ctx *ctx, const double *betas) {
    if (!ctx || !ctx->pt) return fail(EA_ESTATE, "call pt_init first");
    if (!betas) return fail(EA_EINVAL, "null betas");
    const PtState *p = ctx->pt;
    for (int r = 0; r < p->n_real; ++r)
        for (int k = 0; k + 1 < p->M; ++k)
            if (!(betas[(size_t)r * p->M + k + 1] > betas[(size_t)r * p->M + k]))
                return fail(EA_EINVAL, "betas of realization %d must increase with the slot index", r);
    return pt_upload_betas(ctx, betas);
}

extern "C" int pt_get_betas(ea_ctx *ctx, double *betas) {
    if (!ctx || !ctx->pt) return fail(EA_ESTATE, "call pt_init first");
    if (!betas) return fail(EA_EINVAL, "null output");
    const PtState *p = ctx->pt;
    const size_t G = p->n_groups, M = p->M;
    std::vector<double> h(G * M * 32);
    PT_CUDA(cudaMemcpyAsync(h.data(), p->d_beta, h.size() * 8, cudaMemcpyDeviceToHost, ctx->stream));
    PT_CUDA(cudaStreamSynchronize(ctx->stream));
    for (int r = 0; r < p->n_real; ++r)
        for (size_t k = 0; k < M; ++k) betas[(size_t)r * M + k] = h[((r / 32) * M + k) * 32 + r % 32];
    return EA_OK;
}

extern "C" int pt_get_exchange_counts(ea_ctx *ctx, uint32_t *accepted, uint64_t *attempted) {
    if (!ctx || !ctx->pt) return fail(EA_ESTATE, "call pt_init first");
    const PtState *p = ctx->pt;
    const size_t G = p->n_groups, M = p->M;
    if (accepted) {
        std::vector<uint32_t> h(G * M * 32);
        PT_CUDA(cudaMemcpyAsync(h.data(), p->d_xacc, h.size() * 4, cudaMemcpyDeviceToHost, ctx->stream));
        PT_CUDA(cudaStreamSynchronize(ctx->stream));
        for (int r = 0; r < p->n_real; ++r)
            for (size_t k = 0; k + 1 < M; ++k) accepted[(size_t)r * (M - 1) + k] = h[((r / 32) * M + k) * 32 + r % 32];
    }
    if (attempted)
        for (size_t k = 0; k + 1 < M; ++k) {
            const uint64_t first = p->t_win + ((k - p->t_win) & 1u);
            attempted[k] = (first >= p->t) ? 0 : (p->t - 1 - first) / 2 + 1;
        }
    return EA_OK;
}

extern "C" int pt_adapt(ea_ctx *ctx, double eta) {
    if (!ctx || !ctx->pt) return fail(EA_ESTATE, "call pt_init first");
    if (!(eta >= 0.0 && eta <= 1.0)) return fail(EA_EINVAL, "eta must be in [0, 1]");
    PtState *p = ctx->pt;
    pt_adapt_kernel<<<(p->n_real + 127) / 128, 128, 0, ctx->stream>>>(p->d_beta, p->d_xacc, p->M, p->n_real,
                                                                       p->t_win, p->t, eta);
    PT_CUDA(cudaGetLastError());
    pt_planes_kernel<<<p->n_groups * p->M, 32, 0, ctx->stream>>>(p->d_beta, p->dim, p->d_planes);
    PT_CUDA(cudaGetLastError());
    PT_CUDA(cudaStreamSynchronize(ctx->stream));
    p->t_win = p->t;
    return EA_OK;
}

extern "C" int pt_set_rt_bounds(ea_ctx *ctx, const int32_t *e_g, const int32_t *e_hot) {
    if (!ctx || !ctx->pt) return fail(EA_ESTATE, "call pt_init first");
    if (!e_g || !e_hot) return fail(EA_EINVAL, "null bounds");
    PtState *p = ctx->pt;
    std::vector<int32_t> hb((size_t)p->n_groups * 64, 0);
    for (size_t q = 0; q < (size_t)p->n_groups * 32; ++q) {
        const bool in = q < (size_t)p->n_real;
        hb[2 * q] = in ? e_g[q] : -(1 << 30);
        hb[2 * q + 1] = in ? e_hot[q] : (1 << 30);
    }
    PT_CUDA(cudaMemcpyAsync(p->d_bounds, hb.data(), hb.size() * 4, cudaMemcpyHostToDevice, ctx->stream));
    PT_CUDA(cudaStreamSynchronize(ctx->stream));
    return EA_OK;
}

extern "C" int pt_run(ea_ctx *ctx, uint64_t n_sweeps, int count_roundtrips) {
    if (!ctx || !ctx->pt) return fail(EA_ESTATE, "call pt_init first");
    PtState *p = ctx->pt;
    if (p->t + n_sweeps > (1ull << 32)) return fail(EA_EINVAL, "sweep counter would exceed 2^32");
    if (n_sweeps == 0) return EA_OK;
    PT_CUDA(pt_dispatch(p, nullptr, ctx, 1, n_sweeps, count_roundtrips));
    p->t += n_sweeps;
    return EA_OK;
}

extern "C" int pt_get_state(ea_ctx *ctx, int8_t *spins, int32_t *E, int32_t *labels, uint64_t *t) {
    if (!ctx || !ctx->pt) return fail(EA_ESTATE, "call pt_init first");
    PtState *p = ctx->pt;
    const size_t G = p->n_groups, M = p->M, V = p->V;
    std::vector<uint32_t> hs;
    std::vector<int32_t> hE(G * M * 32), hL(G * M * 32);
    if (spins) {
        hs.resize(G * M * V);
        PT_CUDA(cudaMemcpyAsync(hs.data(), p->d_spins, hs.size() * 4, cudaMemcpyDeviceToHost, ctx->stream));
    }
    PT_CUDA(cudaMemcpyAsync(hE.data(), p->d_E, hE.size() * 4, cudaMemcpyDeviceToHost, ctx->stream));
    PT_CUDA(cudaMemcpyAsync(hL.data(), p->d_label, hL.size() * 4, cudaMemcpyDeviceToHost, ctx->stream));
    PT_CUDA(cudaStreamSynchronize(ctx->stream));
    for (int r = 0; r < p->n_real; ++r) {
        const size_t g = r / 32, b = r % 32;
        for (size_t k = 0; k < M; ++k) {
            if (E) E[r * M + k] = hE[(g * M + k) * 32 + b];
            if (labels) labels[r * M + k] = hL[(g * M + k) * 32 + b];
            if (spins)
                for (size_t i = 0; i < V; ++i)
                    spins[(r * M + k) * V + i] = ((hs[(g * M + k) * V + i] >> b) & 1u) ? -1 : 1;
        }
    }
    if (t) *t = p->t;
    return EA_OK;
}

extern "C" int pt_get_roundtrips(ea_ctx *ctx, ea_pt_stats *out, int reset) {
    if (!ctx || !ctx->pt) return fail(EA_ESTATE, "call pt_init first");
    if (!out) return fail(EA_EINVAL, "null output");
    PtState *p = ctx->pt;
    const size_t G = p->n_groups, M = p->M;
    std::vector<PtRt> hr(G * M * 32);
    PT_CUDA(cudaMemcpyAsync(hr.data(), p->d_rt, hr.size() * sizeof(PtRt), cudaMemcpyDeviceToHost, ctx->stream));
    PT_CUDA(cudaStreamSynchronize(ctx->stream));
    for (int r = 0; r < p->n_real; ++r) {
        const size_t g = r / 32, b = r % 32;
        for (size_t l = 0; l < M; ++l) {
            const PtRt &s = hr[(g * M + l) * 32 + b];
            ea_pt_stats &o = out[r * M + l];
            o.n_rt = s.n_rt;
            o.phase = s.phase;
            o.t_first = s.t_first;
            o.t_last = s.t_last;
            o.e_min = s.e_min;
            o.pad = 0;
        }
    }
    if (reset) {
        std::vector<int32_t> hE(G * M * 32), hL(G * M * 32);
        PT_CUDA(cudaMemcpyAsync(hE.data(), p->d_E, hE.size() * 4, cudaMemcpyDeviceToHost, ctx->stream));
        PT_CUDA(cudaMemcpyAsync(hL.data(), p->d_label, hL.size() * 4, cudaMemcpyDeviceToHost, ctx->stream));
        PT_CUDA(cudaStreamSynchronize(ctx->stream));
        for (size_t g = 0; g < G; ++g)
            for (size_t k = 0; k < M; ++k)
                for (int b = 0; b < 32; ++b) {
                    const int lbl = hL[(g * M + k) * 32 + b];
                    PtRt &s = hr[(g * M + lbl) * 32 + b];
                    s.phase = 0;
                    s.n_rt = 0;
                    s.t_first = -1;
                    s.t_last = -1;
                    s.e_min = hE[(g * M + k) * 32 + b];
                }
        PT_CUDA(cudaMemcpyAsync(p->d_rt, hr.data(), hr.size() * sizeof(PtRt), cudaMemcpyHostToDevice, ctx->stream));
        PT_CUDA(cudaStreamSynchronize(ctx->stream));
    }
    return EA_OK;
}

extern "C" int pt_get_swap_counts(ea_ctx *ctx, uint64_t *out) {
    if (!ctx || !ctx->pt) return fail(EA_ESTATE, "call pt_init first");
    if (!out) return fail(EA_EINVAL, "null output");
    PtState *p = ctx->pt;
    PT_CUDA(cudaMemcpyAsync(out, p->d_swaps, (p->M - 1) * 8, cudaMemcpyDeviceToHost, ctx->stream));
    PT_CUDA(cudaStreamSynchronize(ctx->stream));
    return EA_OK;
}
