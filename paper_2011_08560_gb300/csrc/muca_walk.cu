// muca_walk.cu -- a2 + a3 in the colour order (the checkerboard for even L), one warp per chain:
// the multicanonical sweep (Sec. II, Eq. "muca") with the sites of a sweep taken colour by colour,
// each colour in lexicographic order.  It serves every L (3..12), 2D and 3D, and tiles of any
// width; batches that the estimate in eamc_api.cu finds faster with a lane per chain run in
// muca_checker.cu: many chains, and contexts of several sizes, whose code the chains of an SM would
// evict from one another's instruction cache.
//
// What bounds it.  A chain is a serial chain of decisions: attempt i+1's threshold is thr[b][n] at
// the bin b that attempt i leaves.  A kernel that loads the threshold for that bin pays a
// shared-memory load per attempt (35 cycles with both outcomes loaded ahead; muca_checker.cu runs at
// 45.5).  Here the load leaves the chain: in a colour pass no two sites are neighbours, so every
// attempt's class n and random word r are known when the pass begins, and only the bin is not.  A
// lane evaluates ITS attempt for every bin of a window around the current one, accept(b) = r <
// thr[b][n], as a bit mask, and the walk through 32 attempts is then register arithmetic on a
// position p: p += d if the mask has bit p.
//
// The walk is parallel as well.  The batch's 32 attempts are four segments of eight; the eight
// lanes of a segment start it from the eight positions around the current one (p - 4 .. p + 3), so
// the four segments are walked at once, and a chain of three byte selects (segment 0 from p, each
// next one from the end of the one before) picks the lanes whose start was right.  Where a segment's
// start is not among its eight candidates, the attempts before it count (28 of 32 on average on cold
// chains) and the rest of the batch is walked again, with the same masks, from candidates around
// their end.  A batch ends early only where the walk comes to the window's end: the next one begins
// after the attempts that count, in a new window.  While a batch is walked, the masks of the next one are made for the same
// window; the window moves when the position comes near its end.  The bins outside the table are 0
// (never accepted), so a wall needs no test.
//
// L = 8, 1024 power-law chains in production: 112.6 -> 69 ms per 10^4 sweeps (46.6 -> 76 attempts
// per ns; 45.5 -> 28 cycles per attempt of a chain, 22 where a chain has a scheduler to itself);
// 500 chains of L = 7: 13.6 -> 34 attempts/ns, 300 of L = 10 in full tiles 6.5 -> 19.  One warp
// per chain costs 8 to 10 warp instructions per attempt, so that beyond two chains per scheduler
// the issue slots and the half-rate integer pipe are the bound (4096 chains: 109 attempts/ns, pipe
// 68 % and issue 72 % busy).
// Measured and left out: 32 bins instead of 24 (-5 %), 20 bins (within 1 %), the masks from fp16
// codes with an exact check afterwards (-6 %: HSET2 and HFMA2 run at half rate, the carry pair of
// wk_bit at full rate), one serial walk of the batch by every lane (46 cycles per attempt), two
// segments of 16 with 16 candidates for hot chains (-10 %), two to eight chains per warp (longer
// chains: 47 to 130 cycles per attempt), masks made after the walk instead of beside it (-10 %).
//
// Shared memory of a warp (5.8 KB at L = 8, 8 KB at the most, L = 11): the chain's lattice as row words (a nibble per site:
// spins; bonds Jx, Jy, Jz at bits 0, 1, 2), a pass's attempts {random word, entry} (a chunk of 32 or
// 64 rows where a pass has more than 256), 64 bins of the threshold table class by class (reloaded
// around the current bin when the window leaves them), the masks of two batches.
//
// Random words (the colour-order streams): the j-th colour-c site of row r takes word j&3 of
// Philox call (4 r + j/4, t, rid, (5 + c) | stream << 8).
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "eamc_internal.cuh"

namespace eamc {

namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr int kWalkBins = 64;  // bins of the cached part of the table
constexpr int kWin = 24;       // bins of the window
constexpr int kCentre = 10;    // a new window begins this many bins below the current one, or up to 3 more
constexpr int kEdge = 4;       // a batch that ends within this of the window's end moves it

template <int L>
using WkRow = typename std::conditional<(L <= 8), uint32_t, uint64_t>::type;

template <class T, int L>
__device__ __forceinline__ constexpr T wk_mask() {
    return (4 * L == 8 * (int)sizeof(T)) ? ~T(0) : ((T(1) << (4 * L)) - 1);
}
// nibble x <- nibble x+1 (mod L), and nibble x <- nibble x-1
template <class T, int L>
__device__ __forceinline__ T wk_next(T r) {
    return ((r >> 4) | (r << (4 * L - 4))) & wk_mask<T, L>();
}
template <class T, int L>
__device__ __forceinline__ T wk_prev(T r) {
    return ((r << 4) | (r >> (4 * L - 4))) & wk_mask<T, L>();
}

// odd L: the colour of a site is (ax(x) + ax(y) + ax(z)) mod 3 with ax(c) = c mod 3, except
// ax(L-1) = 1 when L - 1 is a multiple of 3 (the PT colouring); the colour-c sites of a row with
// (c - ax(y) - ax(z)) mod 3 = s are the x with ax(x) = s
__host__ __device__ constexpr int wk_ax(int L, int c) { return (c == L - 1 && (L - 1) % 3 == 0) ? 1 : c % 3; }
__host__ __device__ constexpr int wk_count(int L, int s) {
    int n = 0;
    for (int x = 0; x < L; ++x) n += wk_ax(L, x) == s;
    return n;
}
// the x with ax(x) = s, a nibble each
__host__ __device__ constexpr uint32_t wk_list(int L, int s) {
    uint32_t v = 0;
    int n = 0;
    for (int x = 0; x < L; ++x)
        if (wk_ax(L, x) == s) v |= (uint32_t)x << (4 * n++);
    return v;
}
__host__ __device__ constexpr int wk_max3(int a, int b, int c) { return a > b ? (a > c ? a : c) : (b > c ? b : c); }

template <int DIM, int L>
struct WalkGeo {
    using T = WkRow<L>;
    static constexpr bool ODD = (L & 1) != 0;
    static constexpr int NCOL = ODD ? 3 : 2;         // colour passes per sweep
    static constexpr int NR = DIM == 3 ? L * L : L;  // rows along x
    static constexpr int V = NR * L;
    static constexpr int B = ((DIM * V) / 2 >> 1) + 1;
    static constexpr int HALF = ODD ? wk_max3(wk_count(L, 0), wk_count(L, 1), wk_count(L, 2)) : L / 2;
    static constexpr int NGC = (HALF + 3) / 4;       // Philox calls per row and pass
    // rows per chunk: a pass of at most 256 attempts in one, else 32 or 64 rows, one or two per lane
    static constexpr int RCH = NR * HALF <= 256 ? NR : (HALF <= 4 ? 64 : 32);
    static constexpr int NCH = (NR + RCH - 1) / RCH;
    static constexpr int CAP = RCH * HALF;
    static constexpr int CLS = 2 * DIM + 2;              // classes 0 .. 2 DIM, and one that never accepts
    static constexpr int PAD = 2 * DIM + 1;              // that class
    static constexpr int STR = kWalkBins + 4;            // words between the classes of a cached table
    // byte offsets in a warp's shared memory
    static constexpr int WK = 0;                         // [2][32] {accept mask, bin change}
    static constexpr int ENDS = WK + 512;                // [2][32] bytes
    static constexpr int ATT = ENDS + 64;                // [CAP + 64] {random word, entry}
    static constexpr int RS = ATT + (CAP + 64) * 8;
    static constexpr int JB = RS + NR * (int)sizeof(T);
    static constexpr int EXACT = (JB + NR * (int)sizeof(T) + 15) / 16 * 16;  // [CLS][STR] thresholds
    static constexpr int STARTS = EXACT + CLS * STR * 4; // odd L: [NCOL][NR + 1] attempts before a row
    static constexpr size_t SMEM = STARTS + (ODD ? (NCOL * (NR + 1) * 2 + 15) / 16 * 16 : 0);
};

// m <- 2 m + (r < th), nr = ~r: the carry of th + ~r
__device__ __forceinline__ void wk_bit(uint32_t &m, uint32_t th, uint32_t nr) {
    asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %1, %2;\n\taddc.u32 %0, %0, %0;\n\t}" : "+r"(m) : "r"(th), "r"(nr));
}

// accept masks of eight bins and of the window's: bit k = (r < th[k]), nr = ~r
__device__ __forceinline__ uint32_t wk_eight(const uint4 *q, uint32_t nr) {
    const uint4 lo = q[0], hi = q[1];
    uint32_t v = 0u;
    wk_bit(v, hi.w, nr);
    wk_bit(v, hi.z, nr);
    wk_bit(v, hi.y, nr);
    wk_bit(v, hi.x, nr);
    wk_bit(v, lo.w, nr);
    wk_bit(v, lo.z, nr);
    wk_bit(v, lo.y, nr);
    wk_bit(v, lo.x, nr);
    return v;
}
__device__ __forceinline__ uint32_t wk_accepts(const uint32_t *th, uint32_t nr) {
    static_assert(kWin == 24, "three groups of eight bins");
    const uint4 *q = reinterpret_cast<const uint4 *>(th);
    return wk_eight(q, nr) + (wk_eight(q + 2, nr) << 8) + (wk_eight(q + 4, nr) << 16);
}

// one attempt at window position pos: accepted if the mask has the bit (a position outside the
// window, also a negative one, shifts everything out and stays)
__device__ __forceinline__ void wk_try(int &pos, uint32_t &acc, uint32_t m, uint32_t d, uint32_t bit) {
    asm("{\n\t.reg .u32 t;\n\tshr.u32 t, %2, %0;\n\tand.b32 t, t, 1;\n\tmad.lo.u32 %0, t, %3, %0;\n\tmad.lo.u32 %1, t, %4, %1;\n\t}"
        : "+r"(pos), "+r"(acc) : "r"(m), "r"(d), "r"(bit));
}

// byte sel (its low three bits; bit 3 is 0) of the eight bytes lo, hi; the result's upper bytes are
// of no meaning
__device__ __forceinline__ uint32_t wk_pick(uint32_t lo, uint32_t hi, uint32_t sel) {
    uint32_t v;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(v) : "r"(lo), "r"(hi), "r"(sel));
    return v;
}

template <int DIM, int L>
__device__ __forceinline__ void walk_chain(const TileDesc &td, int tile, int ch, SlotState *__restrict__ slots,
                                           uint32_t *__restrict__ spins, const uint32_t *__restrict__ bonds,
                                           const uint32_t *__restrict__ thr, uint32_t *__restrict__ hist,
                                           uint64_t n_sweeps, PhiloxKey key, int count_rt,
                                           unsigned *__restrict__ diag, unsigned char *smem) {
    using G = WalkGeo<DIM, L>;
    using T = typename G::T;
    constexpr bool ODD = G::ODD;
    constexpr int NR = G::NR, NCOL = G::NCOL, HALF = G::HALF, NGC = G::NGC, STR = G::STR;
    const int lane = threadIdx.x & 31, seg = lane >> 3;
    uint2 *wk = reinterpret_cast<uint2 *>(smem + G::WK);
    unsigned char *ends = smem + G::ENDS;
    uint2 *att = reinterpret_cast<uint2 *>(smem + G::ATT);
    T *Rs = reinterpret_cast<T *>(smem + G::RS);
    T *JBs = reinterpret_cast<T *>(smem + G::JB);
    uint32_t *exact = reinterpret_cast<uint32_t *>(smem + G::EXACT);
    uint16_t *starts = reinterpret_cast<uint16_t *>(smem + G::STARTS);

    const int slot = tile * kTile + ch;
    SlotState ss = slots[slot];
    if (!ss.active) {
        if (lane == 0) slots[slot].t = ss.t + n_sweeps;
        return;
    }
    const uint64_t lrow = td.w_base + (uint64_t)ch * G::B;
    uint32_t *gsp = spins + td.spin_off;
    const uint32_t *gbd = bonds + td.bond_off;
    for (int row = lane; row < NR; row += 32) {
        T r = 0, jb = 0;
#pragma unroll
        for (int x = 0; x < L; ++x) {
            const int i = row * L + x;
            r |= T((gsp[i] >> ch) & 1u) << (4 * x);
            uint32_t j = (gbd[i * DIM] >> ch) & 1u;
            j |= ((gbd[i * DIM + 1] >> ch) & 1u) << 1;
            if constexpr (DIM == 3) j |= ((gbd[i * DIM + 2] >> ch) & 1u) << 2;
            jb |= T(j) << (4 * x);
        }
        Rs[row] = r;
        JBs[row] = jb;
    }
    auto row_shift = [](int c, int r) -> int {
        const int y = r % L, z = DIM == 3 ? r / L : 0;
        if constexpr (ODD) return ((c - wk_ax(L, y) - (DIM == 3 ? wk_ax(L, z) : 0)) + 6) % 3;
        else return (c + y + z) & 1;
    };
    if constexpr (ODD) {
        for (int c = 0; c < NCOL; ++c) {
            int at = 0;
            for (int r0 = 0; r0 < NR; r0 += 32) {
                const int r = r0 + lane;
                const int sh = row_shift(c, r < NR ? r : 0);
                const int n = r < NR ? (sh == 0 ? wk_count(L, 0) : sh == 1 ? wk_count(L, 1) : wk_count(L, 2)) : 0;
                int incl = n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl += v;
                }
                if (r < NR) starts[c * (NR + 1) + r] = (uint16_t)(at + incl - n);
                at += __shfl_sync(kFull, incl, 31);
            }
            if (lane == 0) starts[c * (NR + 1) + NR] = (uint16_t)at;
        }
    }

    // bins [cb, cb + kWalkBins) of the chain's table, class by class;
    // bins outside the table never accept
    const uint4 *table = reinterpret_cast<const uint4 *>(thr + lrow * 8);
    auto load_cache = [&](int cb) {
        for (int k = lane; k < kWalkBins; k += 32) {
            const int b = cb + k;
            uint4 lo = make_uint4(0, 0, 0, 0), hi = lo;
            if (b >= 0 && b < G::B) { lo = table[2 * b]; hi = table[2 * b + 1]; }
            exact[k] = lo.x;
            exact[STR + k] = lo.y;
            exact[2 * STR + k] = lo.z;
            exact[3 * STR + k] = lo.w;
            exact[4 * STR + k] = hi.x;
            if constexpr (DIM == 3) {
                exact[5 * STR + k] = hi.y;
                exact[6 * STR + k] = hi.z;
            }
        }
        __syncwarp();
    };
    int b = ss.b;
    int cb = (b - kWalkBins / 2) & ~3;
    for (int k = lane; k < STR; k += 32) exact[G::PAD * STR + k] = 0u;
    load_cache(cb);

    int phase = ss.phase, nrt = ss.n_rt, bmin = ss.b_min, bmax = 0;
    int64_t tf = ss.t_first, tl = ss.t_last;
    const uint64_t t0 = ss.t;
    const uint32_t stream8 = ss.stream << 8;

    for (uint64_t sw = 0; sw < n_sweeps; ++sw) {
        const uint32_t t = (uint32_t)(t0 + sw);
        for (int c = 0; c < NCOL; ++c) {
            for (int r0 = 0; r0 < NR; r0 += G::RCH) {
                const int r1 = (G::NCH == 1) ? NR : min(r0 + G::RCH, NR);
                int a00 = 0, N = (r1 - r0) * HALF;
                if constexpr (ODD) {
                    a00 = starts[c * (NR + 1) + r0];
                    N = starts[c * (NR + 1) + r1] - a00;
                }
                // ---- the chunk's classes and random words, a row per lane
#pragma unroll 2
                for (int r = r0 + lane; r < r1; r += 32) {
                    const int y = r % L, z = DIM == 3 ? r / L : 0;
                    constexpr T M1 = wk_mask<T, L>() & (T)0x1111111111111111ull;
                    const T R = Rs[r], JB = JBs[r];
                    const T uxp = R ^ wk_next<T, L>(R) ^ (JB & M1);
                    const int ryp = (y == L - 1) ? r - (L - 1) : r + 1;
                    const int rym = (y == 0) ? r + (L - 1) : r - 1;
                    T sum = uxp + wk_prev<T, L>(uxp) + (R ^ Rs[ryp] ^ ((JB >> 1) & M1)) +
                            (R ^ Rs[rym] ^ ((JBs[rym] >> 1) & M1));
                    if constexpr (DIM == 3) {
                        const int rzp = (z == L - 1) ? r - (L - 1) * L : r + L;
                        const int rzm = (z == 0) ? r + (L - 1) * L : r - L;
                        sum += (R ^ Rs[rzp] ^ ((JB >> 2) & M1)) + (R ^ Rs[rzm] ^ ((JBs[rzm] >> 2) & M1));
                    }
                    const int sh = row_shift(c, r);
                    int a0, cnt = HALF;
                    uint32_t xs = 0u;
                    if constexpr (ODD) {
                        a0 = starts[c * (NR + 1) + r] - a00;
                        cnt = sh == 0 ? wk_count(L, 0) : sh == 1 ? wk_count(L, 1) : wk_count(L, 2);
                        xs = sh == 0 ? wk_list(L, 0) : sh == 1 ? wk_list(L, 1) : wk_list(L, 2);
                    } else {
                        a0 = (r - r0) * HALF;
                        sum >>= 4 * sh;
                    }
#pragma unroll
                    for (int q = 0; q < NGC; ++q) {
                        const uint4 w = philox4x32_10(make_uint4((uint32_t)(4 * r + q), t, ss.rid,
                                                                 (uint32_t)(5 + c) | stream8), key);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int j = 4 * q + k;
                            if (j < HALF) {
                                uint32_t n, x;
                                if constexpr (ODD) {
                                    x = (xs >> (4 * j)) & 0xFu;
                                    n = (uint32_t)(sum >> (4 * x)) & 0x7u;
                                } else {
                                    x = (uint32_t)(sh + 2 * j);
                                    n = (uint32_t)(sum >> (8 * j)) & 0x7u;
                                }
                                if (!ODD || j < cnt) {
                                    // class, bit of the site in its word of the lattice, that word's offset
                                    const uint32_t word = sizeof(T) == 4 ? (uint32_t)r : 2u * (uint32_t)r + (x >> 3);
                                    const uint32_t nib = sizeof(T) == 4 ? x : (x & 7u);
                                    att[a0 + j] = make_uint2(~min(uint4_get(w, k), kAlways - 1u), n + nib * 32u + word * 1024u);
                                }
                            }
                        }
                    }
                }
                att[N + lane] = make_uint2(0u, (uint32_t)G::PAD);
                att[N + 32 + lane] = make_uint2(0u, (uint32_t)G::PAD);
                __syncwarp();
                // ---- the attempts, in batches of 32
                int s = 0, k = 0, w0 = 0, p = 0;
                uint32_t e = 0u;
                int rlo = 1000000, rhi = -1000000, tlo = 0, thi = 0;
                auto bounds = [&]() {
                    tlo = (count_rt && phase == 1) ? ss.b_g - w0 : -1000000;
                    thi = (count_rt && phase != 1) ? ss.b_top - w0 : 1000000;
                };
                // the masks of the attempts from s, in a window around the current bin
                auto rebuild = [&]() {
                    bmin = min(bmin, w0 + rlo);
                    bmax = max(bmax, w0 + rhi);
                    rlo = 1000000;
                    rhi = -1000000;
                    w0 = (b - kCentre) & ~3;
                    p = b - w0;
                    if (w0 < cb || w0 + kWin > cb + kWalkBins) {
                        cb = (b - kWalkBins / 2) & ~3;
                        load_cache(cb);
                    }
                    const uint2 at = att[s + lane];
                    e = at.y;
                    const int n = (int)(e & 7u);
                    const uint32_t m = wk_accepts(exact + n * STR + (w0 - cb), at.x);
                    wk[k * 32 + lane] = make_uint2(m, (uint32_t)(DIM - n));
                    bounds();
                    __syncwarp();
                };
                // the batch before: flips and measurement taken up while the next is walked.  Lanes of
                // a segment that does not count have H = 0 and an empty range
                uint32_t pe = 0u, pH = 0u;
                int plo = 1000000, phi = -1000000, pw0 = 0, pst = 0;
                auto post = [&]() {
                    const bool flip = ((pH >> (lane & 7)) & 1u) != 0u;
                    rlo = min(rlo, plo);
                    rhi = max(rhi, phi);
                    if (flip) atomicXor(reinterpret_cast<uint32_t *>(reinterpret_cast<unsigned char *>(Rs) + (pe >> 8)), 1u << ((pe >> 3) & 31u));
                    if (__any_sync(kFull, plo <= tlo || phi >= thi)) {
                        int at = flip ? DIM - (int)(pe & 7u) : 0;
#pragma unroll
                        for (int o = 1; o < 8; o <<= 1) {
                            const int u = __shfl_up_sync(kFull, at, o, 8);
                            if ((lane & 7) >= o) at += u;
                        }
                        at += pw0 + pst;  // bin after this lane's attempt
                        const bool in = plo <= phi && (pe & 7u) != (uint32_t)G::PAD;
                        const uint32_t mt = __ballot_sync(kFull, in && at >= ss.b_top);
                        const uint32_t mb = __ballot_sync(kFull, in && at <= ss.b_g);
                        int i0 = 0;
                        while (i0 < 32) {
                            const uint32_t mk = ((phase == 1) ? mb : mt) >> i0;
                            if (mk == 0u) break;
                            i0 += __ffs(mk);
                            if (phase == 0) { tf = (int64_t)(t0 + sw); phase = 1; }
                            else if (phase == 1) { phase = 2; }
                            else { nrt += 1; tl = (int64_t)(t0 + sw); phase = 1; }
                        }
                        bounds();
                    }
                    pH = 0u;
                    plo = 1000000;
                    phi = -1000000;
                };
                rebuild();
                while (s < N) {
                    int base = p - 4;
                    int pos = base + ((lane - base) & 7), lo = 64, hi = -64;
                    uint32_t H = 0u, en = 0u;
                    auto walk = [&]() {
                        const uint4 *wv = reinterpret_cast<const uint4 *>(wk + k * 32 + seg * 8);
#pragma unroll
                        for (int j = 0; j < 8; j += 2) {
                            const uint4 v = wv[j / 2];
                            wk_try(pos, H, v.x, v.y, 1u << j);
                            const int pa = pos;
                            wk_try(pos, H, v.z, v.w, 2u << j);
                            lo = __vimin3_s32(lo, pa, pos);
                            hi = __vimax3_s32(hi, pa, pos);
                        }
                    };
                    // a segment's end as a byte: its three low bits, its two high bits from bit 4, bit 6 not
                    // a candidate of the next segment, bit 7 outside the window
                    auto leave = [&]() {
                        ends[32 * k + lane] = (unsigned char)(pos + (pos & 0x18) + ((uint32_t)(pos - base) > 7u ? 0x40 : 0) |
                                                              ((uint32_t)pos >= (uint32_t)kWin ? 0xC0 : 0));
                    };
                    if (G::NR * HALF > 160 || s + 32 < N) {  // (small passes: not after the last batch)
                        const uint2 next = att[s + 32 + lane];
                        en = next.y;
                        walk();
                        const int n2 = (int)(en & 7u);
                        const uint32_t m2 = wk_accepts(exact + n2 * STR + (w0 - cb), next.x);
                        wk[(k ^ 1) * 32 + lane] = make_uint2(m2, (uint32_t)(DIM - n2));
                    } else {
                        walk();
                    }
                    leave();
                    __syncwarp();
                    const uint4 ma = reinterpret_cast<const uint4 *>(ends + 32 * k)[0], mb = reinterpret_cast<const uint4 *>(ends + 32 * k)[1];
                    const uint32_t v0 = wk_pick(ma.x, ma.y, (uint32_t)(p & 7)), v1 = wk_pick(ma.z, ma.w, v0);
                    const uint32_t v2 = wk_pick(mb.x, mb.y, v1), v3 = wk_pick(mb.z, mb.w, v2);
                    const uint32_t cs = (seg & 2) ? ((seg & 1) ? v2 : v1) : ((seg & 1) ? v0 : (uint32_t)p);
                    const int src = (lane & 24) | (int)(cs & 7u);
                    const uint32_t Hs = __shfl_sync(kFull, H, src);
                    const int los = __shfl_sync(kFull, lo, src), his = __shfl_sync(kFull, hi, src);
                    post();
                    pe = e;
                    pH = Hs;
                    plo = los;
                    phi = his;
                    pw0 = w0;
                    pst = base + (int)((cs - (uint32_t)base) & 7u);
                    uint32_t ve = v3;
                    int kc = 32;
                    if ((((v0 | v1 | v2) & 0xC0u) | (v3 & 0x80u)) != 0u) {
                        // a segment began outside the candidates or left the window: the ones before it count
                        ve = v0;
                        kc = (v0 & 0x80u) ? 0 : 8;
                        if ((v0 & 0xC0u) == 0u && !(v1 & 0x80u)) {
                            ve = v1;
                            kc = 16;
                            if ((v1 & 0xC0u) == 0u && !(v2 & 0x80u)) {
                                ve = v2;
                                kc = 24;
                            }
                        }
                        if (lane >= kc) {
                            pH = 0u;
                            plo = 1000000;
                            phi = -1000000;
                        }
                        // the rest of the batch again, from candidates around the end of the last one that
                        // counts: its masks stand as long as the window does, and so do the next batch's
                        while (kc > 0 && kc < 32) {
                            const int from = (int)((ve & 7u) | ((ve >> 1) & 0x18u)), first = kc >> 3;
                            if ((uint32_t)(from - kEdge) > (uint32_t)(kWin - 1 - 2 * kEdge)) break;
                            post();
                            base = from - 4;
                            pos = base + ((lane - base) & 7);
                            lo = 64;
                            hi = -64;
                            H = 0u;
                            walk();
                            leave();
                            __syncwarp();
                            const uint4 ra = reinterpret_cast<const uint4 *>(ends + 32 * k)[0], rb = reinterpret_cast<const uint4 *>(ends + 32 * k)[1];
                            const uint32_t f = (uint32_t)(from & 7);
                            const uint32_t u1 = wk_pick(ra.z, ra.w, f);  // segment 1 is the first that can be left
                            const uint32_t u2 = wk_pick(rb.x, rb.y, first > 1 ? f : u1);
                            const uint32_t u3 = wk_pick(rb.z, rb.w, first > 2 ? f : u2);
                            int now = kc;
                            bool on = true;
                            if (first <= 1) {
                                if (!(u1 & 0x80u)) { now = 16; ve = u1; }
                                on = (u1 & 0xC0u) == 0u;
                            }
                            if (first <= 2 && on) {
                                if (!(u2 & 0x80u)) { now = 24; ve = u2; }
                                on = (u2 & 0xC0u) == 0u;
                            }
                            if (on && !(u3 & 0x80u)) { now = 32; ve = u3; }
                            const uint32_t cr = seg == first ? f : (seg == 2 ? u1 : u2);
                            const int src = (lane & 24) | (int)(cr & 7u);
                            const uint32_t Hr = __shfl_sync(kFull, H, src);
                            const int lor = __shfl_sync(kFull, lo, src), hir = __shfl_sync(kFull, hi, src);
                            if (seg >= first && lane < now) {
                                pH = Hr;
                                plo = lor;
                                phi = hir;
                            }
                            pst = base + (int)((cr - (uint32_t)base) & 7u);
                            if (now == kc) break;  // the next segment leaves the window
                            kc = now;
                        }
                    }
                    e = en;
                    int pend = (int)((ve & 7u) | ((ve >> 1) & 0x18u));
                    if (kc == 0) {  // attempt by attempt while the next one cannot leave the window
                        pend = p;
                        uint32_t h = 0u;
                        int l = 1000000, u = -1000000;
                        while (kc < 8 && pend >= DIM && pend < kWin - DIM) {
                            const uint2 v = wk[k * 32 + kc];
                            wk_try(pend, h, v.x, v.y, 1u << kc);
                            l = min(l, pend);
                            u = max(u, pend);
                            ++kc;
                        }
                        if (lane < kc) {
                            pH = h;
                            plo = l;
                            phi = u;
                        }
                        __syncwarp();
                    }
                    s += kc;
                    p = pend;
                    k ^= 1;
                    if ((kc < 32 || (uint32_t)(pend - kEdge) > (uint32_t)(kWin - 1 - 2 * kEdge)) && s < N) {
                        b = w0 + p;
                        post();
                        rebuild();
                    }
                }
                post();
                b = w0 + p;
                bmin = min(bmin, w0 + rlo);
                bmax = max(bmax, w0 + rhi);
                __syncwarp();
            }
        }
        if (lane == 0) atomicAdd(&hist[lrow + b], 1u);
    }
    bmin = __reduce_min_sync(kFull, bmin);
    bmax = __reduce_max_sync(kFull, bmax);
    // ---- state back: this chain's bit of every spin word that changed
    for (int i = lane; i < G::V; i += 32) {
        const uint32_t now = (uint32_t)(Rs[i / L] >> (4 * (i % L))) & 1u;
        if (((gsp[i] >> ch) & 1u) != now) atomicXor(&gsp[i], 1u << ch);
    }
    if (lane == 0) {
        ss.b = b;
        ss.b_min = bmin;
        ss.phase = phase;
        ss.n_rt = nrt;
        ss.t_first = tf;
        ss.t_last = tl;
        ss.t = t0 + n_sweeps;
        if (count_rt && energy_of_bin(DIM * G::V, ss.parity, ss.b_min) < ss.e_g) ss.requeue = 1;
        slots[slot] = ss;
        if (diag && (bmin < 0 || bmax > ss.b_top)) atomicOr(diag, 1u);
    }
}

// Block (tile, channel): one warp, one chain; tiles in the order of tile_list (longest chains
// first).  128 registers let 16 warps share an SM: 102.8 against 92.9 attempts/ns with 141 registers
// at 4096 chains of L = 8, the same at 1024 (and 5 % less at 1024 when held to 96).  Single-warp blocks
// are dealt evenly to the SMs and their schedulers.
template <int DIM>
__global__ void __launch_bounds__(32, 16)
muca_walk_kernel(const TileDesc *__restrict__ tiles, const int32_t *__restrict__ tile_list, SlotState *__restrict__ slots,
                 uint32_t *__restrict__ spins, const uint32_t *__restrict__ bonds, const uint32_t *__restrict__ thr,
                 uint32_t *__restrict__ hist, uint64_t n_sweeps, PhiloxKey key, int count_rt,
                 unsigned *__restrict__ diag, int n_sub) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tile = tile_list[blockIdx.x / n_sub], ch = blockIdx.x % n_sub;
    const TileDesc td = tiles[tile];
    if (ch >= td.width) return;
    const uint64_t n_tile = n_sweeps * (uint64_t)(td.sweep_mul > 0 ? td.sweep_mul : 1);
#define EAMC_WK(LL) case LL: walk_chain<DIM, LL>(td, tile, ch, slots, spins, bonds, thr, hist, n_tile, key, count_rt, diag, smem_raw); break;
    switch (td.L) {
        EAMC_WK(3) EAMC_WK(4) EAMC_WK(5) EAMC_WK(6) EAMC_WK(7) EAMC_WK(8) EAMC_WK(9) EAMC_WK(10) EAMC_WK(11) EAMC_WK(12)
        default: break;
    }
#undef EAMC_WK
}

template <int DIM>
size_t walk_smem(int L) {
#define EAMC_WS(LL) case LL: return WalkGeo<DIM, LL>::SMEM;
    switch (L) {
        EAMC_WS(3) EAMC_WS(4) EAMC_WS(5) EAMC_WS(6) EAMC_WS(7) EAMC_WS(8) EAMC_WS(9) EAMC_WS(10) EAMC_WS(11) EAMC_WS(12)
        default: return 0;
    }
#undef EAMC_WS
}

}  // namespace

// the tile widths of the colour order: 32 chains, and in 3D 16 (L = 4..8), 8 (L = 4..10), 4 (L = 11, 12)
bool colour_width_supported(int dim, int L, int width) {
    if (L < 3 || L > 12 || (dim != 2 && dim != 3)) return false;
    if (width == 32) return true;
    if (dim != 3) return false;
    return (width == 16 && L >= 4 && L <= 8) || (width == 8 && L >= 4 && L <= 10) || (width == 4 && L >= 11);
}

size_t walk_smem_bytes(int dim, int L) { return dim == 3 ? walk_smem<3>(L) : walk_smem<2>(L); }

cudaError_t launch_sweeps_walk(const TileDesc *d_tiles, const int32_t *d_list, int n_tiles, int dim, int max_width,
                               size_t smem, SlotState *d_slots, uint32_t *d_spins, const uint32_t *d_bonds,
                               const uint32_t *d_thr, uint32_t *d_hist, uint64_t n_sweeps, PhiloxKey key,
                               int count_rt, unsigned *d_diag, cudaStream_t st) {
    if (n_tiles <= 0 || n_sweeps == 0) return cudaSuccess;
    const int grid = n_tiles * max_width;
    if (dim == 3)
        muca_walk_kernel<3><<<grid, 32, smem, st>>>(d_tiles, d_list, d_slots, d_spins, d_bonds, d_thr, d_hist, n_sweeps,
                                                    key, count_rt, d_diag, max_width);
    else
        muca_walk_kernel<2><<<grid, 32, smem, st>>>(d_tiles, d_list, d_slots, d_spins, d_bonds, d_thr, d_hist, n_sweeps,
                                                    key, count_rt, d_diag, max_width);
    return cudaGetLastError();
}

}  // namespace eamc
