// fragment.cu -- the paper's linear-time meta-heuristic (Sec. II; App. A, Fig. 5) with
// simulated-annealing fragment optimisations, wave by wave on the GPU.
//
// Wave w = a + l*(b + l*c) fixes every spin whose coordinates are congruent to (a, b, c)
// mod l.  The fragment of such a spin is the cube of side l centred on it; with L a
// multiple of l the fragments of one wave are disjoint, so one launch anneals all of
// them.  A warp owns one fragment: its 32 reads are the 32 bits of one word per cube
// site, kept in shared memory for the whole anneal, beside a word of the site's couplings
// and a list of the free sites of each colour.  Sites fixed by earlier waves hold all-equal
// words and are never updated.  The read of lowest cube energy fixes the centre spin in
// global memory.
//
// A half sweep takes the colour's free sites 32 at a time, in two steps.  First a lane has
// a site: for all reads at once it counts P, the weight of the positive bond terms
// J s_i s_k, and keeps d = ceil(M / 2) - P as bit planes, M the weight of all the site's
// bonds.  x = s_i h_i = 2P - M is negative exactly where d > 0 (the others accept), and the
// threshold is then that of k = 2d, or 2d - 1 when M is odd.  Then a lane has a site and
// four of its reads, the reads one Philox block draws for: 32-bit draws leave no other way
// than a block for each four reads, and they are most of the work.  The second step runs
// with all lanes busy however few sites are free, where a lane that stayed with its site
// through its eight blocks left two thirds of them idle on average (the free sites shrink
// from l^3 to one over the waves) and followed branches for each read.
#include <stdint.h>
#include <stdio.h>

#include <algorithm>
#include <vector>

#include "metropolis.cuh"
#include "philox.cuh"
#include "sg_internal.h"

namespace sg {
namespace {

constexpr int kWarps = 4;  // fragments per block
constexpr int kLMax = 7;   // largest fragment side
constexpr int kVMax = kLMax * kLMax * kLMax;

struct FragArgs {
    int8_t* spins;                 // [I][N] logical order; 0 = not fixed yet
    const uint2* const* j6_ptrs;   // per instance: [N] six-coupling records (+x, -x, +y, -y, +z, -z)
    const RunKeys* keys;           // [I]
    const uint32_t* thr;           // [S][kThrRow]
    int L, l, S;
    uint32_t lmagic;               // ceil(2^32 / l) (0 for l = 1)
};

__device__ __forceinline__ int coupling(uint2 r, int q)
{
    return (int)(int8_t)(((q < 4 ? r.x : r.y) >> (8 * (q & 3))) & 0xFFu);
}

// The draws of one fragment: Philox counters (centre, sweep, item, domain), whose first two
// rounds share two of their four multiplies (one of each round's pair sees the centre alone).
struct FragDraws {
    RunKeys key;
    uint32_t sx, sy, sl;
    __device__ __forceinline__ FragDraws(uint32_t centre, const RunKeys& k) : key(k)
    {
        uint32_t hi, lo, h2;
        philox_mulhilo(kPhiloxMulA, centre, &hi, &lo);
        philox_mulhilo(kPhiloxMulB, hi ^ kDomainFragment ^ key.k1, &h2, &sl);
        sx = h2 ^ (key.k0 + kPhiloxWeylA);
        sy = lo ^ (key.k1 + kPhiloxWeylB);
    }
    __device__ __forceinline__ void draw(uint32_t sweep, uint32_t item, uint32_t (&c)[4]) const
    {
        uint32_t hi, lo, h2, l2;
        philox_mulhilo(kPhiloxMulB, item, &hi, &lo);
        philox_mulhilo(kPhiloxMulA, hi ^ sweep ^ key.k0, &h2, &l2);
        c[0] = lo ^ sx, c[1] = sl, c[2] = h2 ^ sy, c[3] = l2;
#pragma unroll
        for (int r = 2; r < 10; ++r) {
            philox_mulhilo(kPhiloxMulA, c[0], &hi, &lo);
            philox_mulhilo(kPhiloxMulB, c[2], &h2, &l2);
            c[0] = mp::logic<mp::kXor3>(h2, c[1], key.k0 + (uint32_t)r * kPhiloxWeylA);
            c[1] = l2;
            c[2] = mp::logic<mp::kXor3>(hi, c[3], key.k1 + (uint32_t)r * kPhiloxWeylB);
            c[3] = lo;
        }
    }
};

// Reads: bit 8m + g of a word is read 4g + m, so that the reads of one Philox block (a g) are
// the same bit of the word's four bytes, and a ballot over (site, g) lanes is a byte a site.
//
// Records: site q of the cube (9 bits), M (4), then six bits each (order +x, -x, +y, -y, +z,
// -z): bonds inside the cube that are positive, of weight 1, of weight 2.
constexpr int kOrAnd = 0xF8;  // (mp::logic) a | (b & c)
constexpr int kRecM = 9, kRecPos = 13, kRecOne = 19, kRecTwo = 25;

__device__ __forceinline__ uint32_t rotate_right(uint32_t x, int n) { return __funnelshift_r(x, x, n); }

// UNITJ: all |J| = 1 (no record has bonds of weight 2).
template <bool UNITJ>
__global__ void __launch_bounds__(kWarps * 32, 8) fragment_wave_kernel(const FragArgs a, int wave)
{
    constexpr unsigned kAll = 0xFFFFFFFFu;
    constexpr int kPad = kLMax * kLMax;  // a bond that leaves the cube still loads a word
    __shared__ uint32_t s_words[kWarps][kVMax + 2 * kPad];
    __shared__ uint32_t s_rec[kWarps][kVMax];
    __shared__ uint16_t s_free[kWarps][2][(kVMax + 1) / 2];  // free sites of each colour
    __shared__ __align__(16) uint4 s_item[kWarps][32];       // of a lane's site: the planes of d, then 8q | odd M << 31
    __shared__ __align__(64) uint32_t s_thr[kWarps][16];     // the sweep's thresholds, [M odd][d]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int inst = blockIdx.y;
    const int L = a.L, l = a.l, h = (l - 1) / 2, ll = l * l, V = ll * l;
    const int per = L / l;
    const int frag = blockIdx.x * kWarps + warp;
    if (frag >= per * per * per) return;  // the whole warp
    const int ca = wave % l, cb = (wave / l) % l, cc = wave / ll;
    const int cx = ca + l * (frag % per), cy = cb + l * ((frag / per) % per), cz = cc + l * (frag / (per * per));
    const int centre = cx + L * (cy + L * cz);
    const FragDraws draws((uint32_t)centre, a.keys[inst]);
    const uint2* __restrict__ j6 = a.j6_ptrs[inst];
    int8_t* __restrict__ sp = a.spins + (size_t)inst * L * L * L;
    uint32_t* const words = s_words[warp] + kPad;
    uint32_t* const recs = s_rec[warp];
    uint4* const items = s_item[warp];
    uint32_t* const thr = s_thr[warp];

    // cube sites: records, the words of fixed sites, and the lists of the free sites of each
    // colour (compacted by ballot, warp-uniform counts)
    int nfree[2] = {0, 0};
    uint32_t fixed = 0;  // of the lane's sites lane, 32 + lane, ...
    for (int base = 0; base < V; base += 32) {
        const int q = base + lane;
        bool free_site = false;
        int colour = 0;
        if (q < V) {
            const int row = l == 1 ? q : (int)__umulhi((uint32_t)q, a.lmagic), dx = q - row * l;
            const int dz = l == 1 ? row : (int)__umulhi((uint32_t)row, a.lmagic), dy = row - dz * l;
            auto wrap = [](int v, int n) { return v < 0 ? v + n : v >= n ? v - n : v; };
            const int x = wrap(cx + dx - h, L), y = wrap(cy + dy - h, L), z = wrap(cz + dz - h, L);
            const int i = x + L * (y + L * z);
            const uint2 r = j6[i];
            const int d[3] = {dx, dy, dz};
            uint32_t M = 0, pos = 0, one = 0, two = 0;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const int J = (k & 1 ? d[k / 2] > 0 : d[k / 2] + 1 < l) ? coupling(r, k) : 0;
                const int weight = J < 0 ? -J : J;
                pos |= (J > 0 ? 1u : 0u) << k;
                one |= (weight == 1 ? 1u : 0u) << k;
                two |= (weight == 2 ? 1u : 0u) << k;
                M += (uint32_t)weight;
            }
            recs[q] = (uint32_t)q | M << kRecM | pos << kRecPos | one << kRecOne | two << kRecTwo;
            // fixed by an earlier wave: its residue class precedes this wave's (its spin is read below)
            if (wrap(ca + dx - h, l) + l * (wrap(cb + dy - h, l) + l * wrap(cc + dz - h, l)) < wave) {
                words[q] = (uint32_t)i;
                fixed |= 1u << (base / 32);
            } else {
                free_site = true;
                colour = (x + y + z) & 1;
            }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const bool mine = free_site && colour == c;
            const unsigned bal = __ballot_sync(kAll, mine);
            if (mine) s_free[warp][c][nfree[c] + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)q;
            nfree[c] += __popc(bal);
        }
    }
    __syncwarp();

    const int g = lane & 7;                                   // second steps: the lane's Philox block
    const uint32_t byte = (uint32_t)(lane & 3) * 0x11u + 0x40u;  // (prmt) bytes lane % 4 of two words
    // Of up to 32 sites, four at a time: bit(e, m) decides read 4g + m of site e; returns the
    // word of the lane's site.
    auto rounds = [&](int n, auto&& prepare, auto&& bit) {
        uint32_t word = 0;
#pragma unroll 2
        for (int r = 0; 4 * r < n; ++r) {
            uint32_t v[4], ctx[2];
            prepare(4 * r + (lane >> 3), v, ctx);
            unsigned b[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) b[m] = __ballot_sync(kAll, bit(m, v, ctx));
            const uint32_t mine = __byte_perm(__byte_perm(b[0], b[1], byte), __byte_perm(b[2], b[3], byte), 0x5410);
            if ((lane >> 2) == r) word = mine;
        }
        return word;
    };

    // initial words: of the free sites, and, once the wave before is done, of the fixed ones
    for (int c = 0; c < 2; ++c) {
        for (int base = 0; base < nfree[c]; base += 32) {
            const int n = min(32, nfree[c] - base);
            const uint16_t* list = s_free[warp][c] + base;
            const uint32_t word = rounds(
                n,
                [&](int e, uint32_t (&v)[4], uint32_t (&)[2]) {
                    draws.draw(kSweepInit, 8u * list[min(e, n - 1)] + (uint32_t)g, v);
                },
                [](int m, const uint32_t (&v)[4], const uint32_t (&)[2]) { return v[m] >> 31; });
            if (lane < n) words[list[lane]] = word;
        }
    }
    mp::wait_for_predecessor();
    mp::allow_successor();
    for (int q = lane; q < V; q += 32)
        if ((fixed >> (q / 32)) & 1u) words[q] = sp[words[q]] < 0 ? kAll : 0u;
    __syncwarp();

    const int entry_k = 2 * (lane & 7) - ((lane >> 3) & 1);  // thr[lane], lane < 16
    auto entry_of = [&](int sw) {
        return lane < 16 && entry_k >= 1 && entry_k < kThrRow && sw < a.S ? a.thr[(size_t)sw * kThrRow + entry_k] : 0u;
    };
    uint32_t entry = entry_of(0);
    for (int sw = 0; sw < a.S; ++sw) {
        if (lane < 16) thr[lane] = entry;
        entry = entry_of(sw + 1);
        for (int c = 0; c < 2; ++c) {
            for (int base = 0; base < nfree[c]; base += 32) {
                const int n = min(32, nfree[c] - base);
                const int q = s_free[warp][c][base + min(lane, n - 1)];
                const uint32_t rec = recs[q];
                const uint32_t self = words[q];
                const uint32_t nb[6] = {words[q + 1],  words[q - 1],  words[q + l],
                                        words[q - l], words[q + ll], words[q - ll]};
                uint32_t pos[6], mask[6], p[6];
                mp::unit_signs((rec >> kRecPos) & 63u, pos);
                mp::unit_signs((rec >> kRecOne) & 63u, mask);
#pragma unroll
                for (int k = 0; k < 6; ++k) p[k] = mp::logic<mp::kXor3>(self, nb[k], pos[k]);
                uint32_t P[4], term[6];
#pragma unroll
                for (int k = 0; k < 6; ++k) term[k] = p[k] & mask[k];
                mp::count_six(term, P[0], P[1], P[2]);
                P[3] = 0;
                if constexpr (!UNITJ) {
                    mp::unit_signs((rec >> kRecTwo) & 63u, mask);
#pragma unroll
                    for (int k = 0; k < 6; ++k) term[k] = p[k] & mask[k];
                    uint32_t t0, t1, t2;
                    mp::count_six(term, t0, t1, t2);
                    const uint32_t k1 = P[1] & t0, k2 = mp::maj3(P[2], t1, k1);
                    P[1] ^= t0;
                    P[2] = mp::logic<mp::kXor3>(P[2], t1, k1);
                    P[3] = t2 ^ k2;
                }
                // d = T - P, its borrow marks P > T
                const int M = (int)(rec >> kRecM) & 15, T = (M + 1) >> 1;
                const uint32_t T0 = mp::plane_mask(T, 0), T1 = mp::plane_mask(T, 1), T2 = mp::plane_mask(T, 2);
                const uint32_t d0 = T0 ^ P[0], b0 = ~T0 & P[0];
                const uint32_t d1 = mp::logic<mp::kXor3>(T1, P[1], b0), b1 = mp::logic<mp::kBorrow>(T1, P[1], b0);
                const uint32_t d2 = mp::logic<mp::kXor3>(T2, P[2], b1), b2 = mp::logic<mp::kBorrow>(T2, P[2], b1);
                const uint32_t need = (d0 | d1 | d2) & ~(b2 | P[3]);
                // the planes where the second step shifts them to: bits 2, 3 and 4 of a byte
                items[lane] = make_uint4(rotate_right(d0, 30), rotate_right(d1, 29), rotate_right(d2, 28),
                                         8u * (uint32_t)q | (uint32_t)M << 31);
                __syncwarp();
                const uint32_t lt = rounds(
                    n,
                    [&](int e, uint32_t (&v)[4], uint32_t (&ctx)[2]) {
                        const uint4 it = items[e];
                        draws.draw((uint32_t)sw, (it.w & 0x7FFFFFFFu) + (uint32_t)g, v);
                        // byte m: offset of read 4g + m's threshold, d * 4 + (M odd) * 32
                        const uint32_t odd = (uint32_t)((int)it.w >> 31) & 0x20202020u;
                        ctx[0] = mp::logic<kOrAnd>(odd, rotate_right(it.x, g), 0x04040404u);
                        ctx[0] = mp::logic<kOrAnd>(ctx[0], rotate_right(it.y, g), 0x08080808u);
                        ctx[0] = mp::logic<kOrAnd>(ctx[0], rotate_right(it.z, g), 0x10101010u);
                    },
                    [&](int m, const uint32_t (&v)[4], const uint32_t (&ctx)[2]) {
                        const uint32_t at = __byte_perm(ctx[0], 0u, 0x4440u + (uint32_t)m);
                        return (uint32_t)(v[m] < *reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(thr) + at));
                    });
                if (lane < n) words[q] = self ^ (~need | lt);
                __syncwarp();
            }
        }
    }

    // lane b: the weight of the positive terms of read b, each bond of the cube once, through
    // vertical counters over the lane's sites and a bit transpose a plane
    constexpr int kPlanesE = UNITJ ? 6 : 7;  // at most 11 sites a lane of weight 3 (6)
    uint32_t C[kPlanesE];
#pragma unroll
    for (int j = 0; j < kPlanesE; ++j) C[j] = 0;
    for (int q = lane; q < V; q += 32) {
        const uint32_t rec = recs[q], self = words[q];
        const uint32_t nb[3] = {words[q + 1], words[q + l], words[q + ll]};
        uint32_t one[3], two[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t p = mp::logic<mp::kXor3>(self, nb[k], mp::plane_mask((int)rec, kRecPos + 2 * k));
            one[k] = p & mp::plane_mask((int)rec, kRecOne + 2 * k);
            two[k] = UNITJ ? 0u : p & mp::plane_mask((int)rec, kRecTwo + 2 * k);
        }
        uint32_t w[4] = {mp::logic<mp::kXor3>(one[0], one[1], one[2]), mp::maj3(one[0], one[1], one[2]), 0u, 0u};
        if constexpr (!UNITJ) {
            const uint32_t t0 = mp::logic<mp::kXor3>(two[0], two[1], two[2]), t1 = mp::maj3(two[0], two[1], two[2]);
            w[2] = t1 ^ (w[1] & t0);
            w[1] ^= t0;
        }
        mp::vadd4(C, w);
    }
    int weight = 0;
#pragma unroll
    for (int j = 0; j < kPlanesE; ++j) weight += __popc(mp::warp_transpose(C[j], lane)) << j;
    // the first read of lowest energy
    const unsigned rank = (unsigned)weight * 32u + (unsigned)(4 * (lane & 7) + (lane >> 3));
    const unsigned least = __reduce_min_sync(kAll, rank);
    if (rank == least) sp[centre] = ((words[h + l * (h + l * h)] >> lane) & 1u) ? (int8_t)-1 : (int8_t)1;
}

// Exact zero-temperature fragment marginals (l = 1 or 3): the centre spin of each fragment
// is set by comparing the lowest cube energy over the cube's free spins with s_c = +1 and
// with s_c = -1 (+1 on a tie).
//
// The minima come from eliminating the spins plane by plane instead of enumerating all
// 2^27 states.  With T(s) the lowest energy of plane 0 (and its bonds to plane 1) given
// plane 1's nine spins s, T starts as plane 0's own energy of every state, and the nine z
// bonds are taken in one at a time: for spin q with z bond J,
//   T'(.., s_q, ..) = min(T(.., s_q, ..) + J, T(.., -s_q, ..) - J),
// a min-plus butterfly over bit q of the 512 states (s_q is plane 0's spin before the step
// and plane 1's after it).  Plane 2 likewise from above, and the two tables plus plane 1's
// own energy give the two minima.  A state that contradicts a fixed spin starts at kBarred.
// About 28 K additions and minima a cube instead of 2^27 energies: 232.4 ms -> 0.18 ms a
// call for four L = 12 lattices (27 launches of 2.4 us, the rest the energies and the host).
//
// A warp owns a fragment: lane holds bits 4 .. 8 of a state (spin q of a plane is bit q,
// q = dx + 3 dy, set meaning -1), its 16 registers bits 0 .. 3, so four butterflies stay in
// registers and five are shuffles.
constexpr int kTropWarps = 4;         // fragments per block
constexpr int kBarred = 1 << 20;      // above any cube energy (54 bonds of |J| <= 2)

__global__ void __launch_bounds__(kTropWarps * 32) fragment_tropical_kernel(int8_t* spins, const uint2* const* j6_ptrs,
                                                                            int L, int l, int wave)
{
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int inst = blockIdx.y, lane = threadIdx.x & 31;
    const int per = L / l;
    const int frag = blockIdx.x * kTropWarps + (int)(threadIdx.x >> 5);
    if (frag >= per * per * per) return;  // the whole warp
    const int ca = wave % l, cb = (wave / l) % l, cc = wave / (l * l);
    const int cx = ca + l * (frag % per), cy = cb + l * ((frag / per) % per), cz = cc + l * (frag / (per * per));
    int8_t* __restrict__ sp = spins + (size_t)inst * L * L * L;
    const int centre = cx + L * (cy + L * cz);
    if (l == 1) {  // no bonds inside the cube: a tie
        if (lane == 0) sp[centre] = 1;
        return;
    }
    // lane q < 27: cube site q, its value (0 = free) and its three forward bonds
    int value = 0, Jx = 0, Jy = 0, Jz = 0, at = 0;
    if (lane < 27) {
        const int dx = lane % 3, dy = (lane / 3) % 3, dz = lane / 9;
        const int x = cx + dx - 1, y = cy + dy - 1, z = cz + dz - 1;
        const int i = (x < 0 ? x + L : x >= L ? x - L : x) +
                      L * ((y < 0 ? y + L : y >= L ? y - L : y) + L * (z < 0 ? z + L : z >= L ? z - L : z));
        at = i;
        const uint2 rec = j6_ptrs[inst][i];
        Jx = coupling(rec, 0);
        Jy = coupling(rec, 2);
        Jz = coupling(rec, 4);
    }
    mp::wait_for_predecessor();  // the wave before: the only writer of spins
    mp::allow_successor();
    if (lane < 27) value = sp[at];
    const uint32_t fixed = __ballot_sync(kAll, value != 0), minus = __ballot_sync(kAll, value < 0);
    auto sign = [&](int bit) { return ((lane >> (bit - 4)) & 1) ? -1 : 1; };  // of a spin held by the lane
    // plane dz's own energy of the lane's 16 states (kBarred where a fixed spin disagrees)
    auto plane_energy = [&](int dz, int (&T)[16]) {
        const int b = 9 * dz;
        const int J01 = __shfl_sync(kAll, Jx, b), J12 = __shfl_sync(kAll, Jx, b + 1);
        const int J34 = __shfl_sync(kAll, Jx, b + 3), J45 = __shfl_sync(kAll, Jx, b + 4);
        const int J67 = __shfl_sync(kAll, Jx, b + 6), J78 = __shfl_sync(kAll, Jx, b + 7);
        const int J03 = __shfl_sync(kAll, Jy, b), J14 = __shfl_sync(kAll, Jy, b + 1);
        const int J25 = __shfl_sync(kAll, Jy, b + 2), J36 = __shfl_sync(kAll, Jy, b + 3);
        const int J47 = __shfl_sync(kAll, Jy, b + 4), J58 = __shfl_sync(kAll, Jy, b + 5);
        const int s4 = sign(4), s5 = sign(5), s6 = sign(6), s7 = sign(7), s8 = sign(8);
        const int high = J45 * s4 * s5 + J67 * s6 * s7 + J78 * s7 * s8 + J47 * s4 * s7 + J58 * s5 * s8;
        const int h1 = J14 * s4, h2 = J25 * s5, h3 = J34 * s4 + J36 * s6;  // fields on spins 1, 2, 3
        const uint32_t m = (fixed >> b) & 511u, v = (minus >> b) & 511u;
        const bool lane_ok = ((((uint32_t)lane << 4) ^ v) & m & 0x1F0u) == 0u;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int s0 = (e & 1) ? -1 : 1, s1 = (e & 2) ? -1 : 1, s2 = (e & 4) ? -1 : 1, s3 = (e & 8) ? -1 : 1;
            const int E = high + s1 * h1 + s2 * h2 + s3 * h3 + s0 * s1 * J01 + s1 * s2 * J12 + s0 * s3 * J03;
            T[e] = lane_ok && (((uint32_t)e ^ v) & m & 15u) == 0u ? E : kBarred;
        }
    };
    // the nine z bonds of plane dz to the plane above it
    auto eliminate = [&](int dz, int (&T)[16]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int J = __shfl_sync(kAll, Jz, 9 * dz + q);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                if (e & (1 << q)) continue;
                const int up = T[e], dn = T[e | (1 << q)];
                T[e] = min(up + J, dn - J);
                T[e | (1 << q)] = min(dn + J, up - J);
            }
        }
#pragma unroll
        for (int q = 4; q < 9; ++q) {
            const int J = __shfl_sync(kAll, Jz, 9 * dz + q);
#pragma unroll
            for (int e = 0; e < 16; ++e) T[e] = min(T[e] + J, __shfl_xor_sync(kAll, T[e], 1 << (q - 4)) - J);
        }
    };
    int U[16], V[16];
    plane_energy(0, U);
    eliminate(0, U);
    plane_energy(2, V);
    eliminate(1, V);
    int W[16];
    plane_energy(1, W);
    int m = 0x7FFFFFFF;
#pragma unroll
    for (int e = 0; e < 16; ++e) m = min(m, U[e] + V[e] + W[e]);
    // the centre is spin 4 of plane 1: bit 0 of the lane
#pragma unroll
    for (int o = 16; o > 1; o >>= 1) m = min(m, __shfl_xor_sync(kAll, m, o));
    const int mm = __shfl_sync(kAll, m, 1);
    if (lane == 0) sp[centre] = m <= mm ? (int8_t)1 : (int8_t)-1;
}

// A launch a wave.  Every wave after the first may start while its predecessor still runs: it
// reads couplings and keys, and draws its first words, before it waits for the predecessor's
// spins (the first one starts when everything before it on the stream is done).  Four L = 12
// lattices, exact: 0.23 -> 0.18 ms a call; one L = 10, annealed in cubes of 5: 6.2 -> 6.0.
template <class F>
int32_t launch_waves(int waves, dim3 grid, int threads, cudaStream_t st, const char* what, F&& launch)
{
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cfg.attrs = attr;
    for (int w = 0; w < waves; ++w) {
        cfg.numAttrs = w > 0 ? 1 : 0;
        const cudaError_t e = launch(&cfg, w);
        if (e != cudaSuccess) {
            cudaGetLastError();
            set_error("%s: %s", what, cudaGetErrorString(e));
            return SG_ECUDA;
        }
    }
    return SG_OK;
}

}  // namespace

int32_t launch_fragment_waves(int8_t* spins, const uint2* const* j6_ptrs, const RunKeys* keys, const uint32_t* thr,
                              int I, int L, int l, int S, bool unit, cudaStream_t st)
{
    FragArgs a{};
    a.spins = spins;
    a.j6_ptrs = j6_ptrs;
    a.keys = keys;
    a.thr = thr;
    a.L = L;
    a.l = l;
    a.S = S;
    a.lmagic = l == 1 ? 0u : (uint32_t)((0x100000000ull + (uint64_t)l - 1) / (uint64_t)l);
    const int per = L / l;
    const int frags = per * per * per;
    const dim3 grid((frags + kWarps - 1) / kWarps, I);
    return launch_waves(l * l * l, grid, kWarps * 32, st, "fragment_wave_kernel", [&](const cudaLaunchConfig_t* cfg, int w) {
        return cudaLaunchKernelEx(cfg, unit ? fragment_wave_kernel<true> : fragment_wave_kernel<false>, a, w);
    });
}

int32_t launch_fragment_tropical_waves(int8_t* spins, const uint2* const* j6_ptrs, int I, int L, int l,
                                       cudaStream_t st)
{
    const int per = L / l;
    const dim3 grid((per * per * per + kTropWarps - 1) / kTropWarps, I);
    return launch_waves(l * l * l, grid, kTropWarps * 32, st, "fragment_tropical_kernel",
                        [&](const cudaLaunchConfig_t* cfg, int w) {
                            return cudaLaunchKernelEx(cfg, fragment_tropical_kernel, spins, j6_ptrs, L, l, w);
                        });
}

}  // namespace sg
