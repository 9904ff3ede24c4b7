// metropolis.cuh -- the per-site Metropolis arithmetic shared by the sweep kernels
// (App. D.1 / D.2: flip when x = s_i * sum_j J_ij s_j >= 0, else when the draw
// u < thr[k], k = -x, thr[k] = floor(2^32 exp(-beta * 2k))).
//
// Spins are bit-packed: bit b of a 32-bit word is replica 32w + b of a site, 1 meaning
// spin -1.  With all |J| = 1 one word update is bit-sliced: for neighbour q with sign
// mask S_q (all ones when J_q < 0) the bond term J_q s_i s_q is negative -- the bond is
// satisfied -- exactly where self ^ n_q ^ S_q has a 1; six such indicator words go through
// a carry-save adder into three bit planes of the satisfied count c (0..6) of all 32
// replicas at once.  The flip costs dE = 2k with k = 2c - 6: free for c <= 3, else a draw
// decides with k = 2, 4, 6 for c = 4, 5, 6.
//
// Draws (our counter contract): the uniform U of replica 32w + b is A * 2^24 + B.  Bit j
// of its leading byte A is bit b of word j % 4 of Philox(site, sweep, 2w + j / 4, 0) --
// two blocks give the eight bit planes of all 32 leading bytes -- and B is the top 24 bits
// of word (32w + b) % 4 of Philox(site, sweep, (32w + b) / 4, 4).  U < thr[k] is decided
// by comparing A with the leading byte of thr[k] through a bit-sliced borrow chain, for
// all 32 replicas at once; only when the two bytes are equal (probability 1/256) is B
// drawn.
#pragma once
#include <stdint.h>

#include "philox.cuh"
#include "sg_internal.h"

namespace sg {
namespace mp {

constexpr int kRep = 32;  // replicas per spin word

// Programmatic dependent launch (PTX griddepcontrol, sm_90 and later).  Both are no-ops
// in a launch made without the programmatic-serialization attribute.
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_successor() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Three-input logic of the updates, spelled out: left to the compiler a word costs about
// eight operations more.
template <int TABLE>
__device__ __forceinline__ uint32_t logic(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(d) : "r"(a), "r"(b), "r"(c), "n"(TABLE));
    return d;
}
constexpr int kXor3 = 0x96, kMaj = 0xE8, kSelect = 0xCA /* a ? b : c */, kBorrow = 0x8E /* majority of ~a, b, c */,
              kAndEqual = 0x90 /* a where b = c */;

__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) { return logic<kMaj>(a, b, c); }

// Bytes of x, or their sign bits replicated, picked by `sel` (prmt).
__device__ __forceinline__ uint32_t sign_bytes(uint32_t x, uint32_t sel)
{
    uint32_t d;
    asm("prmt.b32 %0, %1, %1, %2;" : "=r"(d) : "r"(x), "r"(sel));
    return d;
}

// Sign masks of the six couplings of a site with all |J| = 1, from its byte of sign bits
// (bit q set when J_q < 0; q = +x, -x, +y, -y, +z, -z): two multiplies spread the bits to the
// tops of bytes.
__device__ __forceinline__ void unit_signs(uint32_t bits, uint32_t (&S)[6])
{
    const uint32_t lo = bits * 0x10204080u, hi = bits * 0x408u;
    S[0] = sign_bytes(lo, 0x8888u), S[1] = sign_bytes(lo, 0x9999u), S[2] = sign_bytes(lo, 0xAAAAu);
    S[3] = sign_bytes(lo, 0xBBBBu), S[4] = sign_bytes(hi, 0x8888u), S[5] = sign_bytes(hi, 0x9999u);
}

// How the thresholds of a sweep can accept: not at all (all of them zero), only where the
// leading byte of a draw is 0 (every threshold below 2^24), or by a full compare.
enum Mode { kNoDraws = 0, kTailOnly = 1, kCompare = 2 };

// Bit planes (c0, c1, c2) of the number of satisfied bonds of every replica.
__device__ __forceinline__ void satisfied_count(uint32_t self, const uint32_t (&n)[6], const uint32_t (&S)[6],
                                                uint32_t& c0, uint32_t& c1, uint32_t& c2)
{
    uint32_t a[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) a[q] = logic<kXor3>(self, n[q], S[q]);
    const uint32_t s1 = logic<kXor3>(a[0], a[1], a[2]), k1 = maj3(a[0], a[1], a[2]);
    const uint32_t s2 = logic<kXor3>(a[3], a[4], a[5]), k2 = maj3(a[3], a[4], a[5]);
    c0 = s1 ^ s2;
    const uint32_t t = s1 & s2;
    c1 = logic<kXor3>(k1, k2, t);
    c2 = maj3(k1, k2, t);
}

// The eight bit planes of the leading draw bytes of word w at (site, sweep).
__device__ __forceinline__ void lead_planes(uint32_t site, uint32_t sweep, uint32_t w, const RunKeys& key,
                                            uint32_t (&A)[8])
{
    const Philox4 p0 = philox4x32_10(site, sweep, 2u * w, kDomainMetropolis, key.k0, key.k1);
    const Philox4 p1 = philox4x32_10(site, sweep, 2u * w + 1u, kDomainMetropolis, key.k0, key.k1);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        A[j] = p0.v[j];
        A[4 + j] = p1.v[j];
    }
}

// Threshold planes of a word: tp[8 * m + j], m = 0, 1, 2 for k = 2, 4, 6, has bit b equal to
// bit 24 + j of the threshold of slot 32w + b (of the sweep's row for SA).
__device__ __forceinline__ uint32_t threshold_plane_bit(uint32_t thr, int j) { return (thr >> (24 + j)) & 1u; }

// One word of unit-coupling updates.  valid: replicas that exist.  tp: the word's 24
// threshold planes.  Returns the replicas that flip now in *flip and those whose leading
// bytes tied in *tie (decided later by resolve_tie_bits); c0..c2 are the satisfied-count
// planes before the flip.
__device__ __forceinline__ void update_word_unit(uint32_t self, const uint32_t (&n)[6], const uint32_t (&S)[6],
                                                 uint32_t valid, const uint32_t (&tp)[24], const uint32_t (&A)[8],
                                                 uint32_t* flip, uint32_t* tie, uint32_t* c0, uint32_t* c1,
                                                 uint32_t* c2)
{
    satisfied_count(self, n, S, *c0, *c1, *c2);
    // A < T through the borrow of A - T, least significant plane first: the borrow out
    // of a plane is the majority of (~A_j, T_j, borrow in), one three-input operation
    uint32_t lt = 0, eq = valid & *c2;  // c >= 4: the flip raises the energy
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        // threshold plane of each replica's k: c = 4 -> k = 2, c = 5 -> 4, c = 6 -> 6
        const uint32_t T = logic<kSelect>(*c1, tp[16 + j], logic<kSelect>(*c0, tp[8 + j], tp[j]));
        lt = j == 0 ? T & ~A[0] : logic<kBorrow>(A[j], T, lt);
        eq = logic<kAndEqual>(eq, A[j], T);
    }
    *flip = (~*c2 | lt) & valid;
    *tie = eq;
}

// The same where every threshold is below 2^24 (a draw whose leading byte is 0 ties, every
// other one rejects), and where all thresholds are zero.
__device__ __forceinline__ void update_word_tail(uint32_t self, const uint32_t (&n)[6], const uint32_t (&S)[6],
                                                 uint32_t valid, const uint32_t (&A)[8], uint32_t* flip, uint32_t* tie,
                                                 uint32_t* c0, uint32_t* c1, uint32_t* c2)
{
    satisfied_count(self, n, S, *c0, *c1, *c2);
    const uint32_t any = (A[0] | A[1] | A[2]) | (A[3] | A[4] | A[5]) | (A[6] | A[7]);
    *flip = ~*c2 & valid;
    *tie = valid & *c2 & ~any;
}
__device__ __forceinline__ uint32_t update_word_free(uint32_t self, const uint32_t (&n)[6], const uint32_t (&S)[6],
                                                     uint32_t valid)
{
    uint32_t c0, c1, c2;
    satisfied_count(self, n, S, c0, c1, c2);
    return ~c2 & valid;
}

// Satisfied-count planes after flipping `flip` (a flip turns c into 6 - c).
__device__ __forceinline__ void count_after_flip(uint32_t flip, uint32_t c0, uint32_t& c1, uint32_t& c2)
{
    const uint32_t n1 = c1 ^ (flip & ~c0);
    const uint32_t n2 = c2 ^ (flip & ~(c0 & c1));
    c1 = n1;
    c2 = n2;
}

// Adds the 4-bit value a of every replica to the vertical counter V.
template <int NB>
__device__ __forceinline__ void vadd4(uint32_t (&V)[NB], const uint32_t (&a)[4])
{
    uint32_t c = 0;
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        const uint32_t x = j < 4 ? a[j] : 0u, t = logic<kXor3>(V[j], x, c);
        c = maj3(V[j], x, c);
        V[j] = t;
    }
}

// Adds the 3-bit value (a0, a1, a2) of every replica to the vertical counter V.
template <int NB>
__device__ __forceinline__ void vadd3(uint32_t (&V)[NB], uint32_t a0, uint32_t a1, uint32_t a2)
{
    uint32_t c = V[0] & a0;
    V[0] ^= a0;
    {
        const uint32_t t = V[1] ^ a1 ^ c;
        c = maj3(V[1], a1, c);
        V[1] = t;
    }
    {
        const uint32_t t = V[2] ^ a2 ^ c;
        c = maj3(V[2], a2, c);
        V[2] = t;
    }
#pragma unroll
    for (int j = 3; j < NB; ++j) {
        const uint32_t t = V[j] & c;
        V[j] ^= c;
        c = t;
    }
}

// Value of replica b in the vertical counter V.
template <int NB>
__device__ __forceinline__ int vcount(const uint32_t (&V)[NB], int b)
{
    int v = 0;
#pragma unroll
    for (int j = 0; j < NB; ++j) v |= (int)((V[j] >> b) & 1u) << j;
    return v;
}

// 32 x 32 bit transpose across a full warp: on return lane r holds the word whose bit l
// is bit r of lane l's x.
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, int lane)
{
    const uint32_t masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int st = 0; st < 5; ++st) {
        const int s = 16 >> st;
        const uint32_t m = masks[st];
        const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, x, s);
        x = (lane & s) ? (((other >> s) & m) | (x & ~m)) : ((x & m) | ((other & m) << s));
    }
    return x;
}

// Decides tied draws: for each replica b of `tie`, k from its satisfied count (c0, c1 of
// c = 4, 5, 6), accepted when the threshold has low bits and the draw's low 24 bits are
// below them (a threshold of exactly A * 2^24 rejects).  thr(b, k) = row[b * stride + k].
// Out of line: it runs rarely, and one copy keeps the sweep loops small.
static __device__ __noinline__ uint32_t resolve_tie_bits(uint32_t tie, uint32_t c0, uint32_t c1,
                                                         const uint32_t* __restrict__ row, int stride, uint32_t site,
                                                         uint32_t sweep, uint32_t w, uint32_t k0, uint32_t k1)
{
    uint32_t acc = 0;
    while (tie) {
        const int b = __ffs(tie) - 1;
        tie &= tie - 1u;
        const int c = 4 + (int)((c0 >> b) & 1u) + 2 * (int)((c1 >> b) & 1u);
        const int k = 2 * c - 6;
        const uint32_t low = row[b * stride + k] & 0xFFFFFFu;
        if (!low) continue;
        const uint32_t slot = 32u * w + (uint32_t)b;
        const Philox4 t = philox4x32_10(site, sweep, slot >> 2, kDomainTail, k0, k1);
        const uint32_t m = slot & 3u;
        const uint32_t word = m == 0 ? t.v[0] : m == 1 ? t.v[1] : m == 2 ? t.v[2] : t.v[3];
        if ((word >> 8) < low) acc |= 1u << b;
    }
    return acc;
}

// ---- general couplings: |J| <= 2, bonds may be absent ----
//
// With c the weight of a site's satisfied bonds (sum of their |J|) and M the weight of all six,
// a flip costs dE = 2k, k = 2c - M.  With h = M / 2 rounded down, u = c - h is at least 1 exactly
// where k > 0, and then k = 2u, or 2u - 1 when M is odd: six thresholds a parity, picked by the
// three planes of u.  Replica by replica, as it was, a warp followed its slowest replica through
// 32 branches (19 lanes of 32 active, 30 % of the issue slots): a half sweep of 100 replicas of an
// L = 24 lattice took 8.4 us, one launch of the row kernel.  In planes it takes 3.6, and 2.5 on
// clusters, which need no launch for it.  Tempering sums its energies in the same counters as for
// unit couplings.
//
// Threshold planes of a word: gp[general_plane(odd, j, u)] has bit b equal to bit 24 + j of
// replica b's threshold of k = 2u - odd; j = 8: whether its low 24 bits are nonzero.
constexpr int kGeneralPlanes = 2 * 9 * 8;
__device__ __forceinline__ int general_plane(int odd, int j, int u) { return (odd * 9 + j) * 8 + u - 1; }

// Plane p of a word, one threshold row serving all its replicas; p without a meaning gives 0.
__device__ __forceinline__ uint32_t general_plane_of(int p, const uint32_t* row)
{
    const int u = p % 8 + 1, j = p / 8 % 9;
    if (u > 6) return 0u;
    const uint32_t t = row[2 * u - p / 72];
    return (j < 8 ? threshold_plane_bit(t, j) : (uint32_t)((t & 0xFFFFFFu) != 0u)) ? ~0u : 0u;
}

// The planes of `words` words, thr[32 * w + b][k] the threshold of replica b: a lane takes a
// replica, the warp a word and a k, in turn (a loop over replicas a plane took as long as the
// updates of a small launch).  Threads beyond the last whole warp only help where there is none.
__device__ __forceinline__ void general_planes(uint32_t* gp, const uint32_t* thr, int stride, int words, int tid,
                                               int nthreads)
{
    if (nthreads < 32) {
        for (int q = tid; q < words * kGeneralPlanes; q += nthreads) {
            const int p = q % kGeneralPlanes, u = p % 8 + 1, j = p / 8 % 9;
            uint32_t plane = 0;
            for (int b = 0; u <= 6 && b < 32; ++b) {
                const uint32_t t = thr[(32 * (q / kGeneralPlanes) + b) * stride + 2 * u - p / 72];
                plane |= (j < 8 ? threshold_plane_bit(t, j) : (uint32_t)((t & 0xFFFFFFu) != 0u)) << b;
            }
            gp[q] = plane;
        }
        return;
    }
    const int warps = nthreads >> 5, lane = tid & 31;
    if ((tid >> 5) >= warps) return;
    for (int q = tid >> 5; q < 12 * words; q += warps) {
        const int w = q / 12, k = q % 12 + 1;
        const uint32_t t = thr[(32 * w + lane) * stride + k];
        uint32_t mine = 0;
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const uint32_t plane = __ballot_sync(0xFFFFFFFFu, j < 8 ? (t >> (24 + j)) & 1u : (t & 0xFFFFFFu) != 0u);
            if (lane == j) mine = plane;
        }
        if (lane < 9) gp[w * kGeneralPlanes + general_plane(k & 1, lane, (k + 1) >> 1)] = mine;
    }
}

// Adds the planes of six indicator words: their count 0..6.
__device__ __forceinline__ void count_six(const uint32_t (&a)[6], uint32_t& c0, uint32_t& c1, uint32_t& c2)
{
    const uint32_t s1 = logic<kXor3>(a[0], a[1], a[2]), k1 = maj3(a[0], a[1], a[2]);
    const uint32_t s2 = logic<kXor3>(a[3], a[4], a[5]), k2 = maj3(a[3], a[4], a[5]);
    const uint32_t t = s1 & s2;
    c0 = s1 ^ s2;
    c1 = logic<kXor3>(k1, k2, t);
    c2 = maj3(k1, k2, t);
}

__device__ __forceinline__ uint32_t plane_mask(int v, int bit) { return 0u - ((uint32_t)(v >> bit) & 1u); }

// The satisfied weight from the satisfied bonds of weight 1 and of weight 2.
__device__ __forceinline__ void satisfied_weight(const uint32_t (&one)[6], const uint32_t (&two)[6], uint32_t (&c)[4])
{
    uint32_t o0, o1, o2, t0, t1, t2;
    count_six(one, o0, o1, o2);
    count_six(two, t0, t1, t2);
    c[0] = o0;
    c[1] = o1 ^ t0;
    const uint32_t k1 = o1 & t0;
    c[2] = logic<kXor3>(o2, t1, k1);
    c[3] = t2 ^ maj3(o2, t1, k1);
}

// The replicas of a word that flip.  c: planes of the satisfied weight, M the weight of all
// bonds, gp the word's threshold planes, row[b * stride + k] the threshold of replica b (read
// for ties alone).  Without DRAWS all thresholds are zero.
template <bool DRAWS>
__device__ __forceinline__ uint32_t flips_general(const uint32_t (&c)[4], int M, uint32_t valid,
                                                  const uint32_t* __restrict__ gp, const uint32_t* __restrict__ row,
                                                  int stride, const uint32_t (&A)[8], uint32_t site, uint32_t sweep,
                                                  uint32_t w, const RunKeys& key)
{
    // u = c - h, four planes; its borrow marks c < h
    const int h = M >> 1, odd = M & 1;
    const uint32_t h0 = plane_mask(h, 0), h1 = plane_mask(h, 1), h2 = plane_mask(h, 2);
    const uint32_t u0 = c[0] ^ h0, b0 = ~c[0] & h0;
    const uint32_t u1 = logic<kXor3>(c[1], h1, b0), b1 = logic<kBorrow>(c[1], h1, b0);
    const uint32_t u2 = logic<kXor3>(c[2], h2, b1), b2 = logic<kBorrow>(c[2], h2, b1);
    const uint32_t u3 = c[3] ^ b2, b3 = ~c[3] & b2;
    const uint32_t need = ~b3 & (u0 | u1 | u2 | u3);
    if (!DRAWS) return ~need & valid;
    auto pick = [&](int j) {  // each replica's plane j
        const uint4 x = *reinterpret_cast<const uint4*>(gp + general_plane(odd, j, 1));
        const uint2 y = *reinterpret_cast<const uint2*>(gp + general_plane(odd, j, 5));
        const uint32_t high = logic<kSelect>(u1, y.y, logic<kSelect>(u0, y.x, x.w));   // u = 6, 5, 4
        const uint32_t low = logic<kSelect>(u1, logic<kSelect>(u0, x.z, x.y), x.x);    // u = 3, 2, 1
        return logic<kSelect>(u2, high, low);
    };
    uint32_t lt = 0, tie = need & valid;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t T = pick(j);
        lt = logic<kBorrow>(A[j], T, lt);
        tie = logic<kAndEqual>(tie, A[j], T);
    }
    tie &= pick(8);
    uint32_t flip = (~need | lt) & valid;
    while (tie) {  // (about one word in ten has one)
        const int b = __ffs((int)tie) - 1;
        tie &= tie - 1u;
        const int u = (int)((u0 >> b) & 1u) | (int)((u1 >> b) & 1u) << 1 | (int)((u2 >> b) & 1u) << 2;
        const uint32_t low = row[b * stride + 2 * u - odd] & 0xFFFFFFu;
        const uint32_t slot = 32u * w + (uint32_t)b;
        const Philox4 t = philox4x32_10(site, sweep, slot >> 2, kDomainTail, key.k0, key.k1);
        const uint32_t p = slot & 3u;
        const uint32_t word = p == 0 ? t.v[0] : p == 1 ? t.v[1] : p == 2 ? t.v[2] : t.v[3];
        if ((word >> 8) < low) flip |= 1u << b;
    }
    return flip;
}

// One word of a site with couplings J[q].  Returns the flips; c: the planes of the satisfied
// weight before them, *M the weight of all bonds.
__device__ __forceinline__ uint32_t update_word_general(uint32_t self, const uint32_t (&n)[6], const int (&J)[6],
                                                        uint32_t valid, const uint32_t* __restrict__ gp,
                                                        const uint32_t* __restrict__ row, int stride,
                                                        const uint32_t (&A)[8], uint32_t site, uint32_t sweep,
                                                        uint32_t w, const RunKeys& key, uint32_t (&c)[4], int* M)
{
    uint32_t one[6], two[6];
    int m = 0;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const uint32_t satisfied = logic<kXor3>(self, n[q], J[q] < 0 ? ~0u : 0u);
        const int weight = J[q] < 0 ? -J[q] : J[q];
        one[q] = weight == 1 ? satisfied : 0u;
        two[q] = weight == 2 ? satisfied : 0u;
        m += weight;
    }
    *M = m;
    satisfied_weight(one, two, c);
    return flips_general<true>(c, m, valid, gp, row, stride, A, site, sweep, w, key);
}

// Planes of the satisfied weight after the flips (a flip turns c into M - c).
__device__ __forceinline__ void weight_after_flip(uint32_t flip, int M, uint32_t (&c)[4])
{
    uint32_t borrow = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t m = plane_mask(M, j), d = logic<kXor3>(m, c[j], borrow);
        borrow = logic<kBorrow>(m, c[j], borrow);
        c[j] = logic<kSelect>(flip, d, c[j]);
    }
}

}  // namespace mp
}  // namespace sg
