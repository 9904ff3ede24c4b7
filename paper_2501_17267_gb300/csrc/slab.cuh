// slab.cuh -- sweeps of a lattice held in the shared memory of a thread-block cluster
// (App. D.1 / D.2, unit couplings): the machinery shared by the annealing kernels
// (cluster.cu) and the tempering kernel (ptcluster.cu).
//
// Block r of a cluster of C blocks holds z-planes [r L / C, (r + 1) L / C) of one 32-bit word a
// site, between two halo planes: a copy of the plane below its slab and of the plane above it.
// (C need not divide L; slabs then differ by a plane, and the largest one counts: 20 L = 50
// lattices take C = 7, slabs of at most 8 planes, instead of C = 5.)  A half sweep updates the
// sites of one colour from the words of the other.
//
// Columns.  A lane owns a column (y, j): the colour's site of x pair j in row y of every
// plane of its segment, walked upwards.  With M(z) the other word of the pair in plane z --
// the site's x neighbour -- the site's lower z neighbour is M(z - 1) and its upper one
// M(z + 1), so an item loads five words instead of seven and its addresses follow from the
// previous item's by a few additions.  The draws of an item are made while the one before it
// is decided, so that multiplies and logic share the pipes.  A word of 32 attempts in tempering
// at L = 64 costs 243 warp instructions, 130 of them on the logic pipe, and 403 cycles of a
// partition (289, 155 and 491 when every item worked out its own geometry and drew for
// itself); on this GPU a three-input logic operation takes 2 cycles of that and a widening
// multiply beside it 2.1, 335 for what is left.
//
// Neighbour blocks.  After its part of a half sweep a warp copies its updated words of the
// slab's two faces into the neighbours' halo planes by st.async, whose bytes complete on a
// barrier in the neighbour's shared memory.  A block starts the next half sweep once its own
// warps have met (__syncthreads) and both neighbours' words have arrived.  A cluster barrier
// with release costs 370 to 470 cycles (its fence alone 330), the push about 250, most of
// which the next half sweep's first draws hide.  Nothing else orders the blocks, and
// nothing has to: a face word is pushed only after its warp has read the halo words the
// neighbour is going to overwrite, and the neighbour overwrites them only after all of this
// block's face words have arrived there.  Waits are bounded; a block whose wait gave up still
// waits (bounded too) for the words of the half sweep it is in before it leaves.
//
// Ties (draws whose leading byte equals the threshold's, about 1.5 a warp and item) go to a
// queue of the warp, by ballot, and are decided 32 at a time.
#pragma once
#include <stdint.h>

#include "metropolis.cuh"
#include "philox.cuh"
#include "sg_internal.h"

namespace sg {
namespace slab {

constexpr int kMaxThreads = 512;
constexpr int kMaxC = 16;       // blocks a cluster (more than 8: the kernels ask for it, allow_shared)
constexpr int kTieCap = 64;     // queue entries a warp: decided from 32, an item adds at most 32
constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr long long kDrainCycles = 1ll << 31;  // what a wait that gave up still allows (about a second)

// ---------------------------------------------------------------- PTX primitives
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// the address of `addr` (of this block's shared memory) in block `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank)
{
    uint32_t d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
    return d;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// the one arrival of a phase, with the bytes that complete it
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Polls for phase `parity`; false when it came after `limit` cycles or not at all.  The words on
// their way are waited for beyond the limit too, again with a limit: the block must not leave, nor
// its shared memory serve something else, while they can still arrive.
__device__ __forceinline__ bool mbar_poll(uint64_t* bar, uint32_t parity, long long limit)
{
    const long long t0 = clock64();
    long long t;
    bool here;
    do {
        here = mbar_try(bar, parity);
        t = clock64() - t0;
    } while (!here && t < limit + kDrainCycles);
    return here && t < limit;
}
static __device__ __noinline__ bool mbar_poll_apart(uint64_t* bar, uint32_t parity, long long limit)
{
    return mbar_poll(bar, parity, limit);
}

// Waits for phase `parity`, for `limit` cycles; false when it gave up.  (With a limit of 0 the
// kernels start with their flags set, as if every wait had given up: asking for that here, before
// the first try, cost 40 temperatures at L = 16 3 %.)  APART: the polling out of line, where it
// takes registers from a half sweep that has none to spare (resident blocks: 1.00 ms against 1.04
// at L = 4 with 8 replicas and 1000 sweeps; elsewhere the call costs more: 48 temperatures at
// L = 32 3.66 ms in line, 3.72 apart).
template <bool APART>
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit)
{
    if (mbar_try(bar, parity)) return true;
    return APART ? mbar_poll_apart(bar, parity, limit) : mbar_poll(bar, parity, limit);
}

// one word into another block's shared memory, its four bytes counted on that block's `bar`
__device__ __forceinline__ void push_word(uint32_t addr, uint32_t value, uint32_t bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(value),
                 "r"(bar)
                 : "memory");
}

// shared words and bytes by address: an item's addresses are sums of a few registers
__device__ __forceinline__ uint32_t ld_word(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_byte(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_quad(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(addr)
                 : "memory");
    return v;
}
// the same when `p` is nonzero, predicated rather than branched around
__device__ __forceinline__ void st_word_if(uint32_t p, uint32_t addr, uint32_t v)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.shared.u32 [%1], %2;\n\t}" ::"r"(p), "r"(addr),
                 "r"(v)
                 : "memory");
}
__device__ __forceinline__ void st_quad_if(uint32_t p, uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.shared.v4.u32 [%1], {%2, %3, %4, %5};\n\t}" ::"r"(p),
        "r"(addr), "r"(x), "r"(y), "r"(z), "r"(w)
        : "memory");
}
__device__ __forceinline__ void xor_word(uint32_t addr, uint32_t v)
{
    asm volatile("red.shared.xor.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

using mp::kAndEqual;
using mp::kBorrow;
using mp::kMaj;
using mp::kSelect;
using mp::kXor3;
using mp::logic;
using mp::sign_bytes;

// ---------------------------------------------------------------- draws

// The two blocks of a site's leading-byte planes share their first two rounds but for the
// words that depend on the sweep alone: those are made once a half sweep, and a site costs
// 34 multiplies instead of 40.
struct Draws {
    uint32_t k0, k1;                  // key
    uint32_t x0, y0, z0, x1, y1, z1;  // of the sweep and the word

    __device__ __forceinline__ void set_sweep(uint32_t sweep, uint32_t word)
    {
        const uint32_t r0 = k0 + kPhiloxWeylA, r1 = k1 + kPhiloxWeylB;
        uint32_t hi, lo;
        philox_mulhilo(kPhiloxMulB, 2u * word, &hi, &lo);
        x0 = lo ^ r0;
        philox_mulhilo(kPhiloxMulA, hi ^ sweep ^ k0, &hi, &z0);
        y0 = hi ^ r1;
        philox_mulhilo(kPhiloxMulB, 2u * word + 1u, &hi, &lo);
        x1 = lo ^ r0;
        philox_mulhilo(kPhiloxMulA, hi ^ sweep ^ k0, &hi, &z1);
        y1 = hi ^ r1;
    }
    __device__ __forceinline__ void planes(uint32_t site, uint32_t (&A)[8]) const
    {
        uint32_t hA, lA, hB, lB;
        philox_mulhilo(kPhiloxMulA, site, &hA, &lA);
        philox_mulhilo(kPhiloxMulB, hA ^ kDomainMetropolis ^ k1, &hB, &lB);
        uint32_t p[4] = {hB ^ x0, lB, lA ^ y0, z0}, q[4] = {hB ^ x1, lB, lA ^ y1, z1};
#pragma unroll
        for (int r = 2; r < 10; ++r) {
            const uint32_t r0 = k0 + (uint32_t)r * kPhiloxWeylA, r1 = k1 + (uint32_t)r * kPhiloxWeylB;
            uint32_t ha, la, hb, lb;
            philox_mulhilo(kPhiloxMulA, p[0], &ha, &la);
            philox_mulhilo(kPhiloxMulB, p[2], &hb, &lb);
            p[0] = hb ^ p[1] ^ r0, p[1] = lb, p[2] = ha ^ p[3] ^ r1, p[3] = la;
            philox_mulhilo(kPhiloxMulA, q[0], &ha, &la);
            philox_mulhilo(kPhiloxMulB, q[2], &hb, &lb);
            q[0] = hb ^ q[1] ^ r0, q[1] = lb, q[2] = ha ^ q[3] ^ r1, q[3] = la;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            A[j] = p[j];
            A[4 + j] = q[j];
        }
    }
};

// ---------------------------------------------------------------- geometry

// (Kept in shared memory: most of it is read once a unit.)
struct Geometry {
    int L, H, LL, zc, z0, zdn;    // side, half, plane, planes of the slab, first of them, planes of the slab below
    int cols, chunks;             // columns of a colour, warps of columns
    int segments, seglen, units;  // z segments of a column, their planes, (segment, chunk) pairs
    uint32_t Hmagic, Lmagic;      // ceil(2^32 / H), ceil(2^32 / L)

    // Splits the columns into segments so that the warps of a block finish together: the
    // fewest rounds of items, a segment's start counted as half an item.
    __device__ __forceinline__ void init(int L_, int C, int r, int warps, uint32_t Hmagic_)
    {
        L = L_;
        H = L >> 1;
        LL = L * L;
        z0 = first(L, C, r);
        zc = first(L, C, r + 1) - z0;
        zdn = r == 0 ? L - first(L, C, C - 1) : z0 - first(L, C, r - 1);
        cols = L * H;
        chunks = (cols + 31) / 32;
        Hmagic = Hmagic_;
        Lmagic = 0xFFFFFFFFu / (uint32_t)L + 1u;
        segments = 1;
        seglen = zc;
        int best = 0x7FFFFFFF;
        for (int s = 1; s <= zc; ++s) {
            const int len = (zc + s - 1) / s;
            if ((zc + len - 1) / len != s) continue;  // the last segment would be empty
            const int cost = (chunks * s + warps - 1) / warps * (2 * len + 1);
            if (cost < best) {
                best = cost;
                segments = s;
                seglen = len;
            }
        }
        units = chunks * segments;
    }
    __host__ __device__ static int first(int L, int C, int r) { return r * L / C; }  // block r's first plane
    // of the largest slab: its planes, its words with both halos, its sites
    __host__ __device__ static int planes(int L, int C) { return (L + C - 1) / C; }
    __host__ __device__ static size_t words(int L, int C) { return (size_t)(planes(L, C) + 2) * L * L; }
    __host__ __device__ static size_t sites(int L, int C) { return (size_t)planes(L, C) * L * L; }
};

// Whether clusters of C blocks can hold side L: C of them have a plane, and fewer would not do
// with slabs as thin.
inline bool worth(int L, int C) { return C <= L && (C == 1 || Geometry::planes(L, C) < Geometry::planes(L, C - 1)); }

// Dynamic shared memory of a block: halo, slab and halo words, the slab's sign bytes in
// storage order, the warps' tie queues.
__host__ __device__ inline size_t smem_queue_offset(int L, int C)
{
    return (Geometry::words(L, C) * 4 + Geometry::sites(L, C) + 15) & ~(size_t)15;
}
__host__ __device__ inline size_t smem_bytes(int L, int C, int threads)
{
    return smem_queue_offset(L, C) + (size_t)(threads / 32) * kTieCap * sizeof(uint4);
}

// A lane's column in one unit.  Addresses are bytes of shared memory; f is the offset of
// the far x neighbour (the near one, the pair's other word, is +-4H away).
constexpr uint32_t kOdd = 1, kLive = 2, kBottom = 4, kTop = 8;  // Unit::flags

struct Unit {
    uint32_t base;    // word of the even-x site in the segment's first plane
    int site;         // its logical site
    int f0, fsum;     // offset of the far x neighbour of an even-x site; that plus an odd-x site's
    int yp, ym;       // offsets of the y neighbours
    int n;            // planes
    uint32_t flags;   // (y + z) of the first plane odd; a column of the lattice; at the slab's bottom, top

    __device__ __forceinline__ void locate(const Geometry& g, uint32_t w0, int u, int lane)
    {
        const int L = g.L, H = g.H, LL = g.LL;
        const int seg = g.segments == 1 ? 0 : u / g.chunks, ch = u - seg * g.chunks;
        const int col = ch * 32 + lane;
        const bool live = col < g.cols;
        const int c = live ? col : 0;
        const int y = H == 1 ? c : (int)__umulhi((uint32_t)c, g.Hmagic), j = c - y * H;
        const int zb = seg * g.seglen;
        n = min(g.seglen, g.zc - zb);
        base = w0 + 4u * (uint32_t)((zb * L + y) * L + j);
        site = ((g.z0 + zb) * L + y) * L + 2 * j;
        f0 = 4 * (H + (j == 0 ? H - 1 : -1));
        fsum = 4 * ((j == 0 ? H - 1 : -1) + (j + 1 == H ? 1 - H : 1));
        yp = 4 * (y + 1 == L ? L - LL : L);
        ym = 4 * (y == 0 ? LL - L : -L);
        flags = ((uint32_t)(y + g.z0 + zb) & kOdd) | (live ? kLive : 0u) | (zb == 0 ? kBottom : 0u) |
                (zb + n == g.zc ? kTop : 0u);
    }
};

// Copies the block's planes and both halo planes of a word array [N] (stride words a site)
// and the slab's sign bytes into shared memory.  A sign byte's x bits become (near, far):
// the near neighbour of an even x is at +x, of an odd x at -x.
__device__ __forceinline__ void load_slab(const Geometry& g, const uint32_t* __restrict__ src, int stride,
                                          const uint8_t* __restrict__ j1, uint32_t* w, uint8_t* sgn)
{
    const int slab = g.zc * g.LL;
    const int below = ((g.z0 == 0 ? g.L : g.z0) - 1) * g.LL, above = (g.z0 + g.zc == g.L ? 0 : g.z0 + g.zc) * g.LL;
    const int first = g.z0 * g.LL;
    for (int q = threadIdx.x; q < slab; q += blockDim.x) {
        w[q] = src[(size_t)(first + q) * stride];
        const int row = q / g.L, pos = q - row * g.L;
        const int odd = pos >= g.H, x = odd ? 2 * (pos - g.H) + 1 : 2 * pos;
        const uint32_t b = j1[first + row * g.L + x];
        sgn[q] = (uint8_t)(odd ? (b & 0x3Cu) | ((b & 1u) << 1) | ((b >> 1) & 1u) : b & 0x3Fu);
    }
    for (int q = threadIdx.x; q < g.LL; q += blockDim.x) {
        w[q - g.LL] = src[(size_t)(below + q) * stride];
        w[slab + q] = src[(size_t)(above + q) * stride];
    }
}

__device__ __forceinline__ uint32_t word_valid_bits(int R, int w)
{
    const int left = R - 32 * w;
    return left >= 32 ? 0xFFFFFFFFu : left <= 0 ? 0u : (1u << left) - 1u;
}

// ---------------------------------------------------------------- updates

// What a half sweep does: mp::Mode by its thresholds, or no update at all, for the energies of
// the words as they are.
constexpr int kNoDraws = mp::kNoDraws, kTailOnly = mp::kTailOnly, kCompare = mp::kCompare, kCountOnly = 3;

// Thresholds of a word: plane j of k = 2, 4, 6 in tp[j] (bit b: replica b), and the
// replicas whose threshold has nonzero low 24 bits -- only those can accept on a tie.
struct Planes {
    uint4 tp[8];
    uint4 lz;
};

// Planes of the energy counters: they hold kFoldPairs pairs of items of at most 6 each.  A lane
// of 512 threads has at most 42 items (a slab that fits shared memory has at most 38 K sites,
// 19 K a colour), half of what fits; blocks of fewer threads may have more, which only counts
// (kCountOnly), and folds its counters into the block's sums before they run over.
constexpr int kVBits = 9;
constexpr int kFoldPairs = ((1 << kVBits) - 1) / 12;

// A warp's share of the half sweeps of a launch.
struct Sweeper {
    static constexpr bool kResident = false, kAssisted = false;
    static constexpr int kItems = 1;
    const Geometry& g;
    uint32_t w0, s0;          // addresses of the slab's first word and of its sign byte, less a quarter of w0
    uint32_t queue;           // address of this warp's ties: {word, ties, c0, c1}
    uint32_t planes;          // address of the half sweep's Planes
    const uint32_t* thr;      // ties' threshold rows
    const uint8_t* rung;
    int* E;                   // the block's energy sums (tempering)
    Draws draws;
    uint32_t word, valid, sweep;
    int warp, lane, warps;
    uint32_t below;           // the lanes below this one
    uint32_t V[kVBits];       // energy counters of this lane's items
    int nitems;
    Unit u;                   // the unit at hand; between half sweeps, this warp's first

    __device__ __forceinline__ Sweeper(const Geometry& geo, const uint32_t* words, const uint8_t* signs,
                                       const uint4* queues)
        : g(geo), w0(smem_addr(words)), s0(smem_addr(signs) - w0 / 4u), rung(nullptr), E(nullptr), warp(threadIdx.x >> 5),
          lane(threadIdx.x & 31), warps(blockDim.x >> 5)
    {
        asm("mov.u32 %0, %%lanemask_lt;" : "=r"(below));
        queue = smem_addr(queues) + (uint32_t)(warp * kTieCap) * 16u;
        u.locate(g, w0, warp < g.units ? warp : 0, lane);
    }

    __device__ __forceinline__ void first_draws(uint32_t (&A)[1][8]) const { draws.planes(first_site(0), A[0]); }

    // this warp's first site of a half sweep (between half sweeps)
    __device__ __forceinline__ uint32_t first_site(int colour) const
    {
        return (uint32_t)u.site + ((u.flags ^ (uint32_t)colour) & kOdd);
    }

    // Decides one tie of each of the last up to 32 of the qn queued entries, one a lane; an
    // entry with further ties goes back to the queue, so that later passes run with full warps
    // too.  An accepted flip is xored into the word (its owner has stored it; an entry's bits
    // belong to nobody else) and, in tempering, its energy change added to the replica's sum.
    // A replica's threshold row is thr + 16 rung[b] (annealing: one row for all).
    template <bool TEMPERING, bool ENERGY>
    __device__ __forceinline__ void decide(int& qn)
    {
        const int n = min(qn, 32);
        qn -= n;
        __syncwarp();
        const uint4 t = ld_quad(queue + 16u * (uint32_t)(qn + lane));
        const uint32_t m = lane < n ? t.y : 0u;
        const int b = (31 - __clz((int)m)) & 31;  // the highest tie
        const uint32_t k = 2u + ((t.z >> b) & 1u) * 2u + ((t.w >> b) & 1u) * 4u;
        const uint32_t low = thr[(TEMPERING ? (uint32_t)rung[b] * kThrRow : 0u) + k] & 0xFFFFFFu;
        // the logical site of the word: its row in storage order, its place in it
        const uint32_t at = (t.x - w0) / 4u, row = __umulhi(at, g.Lmagic), pos = at - row * (uint32_t)g.L;
        const uint32_t odd = pos >= (uint32_t)g.H;
        const uint32_t site = (uint32_t)(g.z0 * g.LL) + row * (uint32_t)g.L + 2u * (pos - (odd ? (uint32_t)g.H : 0u)) + odd;
        const uint32_t slot = 32u * word + (uint32_t)b;
        const Philox4 d = philox4x32_10(site, sweep, slot >> 2, kDomainTail, draws.k0, draws.k1);
        const uint32_t v = (slot & 2u) ? ((slot & 1u) ? d.v[3] : d.v[2]) : ((slot & 1u) ? d.v[1] : d.v[0]);
        if (m && (v >> 8) < low) {
            xor_word(t.x, 1u << b);
            if (ENERGY) atomicAdd(&E[b], (int)(2u * k));
        }
        const uint32_t rest = m & ~(1u << b);
        const unsigned who = __ballot_sync(kAll, rest != 0u);  // (every lane has read its entry)
        st_quad_if(rest, queue + 16u * (uint32_t)(qn + __popc(who & below)), t.x, rest, t.z, t.w);
        qn += __popc(who);
        __syncwarp();
    }

    // Where a half sweep stands in the unit at hand.  What alternates with the item's parity is
    // kept for both: index P is the step's, the other one the next step's.
    struct Cursor {
        int q, k;                      // unit, planes left
        uint32_t is;                   // the item's word
        int site;
        int far[2], d[2], ds[2];       // to its far x neighbour; to the next item's word and site
        uint32_t zm, near;             // words below and beside it
        uint32_t alive;
        int qn;                        // queued ties (uniform)
        uint32_t c0, c1, c2;           // energies: counts of the item before (weight 1, 2, 4)
    };

    template <int P>
    __device__ __forceinline__ void enter(Cursor& c, int colour, int H4, int LL4) const
    {
        const bool odd = ((u.flags ^ (uint32_t)colour) & kOdd) != 0u;
        c.k = u.n;
        c.alive = (u.flags & kLive) ? valid : 0u;
        c.is = u.base + (odd ? H4 : 0);
        c.site = u.site + (odd ? 1 : 0);
        c.far[P] = odd ? u.fsum - u.f0 : u.f0;
        c.far[P ^ 1] = u.fsum - c.far[P];
        c.d[P] = odd ? LL4 - H4 : LL4 + H4;
        c.d[P ^ 1] = 2 * LL4 - c.d[P];
        c.ds[P] = LL4 / 4 + (odd ? -1 : 1);
        c.ds[P ^ 1] = LL4 / 2 - c.ds[P];
        c.zm = ld_word(c.is - LL4);
        c.near = ld_word(c.is + (odd ? -H4 : H4));
    }

    // One item: A holds its draws and B receives those of the item after it (of the next unit,
    // or of this warp's first of the next half sweep), whose multiplies run beside this item's
    // logic.  P: even or odd step.  False after the warp's last item.
    template <int MODE, bool TEMPERING, bool ENERGY, int P>
    __device__ __forceinline__ bool step(Cursor& c, const int colour, const int H4, const int LL4,
                                         const uint32_t (&A)[8], uint32_t (&B)[8])
    {
        const uint32_t is = c.is;
        const uint32_t self = ld_word(is), xf = ld_word(is + c.far[P]), yp = ld_word(is + u.yp), ym = ld_word(is + u.ym);
        const uint32_t zp = ld_word(is + LL4);
        const uint32_t sb = ld_byte(s0 + is / 4u);
        const uint32_t near = c.near, zm = c.zm, alive = c.alive;
        bool more = true;
        if (c.k > 1) {
            --c.k;
            c.zm = near;
            c.near = zp;
            c.is += c.d[P];
            c.site += c.ds[P];
        } else {
            c.q += warps;
            more = c.q < g.units;
            if (more || c.q != warp + warps) u.locate(g, w0, more ? c.q : warp, lane);
            if (more) {
                enter<P ^ 1>(c, colour, H4, LL4);
            } else {
                c.site = (int)first_site(colour ^ 1);
                if (colour == 1) draws.set_sweep(sweep + 1u, word);
            }
        }
        constexpr bool kDraws = MODE == kCompare || MODE == kTailOnly;
        if (kDraws) draws.planes((uint32_t)c.site, B);
        // masks of negative couplings: six sign bits spread to the tops of bytes
        const uint32_t m1 = sb * 0x10204080u, m2 = sb * 0x408u;
        const uint32_t a0 = logic<kXor3>(self, near, sign_bytes(m1, 0x8888u));
        const uint32_t a1 = logic<kXor3>(self, xf, sign_bytes(m1, 0x9999u));
        const uint32_t a2 = logic<kXor3>(self, yp, sign_bytes(m1, 0xAAAAu));
        const uint32_t a3 = logic<kXor3>(self, ym, sign_bytes(m1, 0xBBBBu));
        const uint32_t a4 = logic<kXor3>(self, zp, sign_bytes(m2, 0x8888u));
        const uint32_t a5 = logic<kXor3>(self, zm, sign_bytes(m2, 0x9999u));
        const uint32_t s1 = logic<kXor3>(a0, a1, a2), k1 = logic<kMaj>(a0, a1, a2);
        const uint32_t s2 = logic<kXor3>(a3, a4, a5), k2 = logic<kMaj>(a3, a4, a5);
        const uint32_t t = s1 & s2;
        uint32_t c0 = s1 ^ s2, c1 = logic<kXor3>(k1, k2, t), c2 = logic<kMaj>(k1, k2, t);
        uint32_t lt = 0, tie = 0;
        if (MODE == kCompare) {
            uint32_t eq = alive & c2;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint4 p = ld_quad(planes + 16u * j);
                const uint32_t T = logic<kSelect>(c1, p.z, logic<kSelect>(c0, p.y, p.x));
                lt = j == 0 ? T & ~A[0] : logic<kBorrow>(A[j], T, lt);
                eq = logic<kAndEqual>(eq, A[j], T);
            }
            tie = eq;
        } else if (MODE == kTailOnly) {
            const uint32_t any = (A[0] | A[1] | A[2]) | (A[3] | A[4] | A[5]) | (A[6] | A[7]);
            tie = alive & c2 & ~any;
        }
        const uint32_t flip = MODE == kCountOnly ? 0u : (~c2 | lt) & alive;
        if (MODE != kCountOnly) st_word_if(alive, is, self ^ flip);
        if (kDraws) {
            const uint4 lz = ld_quad(planes + 128u);
            tie &= logic<kSelect>(c1, lz.z, logic<kSelect>(c0, lz.y, lz.x));
            const unsigned who = __ballot_sync(kAll, tie != 0u);
            st_quad_if(tie, queue + 16u * (uint32_t)(c.qn + __popc(who & below)), is, tie, c0, c1);
            c.qn += __popc(who);
            while (c.qn >= 32) decide<TEMPERING, ENERGY>(c.qn);
        }
        if (ENERGY) {
            mp::count_after_flip(flip, c0, c1, c2);
            if (!alive) c0 = c1 = c2 = 0u;  // a lane beyond the columns counts nothing
            nitems += alive != 0u;
            if (P == 0) {  // two items are added together
                c.c0 = c0, c.c1 = c1, c.c2 = c2;
            } else {
                add_two(c.c0, c.c1, c.c2, c0, c1, c2);
            }
        }
        return more;
    }

    // Two items' counts into the vertical counters.
    __device__ __forceinline__ void add_two(uint32_t a0, uint32_t a1, uint32_t a2, uint32_t b0, uint32_t b1, uint32_t b2)
    {
        const uint32_t k = logic<kMaj>(V[0], a0, b0);  // weight 2 from weight 1
        V[0] = logic<kXor3>(V[0], a0, b0);
        const uint32_t m = logic<kMaj>(V[1], a1, b1), v1 = logic<kXor3>(V[1], a1, b1);
        V[1] = v1 ^ k;
        const uint32_t n = v1 & k;  // m, n: weight 4
        const uint32_t o = logic<kMaj>(V[2], a2, b2), v2 = logic<kXor3>(V[2], a2, b2);
        const uint32_t r = logic<kMaj>(v2, m, n);  // o, r: weight 8
        V[2] = logic<kXor3>(v2, m, n);
        uint32_t carry = logic<kMaj>(V[3], o, r);
        V[3] = logic<kXor3>(V[3], o, r);
#pragma unroll
        for (int j = 4; j < kVBits; ++j) {
            const uint32_t t = V[j] & carry;
            V[j] ^= carry;
            carry = t;
        }
    }

    __device__ __forceinline__ void clear_counters()
    {
#pragma unroll
        for (int j = 0; j < kVBits; ++j) V[j] = 0;
        nitems = 0;
    }

    // This warp's columns of a half sweep.  A: the draws of its first item, on return those of
    // its first item of the next half sweep.
    template <int MODE, bool TEMPERING, bool ENERGY>
    __device__ __forceinline__ void half(const int colour, uint32_t (&A)[8])
    {
        if (ENERGY) clear_counters();
        if (warp < g.units) {
            const int H4 = 4 * g.H, LL4 = 4 * g.LL;
            Cursor c;
            c.q = warp;
            c.qn = 0;
            enter<0>(c, colour, H4, LL4);
            uint32_t B[8];
            for (int pairs = 1;; ++pairs) {
                if (!step<MODE, TEMPERING, ENERGY, 0>(c, colour, H4, LL4, A, B)) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) A[j] = B[j];
                    if (ENERGY) add_two(c.c0, c.c1, c.c2, 0u, 0u, 0u);
                    break;
                }
                if (!step<MODE, TEMPERING, ENERGY, 1>(c, colour, H4, LL4, B, A)) break;
                if (MODE == kCountOnly && pairs == kFoldPairs) {  // (a warp's lanes are at the same item)
                    energy_to_block();
                    clear_counters();
                    pairs = 0;
                }
            }
            while ((MODE == kCompare || MODE == kTailOnly) && c.qn) decide<TEMPERING, ENERGY>(c.qn);
        }
        __syncwarp();
    }

    // Copies this warp's updated face words to the halo planes of the blocks above and below
    // (up, dn: what to add to an address for the word of the same place there; their barriers),
    // or to its own when the block is alone in its cluster.
    __device__ __forceinline__ void push_faces(const int colour, bool alone, uint32_t up, uint32_t dn, uint32_t up_bar,
                                               uint32_t dn_bar)
    {
        const uint32_t LL4 = 4u * (uint32_t)g.LL, H4 = 4u * (uint32_t)g.H, slab = (uint32_t)g.zc * LL4,
                       slab_dn = (uint32_t)g.zdn * LL4;
        Unit v = u;
        for (int q = warp; q < g.units;) {
            const uint32_t odd = v.flags ^ (uint32_t)colour;
            if ((v.flags & (kBottom | kLive)) == (kBottom | kLive)) {  // to the upper halo of the block below
                const uint32_t is = v.base + ((odd & kOdd) ? H4 : 0u);
                if (alone) st_word_if(1u, is + slab, ld_word(is));
                else push_word(dn + is + slab_dn, ld_word(is), dn_bar);
            }
            if ((v.flags & (kTop | kLive)) == (kTop | kLive)) {  // to the lower halo of the block above
                const uint32_t is = v.base + (uint32_t)(v.n - 1) * LL4 + (((odd ^ (uint32_t)(v.n - 1)) & kOdd) ? H4 : 0u);
                if (alone) st_word_if(1u, is - slab, ld_word(is));
                else push_word(up + is - slab, ld_word(is), up_bar);
            }
            q += warps;
            if (q < g.units) v.locate(g, w0, q, lane);
        }
    }

    // End of a colour-1 half sweep: lane b collects replica b of every lane's counters (a bit
    // transpose a plane, only the planes that can be nonzero) and adds them to the block's sum.
    __device__ __forceinline__ void energy_to_block()
    {
        const int most = __reduce_max_sync(kAll, nitems), items = __reduce_add_sync(kAll, nitems);
        int cnt = 0;
#pragma unroll
        for (int jb = 0; jb < kVBits; ++jb)
            if (jb < 3 || 6 * most >= (1 << jb)) cnt += __popc(mp::warp_transpose(V[jb], lane)) << jb;
        const int e = 6 * items - 2 * cnt;
        if (e) atomicAdd(&E[lane], e);
    }
};


// The same for blocks with at most R x pairs of sites a thread (R = 1 or 2; two sites a pair,
// one of each colour, the lane's for the whole launch).  What a half sweep costs such a block
// is a chain of latencies, so everything of the lane's sites stays in registers: their words
// (only this lane changes them), their couplings, their addresses.  A half sweep loads five
// words a site; its ties are decided on the spot -- the tail draw of every lane's first tie
// runs beside the draws of the next half sweep -- and its face words go to the neighbours
// straight from registers.
//
// ASSISTED (R = 1): a second set of warps makes the draws, a half sweep ahead, and hands them over
// through shared memory (where the queues would be), two buffers by colour; the block barrier
// that ends a half sweep orders both sides.  For blocks of so few pairs that each partition of
// the SM has one warp to run: L = 4 with 8 replicas takes 0.41 us a half sweep (0.53 with the
// draws in line), tempering 20 lattices of L = 4 1.6 us a sweep (1.9), of L = 8 2.06 (2.15).
// (Leaving out the tail draws where no lane has a tie: 0.38 with 8 replicas, but 0.55 instead of
// 0.52 with 20 at L = 8; not kept.)
template <int R, bool ASSISTED = false>
struct Resident {
    static constexpr bool kResident = true, kAssisted = ASSISTED;
    static constexpr int kItems = R;
    const Geometry& g;
    uint32_t w0;
    uint32_t planes;          // address of the half sweep's Planes
    const uint32_t* thr;      // ties' threshold rows
    const uint8_t* rung;
    int* E;                   // the block's energy sums (tempering)
    Draws draws;
    uint32_t word, valid, sweep;
    int warp, lane;
    int LL4;
    uint32_t slab, slab_dn;   // bytes of the slab, and of the one below
    bool idle;                // a warp beyond the pairs (uniform)
    bool drawer;              // of the second set of warps (uniform)
    uint32_t mail, mail_step; // the lane's draws: address of four planes of colour 0, bytes to the next four
    struct Pair {
        // of its site of colour 0 and of colour 1
        uint32_t at[2], value[2], mask[2][R == 1 ? 6 : 1];  // (R = 2: masks are spread from the sign bits)
        int site[2], far[2];
        int yp, ym;
        uint32_t flags;       // Unit's kLive, kBottom, kTop
        uint32_t c0, c1, c2;  // counts after a colour-1 half sweep (energies)
    } pair[R];

    __device__ __forceinline__ Resident(const Geometry& geo, const uint32_t* words, const uint8_t* signs,
                                        const uint4* letters)
        : g(geo), w0(smem_addr(words)), rung(nullptr), E(nullptr), warp(threadIdx.x >> 5), lane(threadIdx.x & 31)
    {
        const int L = g.L, H = g.H, LL = g.LL;
        LL4 = 4 * LL;
        slab = (uint32_t)(g.zc * LL4);
        slab_dn = (uint32_t)(g.zdn * LL4);
        const int set = ASSISTED ? (int)blockDim.x / 64 * 32 : (int)blockDim.x;  // threads with pairs
        const bool second = ASSISTED && (int)threadIdx.x >= set;
        drawer = second && (int)threadIdx.x < 2 * set;
        idle = second || warp * 32 >= g.zc * g.cols;
        mail_step = 16u * (uint32_t)set;
        mail = smem_addr(letters) + 16u * (uint32_t)((int)threadIdx.x - (second ? set : 0));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            Pair& q = pair[r];
            const int n = (int)threadIdx.x + r * (int)blockDim.x - (second ? set : 0);
            const bool live = n < g.zc * g.cols;
            const int p = live ? n : 0;
            const int row = H == 1 ? p : (int)__umulhi((uint32_t)p, g.Hmagic), j = p - row * H;
            const int zl = (int)__umulhi((uint32_t)row, g.Lmagic), y = row - zl * L;
            q.yp = 4 * (y + 1 == L ? L - LL : L);
            q.ym = 4 * (y == 0 ? LL - L : -L);
            q.flags = live && !second ? kLive | (zl == 0 ? kBottom : 0u) | (zl + 1 == g.zc ? kTop : 0u) : 0u;
            q.c0 = q.c1 = q.c2 = 0u;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int odd = (y + g.z0 + zl + c) & 1;
                const int pos = row * L + odd * H + j;
                q.at[c] = w0 + 4u * (uint32_t)pos;
                q.site[c] = (g.z0 * L + row) * L + 2 * j + odd;
                q.far[c] = 4 * (odd ? -H + (j + 1 == H ? 1 - H : 1) : H + (j == 0 ? H - 1 : -1));
                const uint32_t sb = signs[pos];
                if constexpr (R == 1) {
#pragma unroll
                    for (int k = 0; k < 6; ++k) q.mask[c][k] = 0u - ((sb >> k) & 1u);
                } else {
                    q.mask[c][0] = sb;
                }
                q.value[c] = words[pos];
            }
        }
    }

    __device__ __forceinline__ void first_draws(uint32_t (&A)[R][8]) const
    {
#pragma unroll
        for (int r = 0; r < R; ++r) draws.planes((uint32_t)pair[r].site[0], A[r]);
    }

    // (ASSISTED, second set) Hands over the draws of the lane's site of colour C.
    template <int C>
    __device__ __forceinline__ void hand_over() const
    {
        uint32_t A[8];
        draws.planes((uint32_t)pair[0].site[C], A);
        const uint32_t to = mail + (C ? 2u * mail_step : 0u);
        st_quad_if(1u, to, A[0], A[1], A[2], A[3]);
        st_quad_if(1u, to + mail_step, A[4], A[5], A[6], A[7]);
    }

    // A: the draws of the lane's sites of colour C; on return, when `next`, those of its other
    // sites in the half sweep that follows.  (ASSISTED: they come from the second set.)
    template <int C, int MODE, bool TEMPERING, bool ENERGY>
    __device__ __forceinline__ void half(uint32_t (&A)[R][8], bool next)
    {
        if (idle) return;
        if constexpr (ASSISTED && (MODE == kCompare || MODE == kTailOnly)) {
            const uint32_t from = mail + (C ? 2u * mail_step : 0u);
            const uint4 lo = ld_quad(from), hi = ld_quad(from + mail_step);
            A[0][0] = lo.x, A[0][1] = lo.y, A[0][2] = lo.z, A[0][3] = lo.w;
            A[0][4] = hi.x, A[0][5] = hi.y, A[0][6] = hi.z, A[0][7] = hi.w;
        }
        uint32_t flip[R], tie[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            Pair& q = pair[r];
            const uint32_t is = q.at[C], self = q.value[C];
            const uint32_t xf = ld_word(is + q.far[C]), n2 = ld_word(is + q.yp), n3 = ld_word(is + q.ym),
                           n4 = ld_word(is + LL4), n5 = ld_word(is - LL4);
            const uint32_t alive = (q.flags & kLive) ? valid : 0u;
            uint32_t S[6];
            if constexpr (R == 1) {
#pragma unroll
                for (int k = 0; k < 6; ++k) S[k] = q.mask[C][k];
            } else {
                const uint32_t m1 = q.mask[C][0] * 0x10204080u, m2 = q.mask[C][0] * 0x408u;
                S[0] = sign_bytes(m1, 0x8888u), S[1] = sign_bytes(m1, 0x9999u), S[2] = sign_bytes(m1, 0xAAAAu);
                S[3] = sign_bytes(m1, 0xBBBBu), S[4] = sign_bytes(m2, 0x8888u), S[5] = sign_bytes(m2, 0x9999u);
            }
            const uint32_t a0 = logic<kXor3>(self, q.value[C ^ 1], S[0]), a1 = logic<kXor3>(self, xf, S[1]);
            const uint32_t a2 = logic<kXor3>(self, n2, S[2]), a3 = logic<kXor3>(self, n3, S[3]);
            const uint32_t a4 = logic<kXor3>(self, n4, S[4]), a5 = logic<kXor3>(self, n5, S[5]);
            const uint32_t s1 = logic<kXor3>(a0, a1, a2), k1 = logic<kMaj>(a0, a1, a2);
            const uint32_t s2 = logic<kXor3>(a3, a4, a5), k2 = logic<kMaj>(a3, a4, a5);
            const uint32_t t = s1 & s2;
            const uint32_t c0 = s1 ^ s2, c1 = logic<kXor3>(k1, k2, t), c2 = logic<kMaj>(k1, k2, t);
            q.c0 = c0, q.c1 = c1, q.c2 = c2;
            uint32_t lt = 0;
            tie[r] = 0;
            if (MODE == kCompare) {
                uint32_t eq = alive & c2;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint4 p = ld_quad(planes + 16u * j);
                    const uint32_t T = logic<kSelect>(c1, p.z, logic<kSelect>(c0, p.y, p.x));
                    lt = j == 0 ? T & ~A[r][0] : logic<kBorrow>(A[r][j], T, lt);
                    eq = logic<kAndEqual>(eq, A[r][j], T);
                }
                tie[r] = eq;
            } else if (MODE == kTailOnly) {
                const uint32_t any = (A[r][0] | A[r][1] | A[r][2]) | (A[r][3] | A[r][4] | A[r][5]) | (A[r][6] | A[r][7]);
                tie[r] = alive & c2 & ~any;
            }
            flip[r] = MODE == kCountOnly ? 0u : (~c2 | lt) & alive;
        }
        if (C == 1 && !ASSISTED) draws.set_sweep(sweep + 1u, word);
        if (MODE == kCompare || MODE == kTailOnly) {
            const uint4 lz = ld_quad(planes + 128u);
            uint32_t low[R], tail[R], bit[R], more = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) {  // the first tie of each site, beside the next draws
                Pair& q = pair[r];
                tie[r] &= logic<kSelect>(q.c1, lz.z, logic<kSelect>(q.c0, lz.y, lz.x));
                const int b = (31 - __clz((int)tie[r])) & 31;
                bit[r] = 1u << b;
                low[r] = low_of<TEMPERING>(q, b);
                tail[r] = tail_of(q.site[C], b);
                if (!ASSISTED) draws.planes((uint32_t)q.site[C ^ 1], A[r]);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (tie[r] && tail[r] < low[r]) flip[r] |= bit[r];
                tie[r] &= ~bit[r];
                more |= tie[r];
            }
            while (__any_sync(kAll, more != 0u)) {  // further ties
                more = 0;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int b = (31 - __clz((int)tie[r])) & 31;
                    if (tie[r] && tail_of(pair[r].site[C], b) < low_of<TEMPERING>(pair[r], b)) flip[r] |= 1u << b;
                    tie[r] &= ~(1u << b);
                    more |= tie[r];
                }
            }
        } else if (next && !ASSISTED) {
#pragma unroll
            for (int r = 0; r < R; ++r) draws.planes((uint32_t)pair[r].site[C ^ 1], A[r]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            Pair& q = pair[r];
            q.value[C] ^= flip[r];
            st_word_if(q.flags & kLive, q.at[C], q.value[C]);
            if (ENERGY) mp::count_after_flip(flip[r], q.c0, q.c1, q.c2);
        }
    }

    template <bool TEMPERING>
    __device__ __forceinline__ uint32_t low_of(const Pair& q, int b) const
    {
        const uint32_t k = 2u + ((q.c0 >> b) & 1u) * 2u + ((q.c1 >> b) & 1u) * 4u;
        return thr[(TEMPERING ? (uint32_t)rung[b] * kThrRow : 0u) + k] & 0xFFFFFFu;
    }
    __device__ __forceinline__ uint32_t tail_of(int site, int b) const
    {
        const uint32_t slot = 32u * word + (uint32_t)b;
        const Philox4 d = philox4x32_10((uint32_t)site, sweep, slot >> 2, kDomainTail, draws.k0, draws.k1);
        return ((slot & 2u) ? ((slot & 1u) ? d.v[3] : d.v[2]) : ((slot & 1u) ? d.v[1] : d.v[0])) >> 8;
    }

    template <int C>
    __device__ __forceinline__ void push_faces(bool alone, uint32_t up, uint32_t dn, uint32_t up_bar, uint32_t dn_bar) const
    {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const Pair& q = pair[r];
            if (q.flags & kBottom) {
                if (alone) st_word_if(1u, q.at[C] + slab, q.value[C]);
                else push_word(dn + q.at[C] + slab_dn, q.value[C], dn_bar);
            }
            if (q.flags & kTop) {
                if (alone) st_word_if(1u, q.at[C] - slab, q.value[C]);
                else push_word(up + q.at[C] - slab, q.value[C], up_bar);
            }
        }
    }

    __device__ __forceinline__ void energy_to_block() const
    {
        int items = 0, cnt = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t on = (pair[r].flags & kLive) ? ~0u : 0u;
            items += __popc(__ballot_sync(kAll, on != 0u));
            cnt += __popc(mp::warp_transpose(pair[r].c0 & on, lane)) + 2 * __popc(mp::warp_transpose(pair[r].c1 & on, lane)) +
                   4 * __popc(mp::warp_transpose(pair[r].c2 & on, lane));
        }
        const int e = 6 * items - 2 * cnt;
        if (e) atomicAdd(&E[lane], e);
    }
};

// The form a block of `pairs` x pairs takes with at most `threads` threads: pairs a thread (0:
// the Sweeper), and its threads.
__host__ __device__ inline int resident_items(int64_t pairs, int threads)
{
    return pairs <= threads ? 1 : pairs <= 2 * threads ? 2 : 0;
}
// ASSISTED up to so many pairs a block.
constexpr int kAssistedPairs = 128;
inline bool assisted(int64_t pairs, int threads) { return pairs <= (threads < kAssistedPairs ? threads : kAssistedPairs); }
inline int resident_threads(int64_t pairs, int threads)
{
    const int r = resident_items(pairs, threads);
    return r == 0 ? threads : (int)((pairs + 32 * r - 1) / (32 * r)) * 32;
}
__host__ __device__ inline int64_t pairs_of(int L, int C) { return (int64_t)Geometry::planes(L, C) * L * (L / 2); }

}  // namespace slab
}  // namespace sg
