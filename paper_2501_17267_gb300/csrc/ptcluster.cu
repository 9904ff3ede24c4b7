// ptcluster.cu -- parallel tempering (App. D.2) with every sweep of a chunk in one
// launch: one thread-block cluster per instance, its lattice resident in the blocks'
// shared memory for the whole chunk.
//
// Cluster `inst` of C blocks splits the L^3 lattice of its instance into C z-slabs of
// about L / C planes, one 32-bit word of 32 slots per site (slab.cuh: the updates, and how the
// blocks exchange their faces); the spins are written back at the end.
//
// Energies and the exchange.  Each bond joins a colour-0 and a colour-1 site, so the
// colour-1 half sweep sums every slot's energy afresh (6 - 2c per site for unit
// couplings, c the satisfied count after the update), in bit-sliced counters per
// thread reduced through a warp bit transpose.  Every block pushes its 32 sums to every
// block of the cluster (st.async, two buffers by sweep parity, each with its own
// barrier), and every warp of every block decides the exchange itself -- the same integer
// decisions from the same draws -- so that it can make its share of the next sweep's
// threshold planes at once; one block barrier then starts the next sweep.  The exchange
// thresholds are kept in shared memory where they fit, since a lookup of them lies on the
// path of every sweep.
//
// 33 to 64 temperatures are two words a site, each on C blocks of the cluster (4 lattices of
// L = 32, 48 temperatures: 10.3 us a sweep, 15.6 through the row kernels).
//
// Every attempt draws the same counters as the row kernel (site, sweep, word) and the
// exchange the same counters as the stand-alone exchange (pair, sweep), so results are
// bit-identical to the row kernel and to the oracle.
#include <cooperative_groups.h>
#include <stdint.h>
#include <stdlib.h>

#include <algorithm>
#include <atomic>

#include "slab.cuh"
#include "sg_internal.h"

namespace cg = cooperative_groups;

namespace sg {
namespace {

constexpr int kThreads = slab::kMaxThreads;

struct PtcArgs {
    uint32_t* spins;                // [I][N][words] (32 slots of a site a word), storage order
    const uint8_t* const* j1_ptrs;  // per instance: [N] coupling sign bits (all |J| = 1)
    const RunKeys* keys;            // [I]
    const uint32_t* thr;            // [K][kThrRow] thresholds by rung
    uint8_t* rung_of_slot;          // [I][32 words]
    uint8_t* slot_of_rung;          // [I][K]
    int32_t* E;                     // [I][32 words] out: slot energies after the last sweep
    unsigned long long* accepts;    // [I][K-1]
    int32_t* minE;                  // [I]
    const uint32_t* xtab;           // exchange thresholds (exchange.cuh)
    const uint32_t* xoff;
    const uint32_t* xlen;
    const uint32_t* xtail;
    int* status;                    // SG_ETIMEOUT when a bounded wait gave up
    int L, K, C, s_begin, s_end;
    ChunkReport report;             // of a run of one instance
    long long wait_limit;           // cycles a wait for other blocks lasts at most
    uint32_t Hmagic;                // ceil(2^32 / (L / 2))
    int xwords;                     // words of xtab held in shared memory (0: read from global memory)
};

// Shared state of a block, WN words an instance.
template <int WN>
struct PtShared {
    slab::Planes planes;
    slab::Geometry geo;
    uint32_t rthr[32 * WN * kThrRow];  // per rung: its threshold row
    int E[32];                    // the block's energy sums of a colour-1 half sweep
    int Epart[2][slab::kMaxC][32];  // by sweep parity: every block's sums
    uint8_t rung[32];             // slot of the block's word -> rung
    uint8_t inverse[kThreads / 32][32 * WN];  // a warp's scratch: slot -> rung
    uint32_t xoff[32 * WN], xlen[32 * WN], xtail[32 * WN];
    uint64_t bar[2];              // by colour: the neighbours' face words have arrived
    uint64_t ebar[2];             // by sweep parity: every block's energy sums have arrived
    int fail[2];                  // a wait gave up: before the exchange, after it (read after the next block barrier)
};

// S: slab::Sweeper, or slab::Resident when a block has a thread for each of its x pairs.  WN: words
// an instance (K <= 32 WN); a cluster has C blocks for each, which share nothing but the energies.
template <class S, int WN>
__global__ void __launch_bounds__(S::kAssisted ? 2 * slab::kAssistedPairs : kThreads, 1) pt_cluster_kernel(const PtcArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ PtShared<WN> sh;

    cg::cluster_group cluster = cg::this_cluster();
    const int C = a.C, blocks = WN * C;  // of a word, of the cluster
    const int rank = blocks > 1 ? (int)cluster.block_rank() : 0;
    const int word = WN == 1 ? 0 : rank / C, r = rank - word * C;
    const int inst = blockIdx.x / blocks;
    const int K = a.K;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, threads = blockDim.x, warps = threads >> 5;
    const RunKeys key = a.keys[inst];
    const slab::Geometry& geo = sh.geo;
    if (tid == 0) sh.geo.init(a.L, C, r, warps, a.Hmagic);
    __syncthreads();
    uint32_t* w = reinterpret_cast<uint32_t*>(smem) + geo.LL;
    uint8_t* sgn = smem + slab::Geometry::words(a.L, C) * 4;
    uint32_t* g = a.spins + (size_t)inst * geo.LL * a.L * WN + word;
    slab::load_slab(geo, g, WN, a.j1_ptrs[inst], w, sgn);
    uint32_t* xtab_s = reinterpret_cast<uint32_t*>(smem + slab::smem_bytes(a.L, C, threads));
    for (int q = tid; q < a.xwords; q += threads) xtab_s[q] = a.xtab[q];
    const uint32_t* xtab = a.xwords ? xtab_s : a.xtab;

    // slot maps and thresholds; a lane is slots or rungs 32 i + lane.  slot[i]: the rung's slot, in
    // every warp's own registers; rung: of slot `lane` of the block's word.
    int slot[WN];
#pragma unroll
    for (int i = 0; i < WN; ++i) slot[i] = 32 * i + lane < K ? a.slot_of_rung[(size_t)inst * K + 32 * i + lane] : 32 * i + lane;
    int rung = a.rung_of_slot[((size_t)inst * WN + word) * 32 + lane];
    for (int q = tid; q < K * kThrRow; q += threads) sh.rthr[q] = a.thr[q];
    if (tid < 32) {
        sh.rung[tid] = (uint8_t)rung;
        sh.E[tid] = 0;
        for (int k = tid; k + 1 < K; k += 32) {
            sh.xoff[k] = a.xoff[k];
            sh.xlen[k] = a.xlen[k];
            sh.xtail[k] = a.xtail[k];
        }
    }
    if (tid == 0) {
        slab::mbar_init(&sh.bar[0]);
        slab::mbar_init(&sh.bar[1]);
        slab::mbar_init(&sh.ebar[0]);
        slab::mbar_init(&sh.ebar[1]);
        slab::mbar_init_fence();
        sh.fail[0] = sh.fail[1] = blocks > 1 && a.wait_limit == 0;
    }
    int minE = a.minE[inst];
    uint32_t accepted[WN] = {};  // first warp, by the pair's lower rung
    __syncthreads();
    // this warp's share of the threshold planes: planes of the slots' leading bytes, then lz
    auto build_planes = [&]() {
        const uint32_t* row = sh.rthr + rung * kThrRow;
        const uint32_t t2 = row[2], t4 = row[4], t6 = row[6];
        for (int j = warp; j < 9; j += warps) {
            const uint32_t mask = j < 8 ? 1u << (24 + j) : 0xFFFFFFu;
            const uint32_t p2 = __ballot_sync(slab::kAll, (t2 & mask) != 0u), p4 = __ballot_sync(slab::kAll, (t4 & mask) != 0u),
                           p6 = __ballot_sync(slab::kAll, (t6 & mask) != 0u);
            if (lane == 0) *(j < 8 ? &sh.planes.tp[j] : &sh.planes.lz) = make_uint4(p2, p4, p6, 0u);
        }
    };
    build_planes();

    __syncthreads();  // the slab is in place
    S s(geo, w, sgn, reinterpret_cast<const uint4*>(smem + slab::smem_queue_offset(a.L, C)));
    s.planes = slab::smem_addr(&sh.planes);
    s.thr = sh.rthr;
    s.rung = sh.rung;
    s.E = sh.E;
    s.draws.k0 = key.k0;
    s.draws.k1 = key.k1;
    s.word = (uint32_t)word;
    s.valid = slab::word_valid_bits(K, word);
    const uint32_t first = (uint32_t)(word * C);
    const uint32_t up = first + (uint32_t)(r + 1 == C ? 0 : r + 1), dn = first + (uint32_t)(r == 0 ? C - 1 : r - 1);
    uint32_t up_w = 0, dn_w = 0, up_bar = 0, dn_bar = 0;
    if (C > 1) {
        up_w = slab::cluster_addr(s.w0, up) - s.w0;
        dn_w = slab::cluster_addr(s.w0, dn) - s.w0;
        up_bar = slab::cluster_addr(slab::smem_addr(&sh.bar[0]), up);
        dn_bar = slab::cluster_addr(slab::smem_addr(&sh.bar[0]), dn);
    }
    // every block has loaded its halos and set up its barriers before another pushes
    if (blocks > 1) cluster.sync();
    else __syncthreads();

    const uint32_t s_end = (uint32_t)a.s_end;
    uint32_t sweep = (uint32_t)a.s_begin;
    uint32_t phase = 0;  // of bar[0], bar[1]; of ebar: bits 2, 3
    bool ok = true;
    uint32_t A[S::kItems][8];
    s.draws.set_sweep(sweep, s.word);
    if constexpr (S::kAssisted) {
        if (s.drawer) s.template hand_over<0>();
        __syncthreads();
    } else {
        s.first_draws(A);
    }
    for (; sweep < s_end; ++sweep) {
        s.sweep = sweep;
        // colour 0
        if (C > 1 && tid == 0) slab::mbar_expect(&sh.bar[0], (uint32_t)geo.LL * 4u);
        if constexpr (S::kResident) {
            if (S::kAssisted && s.drawer) {
                s.template hand_over<1>();
            } else {
                s.template half<0, slab::kCompare, true, false>(A, true);
                s.template push_faces<0>(C == 1, up_w, dn_w, up_bar, dn_bar);
            }
        } else {
            s.template half<slab::kCompare, true, false>(0, A[0]);
            s.push_faces(0, C == 1, up_w, dn_w, up_bar, dn_bar);
        }
        __syncthreads();
        // Flags are set before a block barrier and read after it, the same for every thread.  A
        // block that lost a wait leaves at the end of the sweep, when nothing is on its way to it.
        bool lost = false;
        if (blocks > 1) lost = sh.fail[1] != 0;
        if (C > 1) {
            if (!slab::mbar_wait<S::kResident>(&sh.bar[0], phase & 1u, a.wait_limit)) sh.fail[0] = 1;
            phase ^= 1u;
        }
        // colour 1, with the energies
        const uint32_t par = sweep & 1u;
        if (blocks > 1 && tid == 0) {
            if (C > 1) slab::mbar_expect(&sh.bar[1], (uint32_t)geo.LL * 4u);
            slab::mbar_expect(&sh.ebar[par], (uint32_t)blocks * 128u);
        }
        if constexpr (S::kResident) {
            if (S::kAssisted && s.drawer) {
                s.draws.set_sweep(sweep + 1u, s.word);
                s.template hand_over<0>();
            } else {
                s.template half<1, slab::kCompare, true, true>(A, true);
                s.template push_faces<1>(C == 1, up_w, dn_w, up_bar + 8u, dn_bar + 8u);
                s.energy_to_block();
            }
        } else {
            s.template half<slab::kCompare, true, true>(1, A[0]);
            s.push_faces(1, C == 1, up_w, dn_w, up_bar + 8u, dn_bar + 8u);
            s.energy_to_block();
        }
        __syncthreads();
        if (blocks > 1) {
            // the block's sums to every block, a warp a block
            for (int q = warp; q < blocks; q += warps) {
                const uint32_t base = slab::cluster_addr(slab::smem_addr(&sh.Epart[par][rank][lane]), (uint32_t)q);
                slab::push_word(base, (uint32_t)sh.E[lane], slab::cluster_addr(slab::smem_addr(&sh.ebar[par]), (uint32_t)q));
            }
        }
        // the exchange (App. D.2): pairs (k, k + 1) with k = sweep mod 2, accepted when
        // d = E_a - E_b <= 0 or the draw u < T_k(d); a lane is a rung of a pair (WN of them)
        int k[WN];
        uint32_t u[WN];
#pragma unroll
        for (int i = 0; i < WN; ++i) {
            k[i] = ((32 * i + lane - (int)par) & ~1) + (int)par;
            u[i] = philox4x32_10((uint32_t)k[i], sweep, 0u, kDomainExchange, key.k0, key.k1).v[0];
        }
        int Eq[WN];  // of slots 32 i + lane
        if (blocks > 1) {
            if (!slab::mbar_wait<S::kResident>(&sh.ebar[par], (phase >> (2 + par)) & 1u, a.wait_limit)) sh.fail[0] = 1;
            phase ^= 4u << par;
#pragma unroll
            for (int i = 0; i < WN; ++i) {
                Eq[i] = 0;
                for (int q = 0; q < C; ++q) Eq[i] += sh.Epart[par][i * C + q][lane];
            }
        } else {
            Eq[0] = sh.E[lane];
        }
        // v[at], at = 32 i + lane of a lane's array
        auto gather = [&](const int (&v)[WN], int at) {
            int x = __shfl_sync(slab::kAll, v[0], at & 31);
#pragma unroll
            for (int i = 1; i < WN; ++i) {
                const int y = __shfl_sync(slab::kAll, v[i], at & 31);
                if (at >> 5 == i) x = y;
            }
            return x;
        };
        int E_rung[WN], slot_now[WN];  // of the slot at this rung
        bool swapped[WN];
#pragma unroll
        for (int i = 0; i < WN; ++i) {
            E_rung[i] = gather(Eq, slot[i]);
            slot_now[i] = slot[i];
        }
#pragma unroll
        for (int i = 0; i < WN; ++i) {
            const int at = 32 * i + lane, other = (at == k[i] ? at + 1 : at - 1) & (32 * WN - 1);
            const bool pair = k[i] >= 0 && k[i] + 1 < K;
            const int E_other = gather(E_rung, other), slot_other = gather(slot_now, other);
            const int d = at == k[i] ? E_rung[i] - E_other : E_other - E_rung[i];
            bool accept = pair && d <= 0;
            if (pair && d > 0) {
                const uint32_t T =
                    (uint32_t)d <= sh.xlen[k[i]] ? xtab[sh.xoff[k[i]] + (uint32_t)(d - 1)] : sh.xtail[k[i]];
                accept = u[i] < T;
            }
            if (accept) slot[i] = slot_other;
            if (at < K) sh.inverse[warp][slot[i]] = (uint8_t)at;
            swapped[i] = accept && at == k[i];
        }
        __syncwarp();
        rung = 32 * word + lane < K ? sh.inverse[warp][32 * word + lane] : 0;
        build_planes();
        if (warp == 0) {
            sh.rung[lane] = (uint8_t)rung;
            int least = 0x7FFFFFFF;
#pragma unroll
            for (int i = 0; i < WN; ++i) {
                accepted[i] += swapped[i];
                if (32 * i + lane < K) least = min(least, Eq[i]);
                if (rank == 0 && sweep + 1 == s_end) a.E[((size_t)inst * WN + i) * 32 + lane] = Eq[i];
            }
            minE = min(minE, __reduce_min_sync(slab::kAll, least));
        }
        __syncthreads();  // the next sweep's planes are complete, and E has been read
        if (warp == 0) sh.E[lane] = 0;
        if (blocks > 1) lost |= sh.fail[0] != 0;
        if (C > 1) {
            if (!slab::mbar_wait<S::kResident>(&sh.bar[1], (phase >> 1) & 1u, a.wait_limit)) sh.fail[1] = 1;
            phase ^= 2u;
        }
        if (lost) {
            ok = false;
            break;
        }
    }
    __syncthreads();
    ok = ok && !sh.fail[0] && !sh.fail[1];
    if (!ok && tid == 0) atomicExch(a.status, SG_ETIMEOUT);

    // ---- write back ----
    if (ok) {
        const int n = geo.zc * geo.LL;
        for (int q = tid; q < n; q += threads) g[((size_t)geo.z0 * geo.LL + q) * WN] = w[q];
        if (r == 0 && warp == 0) a.rung_of_slot[((size_t)inst * WN + word) * 32 + lane] = (uint8_t)rung;
        if (rank == 0 && warp == 0) {
#pragma unroll
            for (int i = 0; i < WN; ++i) {
                const int k = 32 * i + lane;
                if (k < K) a.slot_of_rung[(size_t)inst * K + k] = (uint8_t)slot[i];
                if (k + 1 < K) a.accepts[(size_t)inst * (K - 1) + k] += (unsigned long long)accepted[i];
            }
            if (lane == 0) a.minE[inst] = minE;
        }
    }
    __syncthreads();
    if (blocks > 1) cluster.sync();  // no block leaves while another may still push to it; the status is complete
    if (a.report.out && rank == 0 && tid == 0) a.report.write(minE, *static_cast<volatile int*>(a.status));
}

int block_threads(int L, int C)
{
    const int64_t pairs = slab::pairs_of(L, C);
    return slab::resident_threads(pairs, kThreads) * (slab::assisted(pairs, kThreads) ? 2 : 1);
}
template <int WN>
const void* kernel_of(int L, int C)
{
    if (slab::assisted(slab::pairs_of(L, C), kThreads)) return (const void*)pt_cluster_kernel<slab::Resident<1, true>, WN>;
    switch (slab::resident_items(slab::pairs_of(L, C), kThreads)) {
        case 1: return (const void*)pt_cluster_kernel<slab::Resident<1>, WN>;
        case 2: return (const void*)pt_cluster_kernel<slab::Resident<2>, WN>;
        default: return (const void*)pt_cluster_kernel<slab::Sweeper, WN>;
    }
}
constexpr int kMaxWords = 2;
const void* kernel_of(int L, int C, int words) { return words == 1 ? kernel_of<1>(L, C) : kernel_of<2>(L, C); }
size_t dyn_smem(int L, int C) { return slab::smem_bytes(L, C, block_threads(L, C)); }
// (with the static part, without the exchange thresholds, which take what is left)
size_t all_smem(int L, int C, int words)
{
    return dyn_smem(L, C) + (words == 1 ? sizeof(PtShared<1>) : sizeof(PtShared<2>));
}
// Clusters of side L, C blocks for each of `words` words, that fit the device at once.
int resident(int L, int C, int words)
{
    return resident_clusters(kernel_of(L, C, words), C * words, dyn_smem(L, C), block_threads(L, C));
}
bool runs(int L, int K) { return K >= 1 && K <= 32 * kMaxWords && L >= 2 && !(L & 1); }

}  // namespace

namespace {
// The current device's SM clock in Hz (asking the driver costs about 250 us: it is kept).
double device_hz()
{
    static std::atomic<int> khz_of[64];
    int dev = 0;
    cudaGetDevice(&dev);
    std::atomic<int>* const kept = dev >= 0 && dev < 64 ? &khz_of[dev] : nullptr;
    int khz = kept ? kept->load() : 0;
    if (khz == 0) {
        if (cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev) != cudaSuccess || khz <= 0) {
            cudaGetLastError();
            khz = 2070000;
        }
        if (kept) kept->store(khz);
    }
    return 1e3 * (double)khz;
}

// Seconds a sweep of one instance takes on a cluster of C blocks, and of I instances through
// the row kernels on `sms` SMs, fitted to measurements on a GB300 (K = 32): clusters 2.1 us at
// L = 8 (C = 2), 2.7 at L = 16, 6.1 at L = 24, 9.4 at L = 32, 49.6 at L = 64 (C = 8); row
// kernels about 10 us of launches and 6.2 attempts per SM clock.  On C = 16: 2.4 us at L = 16, 5.1
// at 24, 6.5 at 32, 12.5 at 40 (the row kernels 11.9).  The line fits from L = 24 on.  Smaller
// lattices sit in resident blocks, for which it gives about 4 us where 2.1 to 2.7 were measured;
// that is far enough below the row kernels' 10 us for the choice to be the same.
double cluster_seconds(int L, int C, double hz) { return 3.7e-6 + 64.0 * slab::pairs_of(L, C) / (11.0 * hz); }
double row_seconds(double work, int I, int sms, double hz) { return 10e-6 + I * work / (sms * 6.2 * hz); }
}  // namespace

// Blocks per word for a PT run of I instances of side L with K <= 64 temperatures and
// unit couplings, or 0 when the row kernels should run it.  C is the largest, up to 16 blocks a
// cluster, that makes the slabs thinner, whose largest slab fits shared memory and for which
// all I clusters are resident at once (one wave) -- but no larger than leaves a block 128 pairs
// of sites, a warp for each partition of its SM (L = 8: 2.11 us a sweep on one or two blocks,
// 2.45 on eight).  The cluster form is taken when its estimated time per sweep is below the row
// kernels'.  Knob SG_PT_CLUSTER = 0 turns the form off, = 1 takes it whenever a slab fits.
int pt_cluster_blocks(int I, int L, int K, double* seconds)
{
    if (seconds) *seconds = 0;
    const char* e = getenv("SG_PT_CLUSTER");
    const int knob = e ? atoi(e) : -1;
    if (knob == 0 || !runs(L, K) || I < 1) return 0;
    int dev = 0, smem = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const double hz = device_hz();
    const int words = words_for(K);
    const char* fc = getenv("SG_PT_CLUSTER_C");  // tuning knob: force C (when it fits)
    const int forced = fc ? atoi(fc) : 0;
    for (int C = slab::kMaxC / words; C >= 1; --C) {
        if (forced > 0 ? C != forced || C > L : !slab::worth(L, C)) continue;
        if (all_smem(L, C, words) > (size_t)smem) continue;
        const int fit = resident(L, C, words);
        if ((knob == 1 || forced > 0) && fit > 0) return C;
        if (fit < I) continue;
        bool smaller = false;  // a smaller cluster with blocks of at most 128 pairs
        for (int c = C - 1; c >= 1 && !smaller; --c) smaller = slab::pairs_of(L, c) <= 128;
        if (smaller) continue;
        const double work = (double)L * L * L * 32.0 * words;  // attempts per sweep of one instance (whole words)
        const double t = cluster_seconds(L, C, hz);
        if (seconds) *seconds = t;
        return t < 0.95 * row_seconds(work, I, sms, hz) ? C : 0;
    }
    return 0;
}

// Blocks per cluster for one request of a server with `busy` requests in service (0: row
// kernels).  A form's time per sweep is its own or, where that is longer, busy times its share
// of the device: the row kernels spread an instance over every SM and take the least time
// alone, but at L = 64 a sweep costs them 4.3 us of the whole device and a cluster of eight
// blocks 2.6; small lattices share the device best on few blocks each.
int pt_cluster_blocks_shared(int L, int K, int busy)
{
    const char* e = getenv("SG_PT_CLUSTER");
    if (e || busy <= 1) return pt_cluster_blocks(1, L, K);
    if (!runs(L, K) || words_for(K) > 1) return 0;
    int dev = 0, smem = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const double hz = device_hz();
    const double work = (double)L * L * L * 32.0;
    double best = 0.95 * std::max(row_seconds(work, 1, sms, hz), busy * (row_seconds(work, 1, sms, hz) - 10e-6));
    int bestC = 0;
    for (int C = 8; C >= 1; --C) {
        if (!slab::worth(L, C) || all_smem(L, C, 1) > (size_t)smem) continue;
        const double t = cluster_seconds(L, C, hz), shared = std::max(t, busy * C * t / sms);
        if (shared < best && resident(L, C, 1) > 0) {
            best = shared;
            bestC = C;
        }
    }
    return bestC;
}

// A batch with more instances than clusters fit at once: the first M instances on clusters
// (one wave), the other I - M through the row kernels on the SMs the clusters leave, both
// at the same time.  With the rates above, M minimises the longer of the two parts' times
// per sweep, and the split is taken when that beats the row kernels on the whole GPU.  At
// L = 64 with 16 instances of 32 temperatures: 15 clusters of 8 blocks on 120 SMs, one
// instance on the other 32.  Knob SG_PT_HYBRID = 0 turns the split off; SG_PT_CLUSTER = 0
// turns off every cluster form.
int pt_cluster_split(int I, int L, int K, int* M, int* side_sms, double* seconds)
{
    *seconds = 0;
    *M = 0;
    *side_sms = 0;
    const char* e = getenv("SG_PT_HYBRID");
    if (e && atoi(e) == 0) return 0;
    const char* c = getenv("SG_PT_CLUSTER");
    if ((c && atoi(c) == 0) || !runs(L, K) || I < 2) return 0;
    int dev = 0, smem = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const double hz = device_hz();
    const int words = words_for(K);
    const double work = (double)L * L * L * 32.0 * words;  // whole words
    double best = 0.95 * row_seconds(work, I, sms, hz);
    int bestC = 0;
    for (int C = slab::kMaxC / words; C >= 1; --C) {
        if (!slab::worth(L, C) || all_smem(L, C, words) > (size_t)smem) continue;
        const int active = resident(L, C, words);
        if (active >= I || active < 1) continue;  // one wave: pt_cluster_blocks decides
        const int per_sm = std::max(1, (active * C * words + sms - 1) / sms);  // blocks an SM holds
        const double t_cluster = cluster_seconds(L, C, hz);
        for (int m = active; m >= 1; --m) {
            const int left = sms - (m * C * words + per_sm - 1) / per_sm;
            if (left < 1) continue;
            const double t_side = row_seconds(work, I - m, left, hz);
            const double t = t_cluster > t_side ? t_cluster : t_side;
            if (t < best) {
                best = t;
                bestC = C;
                *M = m;
                *side_sms = left;
            }
        }
    }
    *seconds = best;
    return bestC;
}

int32_t launch_pt_cluster(int8_t* spins, const uint8_t* const* j1_ptrs, const RunKeys* keys, const uint32_t* thr,
                          uint8_t* rung_of_slot, uint8_t* slot_of_rung, int32_t* E, unsigned long long* accepts,
                          int32_t* minE, const ExchangeTablesDev& xt, int* status, int I, int L, int K, int C,
                          int s_begin, int s_end, cudaStream_t st, const ChunkReport& report)
{
    PtcArgs a{};
    a.report = report;
    a.wait_limit = wait_limit_cycles();
    a.spins = reinterpret_cast<uint32_t*>(spins);
    a.j1_ptrs = j1_ptrs;
    a.keys = keys;
    a.thr = thr;
    a.rung_of_slot = rung_of_slot;
    a.slot_of_rung = slot_of_rung;
    a.E = E;
    a.accepts = accepts;
    a.minE = minE;
    a.xtab = xt.tab;
    a.xoff = xt.off;
    a.xlen = xt.len;
    a.xtail = xt.tail;
    a.status = status;
    a.L = L;
    a.K = K;
    a.C = C;
    a.s_begin = s_begin;
    a.s_end = s_end;
    const int H = L / 2;
    a.Hmagic = H == 1 ? 0u : (uint32_t)((0x100000000ull + (uint64_t)H - 1) / (uint64_t)H);
    int dev = 0, most = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    // the exchange thresholds in shared memory when they fit beside the slab
    const size_t xbytes = sizeof(uint32_t) * xt.words;
    const int words = words_for(K);
    const void* const fn = kernel_of(L, C, words);
    a.xwords = all_smem(L, C, words) + xbytes <= (size_t)most ? (int)xt.words : 0;
    const size_t smem = dyn_smem(L, C) + sizeof(uint32_t) * (size_t)a.xwords;
    if (!allow_shared(fn)) {
        set_error("pt_cluster_kernel: cannot use %zu bytes of shared memory", smem);
        return SG_ECUDA;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C * words;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(C * words * I, 1, 1);
    cfg.blockDim = dim3(block_threads(L, C), 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[] = {&a};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("pt_cluster_kernel launch failed: %s", cudaGetErrorString(e));
        return SG_ECUDA;
    }
    return SG_OK;
}

}  // namespace sg
