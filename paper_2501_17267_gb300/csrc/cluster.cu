// cluster.cu -- simulated annealing (App. D.1) with every sweep in one launch: each word of
// 32 replicas on its own thread-block cluster.
//
// A half sweep of a small lattice is too little work to pay for a launch, and a whole
// lattice per block (batch.cu) leaves most SMs idle when an instance has few words.
// Here cluster (word, instance) of C blocks splits the lattice into C slabs of about L / C
// z-planes, block r keeping slab r of the word in its shared memory for the whole run
// (slab.cuh: the updates, and how the blocks exchange their faces).  Every attempt draws
// the same counters as the row kernel (site, sweep, word), so the results are
// bit-identical to it and to the oracle.
//
// One row of thresholds serves a whole sweep, which says beforehand how much a half sweep
// has to do: at beta > 1.4 every threshold that can matter is below 2^24, a draw can only
// accept when its leading byte is 0, and the byte-by-byte compare falls away; at
// beta > 5.6 the thresholds are all 0 and there is nothing to draw.
#include <cooperative_groups.h>
#include <stdint.h>
#include <stdlib.h>

#include <algorithm>
#include <cstdint>
#include <map>
#include <mutex>
#include <tuple>

#include "slab.cuh"
#include "sg_internal.h"

namespace cg = cooperative_groups;

namespace sg {
namespace {

constexpr int kListBlock = 512;  // threads a block of the batch form

struct ClusterArgs {
    uint32_t* spins;                // [I][N][Wn] words, storage order
    const uint8_t* const* j1_ptrs;  // per instance: [N] coupling sign bits (all |J| = 1)
    const RunKeys* keys;            // [I]
    const uint32_t* thr;            // [S][kThrRow]
    int* status;                    // SG_ETIMEOUT when a bounded wait gave up
    int L, Wn, R, C;                // side, words, replicas, blocks per cluster
    int s_begin, s_end;             // sweeps [s_begin, s_end)
    ChunkReport report;             // of a run of one instance and word
    long long wait_limit;           // cycles a wait for the neighbours lasts at most
    uint32_t Hmagic;                // ceil(2^32 / (L / 2))
};

// One word of one lattice, annealed by a cluster of C blocks (block r: z-slab r): the
// plane's word of site s is g[s * stride]; the draws use word index w of the instance.
struct PlaneRun {
    uint32_t* g;
    int stride;
    const uint8_t* j1;    // [N] coupling sign bits (all |J| = 1)
    const uint32_t* thr;  // [S][kThrRow]
    RunKeys key;
    int L, w, R, s_begin, s_end;  // side, word, replicas of the instance, sweeps [s_begin, s_end)
    uint32_t Hmagic;              // ceil(2^32 / (L / 2))
};

// Shared state of a block, two sweeps' tables by sweep parity.
struct Shared {
    slab::Planes planes[2];
    slab::Geometry geo;
    uint32_t row[2][kThrRow];
    int mode[2];
    uint64_t bar[2];  // by colour: the neighbours' face words of that colour have arrived
    int fail[2];      // by colour: a wait for that barrier gave up (read one half sweep later)
    int E[32];        // report: the block's energies, and in block 0 the cluster's
    int E_cluster[32];
};

// Called by every thread of every block of the cluster once the barriers are initialised;
// phase: the barriers' phase bits, kept from plane to plane.  Ends with the plane written
// back.  Returns false when a wait gave up (after `limit` cycles).
template <class S>
__device__ __forceinline__ bool anneal_plane(const PlaneRun& p, const int C, unsigned char* smem, Shared& sh,
                                             uint32_t& phase, const long long limit, bool energies = false)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int r = C > 1 ? (int)cluster.block_rank() : 0;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, warps = blockDim.x >> 5;
    const slab::Geometry& geo = sh.geo;
    if (tid == 0) sh.geo.init(p.L, C, r, warps, p.Hmagic);
    __syncthreads();
    uint32_t* w = reinterpret_cast<uint32_t*>(smem) + geo.LL;
    uint8_t* sgn = smem + slab::Geometry::words(p.L, C) * 4;
    slab::load_slab(geo, p.g, p.stride, p.j1, w, sgn);

    // Thresholds of sweep `sw` into the tables of its parity, by the last warp (lane k holds
    // the row's entry k): lane 3 j + m makes plane j of k = 2 + 2 m, lanes 24 .. 26 lz.
    const int src = 2 + 2 * (lane % 3), bit = 24 + (lane / 3) % 8;
    const int slot = lane / 3 * 4 + lane % 3;  // of Planes: tp[j] = {x, y, z, -}, then lz
    auto set_tables = [&](int sw, uint32_t entry) {
        const int b = sw & 1;
        const uint32_t t = __shfl_sync(slab::kAll, entry, src);
        const unsigned any = __ballot_sync(slab::kAll, t != 0u), lead = __ballot_sync(slab::kAll, t >> 24 != 0u);
        const uint32_t low = (t & 0xFFFFFFu) ? ~0u : 0u;
        if (lane < 27) reinterpret_cast<uint32_t*>(&sh.planes[b])[slot] = lane < 24 ? 0u - ((t >> bit) & 1u) : low;
        if (lane < kThrRow) sh.row[b][lane] = entry;
        if (lane == 0) sh.mode[b] = !any ? slab::kNoDraws : !lead ? slab::kTailOnly : slab::kCompare;
    };
    auto entry_of = [&](int sw) {
        return lane < kThrRow && sw < p.s_end ? p.thr[(size_t)sw * kThrRow + lane] : 0u;
    };
    uint32_t entry = 0;  // last warp: the next sweep's row, loaded a sweep ahead of its use
    if (warp == warps - 1) {
        set_tables(p.s_begin, entry_of(p.s_begin));
        entry = entry_of(p.s_begin + 1);
    }

    __syncthreads();  // the slab is in place
    S s(geo, w, sgn, reinterpret_cast<const uint4*>(smem + slab::smem_queue_offset(p.L, C)));
    s.draws.k0 = p.key.k0;
    s.draws.k1 = p.key.k1;
    s.word = (uint32_t)p.w;
    s.valid = slab::word_valid_bits(p.R, p.w);
    const uint32_t up = (uint32_t)(r + 1 == C ? 0 : r + 1), dn = (uint32_t)(r == 0 ? C - 1 : r - 1);
    uint32_t up_w = 0, dn_w = 0, up_bar = 0, dn_bar = 0;
    if (C > 1) {
        up_w = slab::cluster_addr(s.w0, up) - s.w0;
        dn_w = slab::cluster_addr(s.w0, dn) - s.w0;
        up_bar = slab::cluster_addr(slab::smem_addr(&sh.bar[0]), up);
        dn_bar = slab::cluster_addr(slab::smem_addr(&sh.bar[0]), dn);
        cluster.sync();  // every block has loaded its halos before a neighbour pushes into them
    } else {
        __syncthreads();
    }

    uint32_t A[S::kItems][8];
    bool ok = true;
    s.draws.set_sweep((uint32_t)p.s_begin, s.word);
    if constexpr (S::kAssisted) {
        if (s.drawer) s.template hand_over<0>();
        __syncthreads();
    } else {
        s.first_draws(A);
    }
    for (int sw = p.s_begin; sw < p.s_end && ok; ++sw) {
        const int b = sw & 1;
        const int mode = sh.mode[b];
        s.sweep = (uint32_t)sw;
        s.planes = slab::smem_addr(&sh.planes[b]);
        s.thr = sh.row[b];
        if (warp == warps - 1) {  // the other parity's tables were last read before the barrier that ended sweep sw - 1
            set_tables(sw + 1, entry);
            entry = entry_of(sw + 2);
        }
        // The end of a half sweep: the faces pushed, the block met, the neighbours' faces here.
        // False when the wait of the half sweep before gave up (its flag was set before this
        // barrier and is the same for every thread); this one's faces are waited for first, so
        // that none is on its way when the block leaves.
        auto finish = [&](int colour) {
            __syncthreads();
            if (C > 1) {
                const bool lost = sh.fail[colour ^ 1] != 0;
                if (!slab::mbar_wait<S::kResident>(&sh.bar[colour], (phase >> colour) & 1u, limit)) sh.fail[colour] = 1;
                phase ^= 1u << colour;
                if (lost) return false;
            }
            return true;
        };
        auto expect = [&](int colour) {
            if (C > 1 && tid == 0) slab::mbar_expect(&sh.bar[colour], (uint32_t)geo.LL * 4u);
        };
        if constexpr (S::kAssisted) {
            if (s.drawer) {
                if (mode != slab::kNoDraws) s.template hand_over<1>();
                if (!(ok = finish(0))) break;
                s.draws.set_sweep((uint32_t)sw + 1u, s.word);
                if (sh.mode[b ^ 1] != slab::kNoDraws) s.template hand_over<0>();
                ok = finish(1);
                continue;
            }
        }
        if constexpr (S::kResident) {
            expect(0);
            if (mode == slab::kCompare) s.template half<0, slab::kCompare, false, false>(A, true);
            else if (mode == slab::kTailOnly) s.template half<0, slab::kTailOnly, false, false>(A, true);
            else s.template half<0, slab::kNoDraws, false, false>(A, false);
            s.template push_faces<0>(C == 1, up_w, dn_w, up_bar, dn_bar);
            if (!(ok = finish(0))) break;
            const bool next = sh.mode[b ^ 1] != slab::kNoDraws;
            expect(1);
            if (mode == slab::kCompare) s.template half<1, slab::kCompare, false, false>(A, next);
            else if (mode == slab::kTailOnly) s.template half<1, slab::kTailOnly, false, false>(A, next);
            else s.template half<1, slab::kNoDraws, false, false>(A, next);
            s.template push_faces<1>(C == 1, up_w, dn_w, up_bar + 8u, dn_bar + 8u);
            ok = finish(1);
        } else {
            for (int colour = 0; colour < 2 && ok; ++colour) {
                expect(colour);
                if (mode == slab::kCompare) s.template half<slab::kCompare, false, false>(colour, A[0]);
                else if (mode == slab::kTailOnly) s.template half<slab::kTailOnly, false, false>(colour, A[0]);
                else {
                    s.template half<slab::kNoDraws, false, false>(colour, A[0]);
                    if (colour == 1 && sh.mode[b ^ 1] != slab::kNoDraws) s.first_draws(A);
                }
                s.push_faces(colour, C == 1, up_w, dn_w, up_bar + 8u * colour, dn_bar + 8u * colour);
                ok = finish(colour);
            }
        }
    }
    if (C > 1) {
        __syncthreads();
        ok = ok && !sh.fail[0] && !sh.fail[1];
    }
    const int n = geo.zc * geo.LL;
    uint32_t* dst = p.g + (size_t)geo.z0 * geo.LL * p.stride;
    if (ok)
        for (int q = tid; q < n; q += blockDim.x) dst[(size_t)q * p.stride] = w[q];
    if (energies) {  // of the words as they are (each bond joins a colour-0 and a colour-1 site), in block 0
        if (tid < 32) sh.E[tid] = sh.E_cluster[tid] = 0;
        __syncthreads();
        s.E = sh.E;
        if constexpr (S::kResident) s.template half<1, slab::kCountOnly, false, true>(A, false);
        else s.template half<slab::kCountOnly, false, true>(1, A[0]);
        s.energy_to_block();
        __syncthreads();
        if (C > 1) cluster.sync();  // block 0's sums are cleared
        if (warp == 0) atomicAdd(C > 1 ? cluster.map_shared_rank(&sh.E_cluster[lane], 0) : &sh.E_cluster[lane], sh.E[lane]);
    }
    __syncthreads();
    return ok;
}

// given_up: every wait counts as one that gave up.
__device__ __forceinline__ void init_shared(Shared& sh, bool given_up)
{
    if (threadIdx.x == 0) {
        slab::mbar_init(&sh.bar[0]);
        slab::mbar_init(&sh.bar[1]);
        slab::mbar_init_fence();
        sh.fail[0] = sh.fail[1] = given_up;
    }
    __syncthreads();
}

// S: slab::Sweeper, or slab::Resident when a block has a thread for each of its x pairs, or for
// every two.  A resident block has a warp more than that takes, whose first work is the tables
// (with one pair a thread it has no other).
template <class S>
__global__ void __launch_bounds__(S::kAssisted   ? 2 * slab::kAssistedPairs + 32
                                  : S::kResident ? slab::kMaxThreads + 32
                                                 : slab::kMaxThreads,
                                  1)
sa_cluster_kernel(const ClusterArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ Shared sh;
    const int w = blockIdx.y, inst = blockIdx.z;
    PlaneRun p;
    p.g = a.spins + (size_t)inst * a.L * a.L * a.L * a.Wn + w;
    p.stride = a.Wn;
    p.j1 = a.j1_ptrs[inst];
    p.thr = a.thr;
    p.key = a.keys[inst];
    p.L = a.L;
    p.w = w;
    p.R = a.R;
    p.s_begin = a.s_begin;
    p.s_end = a.s_end;
    p.Hmagic = a.Hmagic;
    init_shared(sh, a.C > 1 && a.wait_limit == 0);
    uint32_t phase = 0;
    if (!anneal_plane<S>(p, a.C, smem, sh, phase, a.wait_limit, a.report.out != nullptr) && threadIdx.x == 0)
        atomicExch(a.status, SG_ETIMEOUT);
    // no block leaves while another may still push to it; energies and status are complete
    if (a.C > 1) cg::this_cluster().sync();
    else __syncthreads();
    if (a.report.out && (a.C == 1 || cg::this_cluster().block_rank() == 0) && threadIdx.x < 32) {
        const int left = a.R - 32 * w, lane = threadIdx.x;
        const int least = __reduce_min_sync(slab::kAll, lane < left ? sh.E_cluster[lane] : 0x7FFFFFFF);
        if (lane == 0) a.report.write(least, *static_cast<volatile int*>(a.status));
    }
}

// Persistent form for batches (batch.cu's planes of one word, [N][1]).  Clusters take planes
// order[0 .. n_cluster) through the counter next[0] until none is left (no side below C), then each
// block by itself planes order[n_cluster .. n) through next[1]: a small lattice does not fill a
// cluster, its half sweep being a chain of latencies, and four of them side by side take little
// longer than one.  next[2]: status word.
__global__ void __launch_bounds__(kListBlock, 1) sa_cluster_list_kernel(const Plane* __restrict__ planes,
                                                                        const int* __restrict__ order, int n_cluster,
                                                                        int n, unsigned* __restrict__ next, int C,
                                                                        long long wait_limit)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ Shared sh;
    __shared__ int s_item;
    cg::cluster_group cluster = cg::this_cluster();
    const int r = (int)cluster.block_rank();
    init_shared(sh, C > 1 && wait_limit == 0);
    uint32_t phase = 0;
    bool ok = true;
    auto run = [&](int it, int blocks) {
        const Plane& q = planes[order[it]];
        PlaneRun p;
        p.g = q.spins;
        p.stride = 1;
        p.j1 = q.j1;
        p.thr = q.thr;
        p.key = RunKeys{q.k0, q.k1};
        p.L = q.L;
        p.w = q.w0;
        p.R = q.R;
        p.s_begin = q.s_begin;
        p.s_end = ok ? q.s_end : q.s_begin;  // after a wait gave up: no more sweeps
        p.Hmagic = q.Hmagic;
        bool done;
        switch (slab::resident_items(slab::pairs_of(q.L, blocks), kListBlock)) {
            case 1: done = anneal_plane<slab::Resident<1>>(p, blocks, smem, sh, phase, wait_limit); break;
            case 2: done = anneal_plane<slab::Resident<2>>(p, blocks, smem, sh, phase, wait_limit); break;
            default: done = anneal_plane<slab::Sweeper>(p, blocks, smem, sh, phase, wait_limit); break;
        }
        if (!done) {
            ok = false;
            if (threadIdx.x == 0) atomicExch(reinterpret_cast<int*>(next + 2), SG_ETIMEOUT);
        }
    };
    for (;;) {
        if (r == 0 && threadIdx.x == 0) {  // claim the next plane for the whole cluster
            const int it = (int)atomicAdd(next, 1u);
            for (int k = 0; k < C; ++k) *cluster.map_shared_rank(&s_item, k) = it;
        }
        cluster.sync();
        const int it = s_item;
        if (it >= n_cluster) break;
        run(it, C);
        cluster.sync();  // s_item is read in every block before it is written again
    }
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = n_cluster + (int)atomicAdd(next + 1, 1u);
        __syncthreads();
        const int it = s_item;
        if (it >= n) break;
        run(it, 1);
    }
    cluster.sync();  // no block leaves while rank 0 may still write its s_item
}

}  // namespace

// The driver's answer depends on nothing but these arguments and the device, and asking costs
// tens of microseconds a shape: it is kept (one entry a kernel and shape, a few hundred at most).
int resident_clusters(const void* fn, int C, size_t smem, int threads)
{
    static std::mutex mu;
    static std::map<std::tuple<int, const void*, int, size_t, int>, int> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const auto key = std::make_tuple(dev, fn, C, smem, threads);
    std::lock_guard<std::mutex> lock(mu);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(C, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int active = 0;
    if (!allow_shared(fn) || cudaOccupancyMaxActiveClusters(&active, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (known.size() < 4096) known.emplace(key, active);
    return active;
}

// Lets `fn` use clusters of up to 16 blocks, and as much dynamic shared memory as a block can
// have beside its static one.  (The limit is always the same one, so that launches from several
// threads do not lower it under one another.)
bool allow_shared(const void* fn)
{
    int dev = 0, most = 0;
    cudaFuncAttributes at{};
    if (cudaGetDevice(&dev) != cudaSuccess || cudaFuncGetAttributes(&at, fn) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)at.sharedSizeBytes) !=
            cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return true;
}

namespace {
// The kernel for a block of at most `threads` threads, and its threads: the resident forms get
// a warp more, for the tables, and the assisted form another set for the draws.
const void* sa_cluster_fn(int L, int C, int threads)
{
    const int64_t pairs = slab::pairs_of(L, C);
    if (slab::assisted(pairs, threads)) return (const void*)sa_cluster_kernel<slab::Resident<1, true>>;
    switch (slab::resident_items(pairs, threads)) {
        case 1: return (const void*)sa_cluster_kernel<slab::Resident<1>>;
        case 2: return (const void*)sa_cluster_kernel<slab::Resident<2>>;
        default: return (const void*)sa_cluster_kernel<slab::Sweeper>;
    }
}
int sa_block_threads(int L, int C, int threads)
{
    const int64_t pairs = slab::pairs_of(L, C);
    return slab::resident_threads(pairs, threads) * (slab::assisted(pairs, threads) ? 2 : 1) +
           (slab::resident_items(pairs, threads) ? 32 : 0);
}
// Cycles of a half sweep with `per_sm` blocks of at most `threads` threads on an SM (see below).
double half_sweep_cycles(int L, int C, int threads, int per_sm)
{
    const int64_t pairs = slab::pairs_of(L, C);
    const double warps = std::max(1.0, (double)per_sm * (double)((pairs + 31) / 32) / 4.0);
    return slab::assisted(pairs, threads)         ? 500.0 + 400.0 * warps
           : slab::resident_items(pairs, threads) ? 750.0 + 400.0 * warps
                                                  : 2000.0 + 350.0 * warps;
}
}  // namespace

// Blocks per cluster (and the threads to plan a block with) for an SA run of I instances of
// side L with Wn words, or 0 when the row kernel should run it.  Candidates are the C <= 16 (8 in
// a loaded server) whose largest slab fits shared memory and is thinner than with fewer blocks;
// clusters that are not resident at once (as the driver reports for the kernel) run in waves.  A
// half sweep's cycles, fitted to measurements on a GB300 (us at 2.07 GHz), times the waves:
//   resident blocks  750 + 400 per warp of pairs an SM partition holds (L = 16 with 1024
//                    replicas on C = 4 blocks of 16 warps 1.2), 500 + 400 where a second set of
//                    warps draws (L = 4 on one block of one warp 0.41)
//   other blocks     2000 + 350 per warp of items (hot schedules: 20 x L = 50 on C = 6, one wave,
//                    16.2, 4 x L = 64 on C = 16 11.9, 32 words of L = 64 on C = 8, three waves,
//                    59.8; cold ones, which seldom compare, down to 300)
//   row kernels      6500 + 520 per warp of items over the whole GPU (17.7, 10.0 and 54.5 for the
//                    same)
// The fewest cycles win, fewer blocks among equals.  With `busy` runs of the kind sharing the
// device (a loaded server) a form's time is its own or, if that is longer, busy times its share
// of the device.  One run alone: L = 16 with 1024 replicas takes C = 4 (2.4 ms a run of 1000
// sweeps against 5.1 at C = 2), L = 4 one block (0.82 ms; in line 1.05, 1.20 at C = 2 and 1.25 at
// C = 4).  force: a cluster form whatever the row kernel would take.  Knobs: SG_SA_CLUSTER_C
// forces C, SG_SA_CLUSTER_THREADS the threads.
int sa_cluster_blocks(int I, int L, int Wn, bool force, int* threads, int busy)
{
    *threads = slab::kMaxThreads;
    int dev = 0, smem = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t clusters = (int64_t)I * Wn;
    const char* e = getenv("SG_SA_CLUSTER_C");
    const int forced = e ? atoi(e) : 0;
    const char* et = getenv("SG_SA_CLUSTER_THREADS");
    const int t = et && atoi(et) >= 32 && atoi(et) <= slab::kMaxThreads ? atoi(et) / 32 * 32 : slab::kMaxThreads;
    *threads = t;
    const double row_items = (double)clusters * L * L * (L / 2) / 32.0;  // warps of items a half sweep
    const double row_share = 520.0 * row_items / (4.0 * sms);
    double best = force || forced ? 1e300 : 0.95 * std::max(6500.0 + row_share, busy * row_share);
    int bestC = 0;
    for (int C = 1; C <= (busy > 1 ? 8 : slab::kMaxC); ++C) {
        if (forced ? C != forced || C > L : !slab::worth(L, C)) continue;
        const int bt = sa_block_threads(L, C, t);
        const size_t bytes = slab::smem_bytes(L, C, bt);
        if (bytes + 2048 > (size_t)smem) continue;
        const int64_t active = resident_clusters(sa_cluster_fn(L, C, t), C, bytes, bt);
        if (active < 1) continue;
        const int64_t waves = (clusters + active - 1) / active;
        if (C > 8 && waves > 1 && !forced) continue;  // (a wave of these follows another slowly)
        const int64_t per_sm = (std::min(clusters, active) * C + sms - 1) / sms;  // blocks on the busiest SM
        double cost = waves * half_sweep_cycles(L, C, t, (int)per_sm);
        cost = std::max(cost, cost * busy * (double)(std::min(clusters, active) * C) / sms);
        if (cost < best) {
            best = cost;
            bestC = C;
        }
    }
    return bestC;
}

namespace {
// Shared memory of a block of the batch form: its slab of the largest lattice, or a whole small one.
size_t sa_list_smem(int max_L, int C)
{
    return std::max(slab::smem_bytes(max_L, C, kListBlock), slab::smem_bytes(std::min(max_L, kListAloneL), 1, kListBlock));
}
}  // namespace

// Blocks per cluster for a batch: the C with the least estimated time, max(all work over the
// clusters, the longest member on one).  14 lattices of sides 22, 40 and 44, 12 replicas: 1.0 ms
// a call; 7.4 where clusters had to divide every side, which left planes of one block each.
int sa_cluster_list_blocks(const int* Ls, const int* sweeps, const int* words, int n)
{
    int dev = 0, smem = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int max_L = *std::max_element(Ls, Ls + n), min_L = *std::min_element(Ls, Ls + n);
    int64_t small = 0;
    for (int k = 0; k < n; ++k) small += Ls[k] <= kListAloneL ? words[k] : 0;
    const bool alone = small >= sms;  // those run on single blocks
    double best = 1e300;
    int bestC = 0;
    for (int C = 1; C <= std::min(slab::kMaxC, min_L); ++C) {
        const size_t bytes = sa_list_smem(max_L, C);
        if (bytes + 2048 > (size_t)smem) continue;
        const int clusters = resident_clusters((const void*)sa_cluster_list_kernel, C, bytes, kListBlock);
        if (clusters < 1) continue;
        double total = 0, longest = 0;
        for (int k = 0; k < n; ++k) {
            const bool one = alone && Ls[k] <= kListAloneL;
            const double t = sweeps[k] * half_sweep_cycles(Ls[k], one ? 1 : C, kListBlock, 1);
            total += words[k] * (one ? t / C : t);
            longest = std::max(longest, t);
        }
        const double t = std::max(total / clusters, longest);
        if (t < best) {
            best = t;
            bestC = C;
        }
    }
    return bestC;
}

int32_t launch_sa_cluster_planes(const Plane* d_planes, const int* d_order, int n_cluster, int n, unsigned* d_next,
                                 int C, int max_L, cudaStream_t st)
{
    const size_t smem = sa_list_smem(max_L, C);
    const int clusters = resident_clusters((const void*)sa_cluster_list_kernel, C, smem, kListBlock);
    if (clusters < 1) {
        set_error("sa_cluster_list_kernel: no cluster of %d blocks with %zu bytes fits", C, smem);
        return SG_ECUDA;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(C * std::min(clusters, std::max(n_cluster, (n - n_cluster + C - 1) / C)), 1, 1);
    cfg.blockDim = dim3(kListBlock, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, sa_cluster_list_kernel, d_planes, d_order, n_cluster, n, d_next, C,
                                             wait_limit_cycles());
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("sa_cluster_list_kernel launch failed: %s", cudaGetErrorString(e));
        return SG_ECUDA;
    }
    return SG_OK;
}

int32_t launch_sa_cluster(int8_t* spins, const uint8_t* const* j1_ptrs, const RunKeys* keys, const uint32_t* thr,
                          int* status, int I, int L, int Wn, int R, int s_begin, int s_end, int C, int threads,
                          cudaStream_t st, const ChunkReport& report)
{
    if (threads < 32 || threads > slab::kMaxThreads || threads % 32) {
        set_error("sa_cluster_kernel: %d threads a block (a multiple of 32 up to %d)", threads, slab::kMaxThreads);
        return SG_EINVAL;
    }
    ClusterArgs a{};
    a.spins = reinterpret_cast<uint32_t*>(spins);
    a.j1_ptrs = j1_ptrs;
    a.keys = keys;
    a.thr = thr;
    a.status = status;
    a.L = L;
    a.Wn = Wn;
    a.R = R;
    a.s_begin = s_begin;
    a.s_end = s_end;
    a.report = report;
    a.wait_limit = wait_limit_cycles();
    a.C = C;
    const int H = L / 2;
    a.Hmagic = H == 1 ? 0u : (uint32_t)((0x100000000ull + (uint64_t)H - 1) / (uint64_t)H);
    const void* fn = sa_cluster_fn(L, C, threads);
    threads = sa_block_threads(L, C, threads);
    const size_t smem = slab::smem_bytes(L, C, threads);
    if (smem > 48 * 1024 && !allow_shared(fn)) {
        set_error("sa_cluster_kernel: cannot use %zu bytes of shared memory", smem);
        return SG_ECUDA;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(C, Wn, I);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[] = {&a};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("sa_cluster_kernel launch failed: %s", cudaGetErrorString(e));
        return SG_ECUDA;
    }
    return SG_OK;
}

}  // namespace sg
