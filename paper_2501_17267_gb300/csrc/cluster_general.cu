// cluster_general.cu -- simulated annealing (App. D.1) of lattices whose couplings are not all
// +-1, with every sweep of a run in one launch: one thread-block cluster of C blocks per (word,
// instance), each holding a z-slab of the word's lattice in its shared memory (slab.cuh: the
// geometry and how neighbours exchange their faces).
//
// A thread takes pairs of sites n, n + threads, ...; a half sweep updates the pair's site of its
// colour.  A site's six couplings are one word of shared memory beside its spins; the update is
// the row kernels' (metropolis.cuh).  A face word goes to the neighbour as soon as its site is
// decided: nothing in the neighbour reads words of this colour in this half sweep, and it has
// finished with the old ones, which its own face words of the half sweep before told.
//
// What it is for: a half sweep of a small lattice is over sooner than its launch.  An L = 24
// lattice with 100 replicas takes 2.5 us a half sweep here and 3.6 through the row kernels, which
// also pay for the capture of their graphs (0.5 ms of a 2 ms call).  A warp's item takes about
// 670 cycles of an SM partition, its chain of draws, planes and tie decisions; a half sweep of
// nothing but its barriers and one item 1.1 us.
#include <cooperative_groups.h>
#include <stdint.h>
#include <stdlib.h>

#include <algorithm>

#include "metropolis.cuh"
#include "slab.cuh"
#include "sg_internal.h"

namespace cg = cooperative_groups;

namespace sg {
namespace {

constexpr int kThreads = slab::kMaxThreads;

struct GeneralArgs {
    uint32_t* spins;               // [I][N][Wn] words, storage order
    const uint2* const* j6_ptrs;   // per instance: [N] six-coupling records
    const RunKeys* keys;           // [I]
    const uint32_t* thr;           // [S][kThrRow]
    int* status;                   // SG_ETIMEOUT when a bounded wait gave up
    int L, Wn, R, C, S;            // side, words, replicas, blocks per cluster, sweeps
    long long wait_limit;          // cycles a wait for the neighbours lasts at most
    uint32_t Hmagic;               // ceil(2^32 / (L / 2))
};

// Records: six bits each of bonds that are negative, of weight 1, of weight 2 (order: near x,
// far x, +y, -y, +z, -z; the near x neighbour is the pair's other site), then the total weight.
constexpr int kRecOne = 6, kRecTwo = 12, kRecM = 18;

struct Shared {  // two sweeps' tables by sweep parity
    __align__(16) uint32_t planes[2][mp::kGeneralPlanes];
    slab::Geometry geo;
    uint32_t row[2][kThrRow];
    int draws[2];
    uint64_t bar[2];  // by colour: the neighbours' face words of that colour have arrived
    int fail[2];      // by colour: a wait for that barrier gave up (read one half sweep later)
};

__global__ void __launch_bounds__(kThreads, 1) sa_general_cluster_kernel(const GeneralArgs a)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ Shared sh;
    cg::cluster_group cluster = cg::this_cluster();
    const int C = a.C, L = a.L, H = L >> 1, LL = L * L;
    const int r = C > 1 ? (int)cluster.block_rank() : 0;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, threads = blockDim.x, warps = threads >> 5;
    const int word = blockIdx.y, inst = blockIdx.z;
    const slab::Geometry& geo = sh.geo;
    if (tid == 0) {
        sh.geo.init(L, C, r, warps, a.Hmagic);
        slab::mbar_init(&sh.bar[0]);
        slab::mbar_init(&sh.bar[1]);
        slab::mbar_init_fence();
        sh.fail[0] = sh.fail[1] = C > 1 && a.wait_limit == 0;
    }
    __syncthreads();
    const int zc = geo.zc, z0 = geo.z0, sites = zc * LL;
    uint32_t* const w = smem + LL;                              // the slab, a halo plane on either side
    uint32_t* const recs = smem + slab::Geometry::words(L, C);  // of its sites, in storage order
    uint32_t* const g = a.spins + (size_t)inst * LL * L * a.Wn + word;
    const uint2* __restrict__ j6 = a.j6_ptrs[inst];
    const int below = ((z0 == 0 ? L : z0) - 1) * LL, above = (z0 + zc == L ? 0 : z0 + zc) * LL;
    for (int q = tid; q < sites; q += threads) {
        w[q] = g[(size_t)(z0 * LL + q) * a.Wn];
        const int row = q / L, pos = q - row * L, odd = pos >= H;
        const uint2 rec = j6[z0 * LL + row * L + (odd ? 2 * (pos - H) + 1 : 2 * pos)];
        uint32_t bits = 0, M = 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int at = k < 2 && odd ? k ^ 1 : k;
            const int J = (int)(int8_t)(((at < 4 ? rec.x : rec.y) >> (8 * (at & 3))) & 0xFFu), weight = J < 0 ? -J : J;
            bits |= (J < 0 ? 1u : 0u) << k | (weight == 1 ? 1u : 0u) << (kRecOne + k) |
                    (weight == 2 ? 1u : 0u) << (kRecTwo + k);
            M += (uint32_t)weight;
        }
        recs[q] = bits | M << kRecM;
    }
    for (int q = tid; q < LL; q += threads) {
        w[q - LL] = g[(size_t)(below + q) * a.Wn];
        w[sites + q] = g[(size_t)(above + q) * a.Wn];
    }

    // Tables of sweep `sw`, by the last warp (lane k holds the row's entry k).
    auto set_tables = [&](int sw, uint32_t entry) {
        const int b = sw & 1;
        if (lane < kThrRow) sh.row[b][lane] = entry;
        const unsigned any = __ballot_sync(slab::kAll, entry != 0u && lane >= 1);
        if (lane == 0) sh.draws[b] = any != 0u;
        __syncwarp();
        for (int q = lane; q < mp::kGeneralPlanes; q += 32) sh.planes[b][q] = mp::general_plane_of(q, sh.row[b]);
    };
    auto entry_of = [&](int sw) { return lane < kThrRow && sw < a.S ? a.thr[(size_t)sw * kThrRow + lane] : 0u; };
    uint32_t entry = 0;  // last warp: the next sweep's row, loaded a sweep ahead of its use
    if (warp == warps - 1) {
        set_tables(0, entry_of(0));
        entry = entry_of(1);
    }

    slab::Draws draws;
    draws.k0 = a.keys[inst].k0;
    draws.k1 = a.keys[inst].k1;
    const RunKeys key = a.keys[inst];
    const uint32_t valid = slab::word_valid_bits(a.R, word);
    const uint32_t w0 = slab::smem_addr(w), up = (uint32_t)(r + 1 == C ? 0 : r + 1), dn = (uint32_t)(r == 0 ? C - 1 : r - 1);
    // what to add to the address of a face word for its copy above and below
    uint32_t up_w = 0u - (uint32_t)sites * 4u, dn_w = (uint32_t)sites * 4u, up_bar = 0, dn_bar = 0;
    if (C > 1) {
        up_w += slab::cluster_addr(w0, up) - w0;
        dn_w = slab::cluster_addr(w0, dn) - w0 + (uint32_t)(geo.zdn * LL) * 4u;
        up_bar = slab::cluster_addr(slab::smem_addr(&sh.bar[0]), up);
        dn_bar = slab::cluster_addr(slab::smem_addr(&sh.bar[0]), dn);
        cluster.sync();  // every block has loaded its halos before a neighbour pushes into them
    } else {
        __syncthreads();
    }

    const int pairs = zc * L * H;
    struct Item {
        int row, j, zl, y, odd;
    };
    auto item = [&](int n, int colour) {
        Item it;
        it.row = H == 1 ? n : (int)__umulhi((uint32_t)n, a.Hmagic);
        it.j = n - it.row * H;
        it.zl = (int)__umulhi((uint32_t)it.row, geo.Lmagic);
        it.y = it.row - it.zl * L;
        it.odd = (it.y + z0 + it.zl + colour) & 1;
        return it;
    };
    auto site_of = [&](const Item& it) { return (uint32_t)((z0 * L + it.row) * L + 2 * it.j + it.odd); };
    uint32_t A[8];
    uint32_t phase = 0;
    bool ok = true;
    draws.set_sweep(0u, (uint32_t)word);
    if (tid < pairs) draws.planes(site_of(item(tid, 0)), A);
    for (int sw = 0; sw < a.S && ok; ++sw) {
        const int b = sw & 1;
        const bool drawn = sh.draws[b] != 0;
        if (warp == warps - 1) {  // the other parity's tables were last read before the barrier that ended sweep sw - 1
            set_tables(sw + 1, entry);
            entry = entry_of(sw + 2);
        }
        for (int colour = 0; colour < 2; ++colour) {
            if (C > 1 && tid == 0) slab::mbar_expect(&sh.bar[colour], (uint32_t)LL * 4u);
            for (int n = tid; n < pairs; n += threads) {
                const Item it = item(n, colour);
                const int pos = it.row * L + it.odd * H + it.j;
                const uint32_t is = w0 + 4u * (uint32_t)pos;
                const uint32_t site = site_of(it);
                if (n != tid && drawn) draws.planes(site, A);
                const uint32_t self = slab::ld_word(is);
                const uint32_t nb[6] = {
                    slab::ld_word(is + 4 * (it.odd ? -H : H)),
                    slab::ld_word(is + 4 * (it.odd ? -H + (it.j + 1 == H ? 1 - H : 1) : H + (it.j == 0 ? H - 1 : -1))),
                    slab::ld_word(is + 4 * (it.y + 1 == L ? L - LL : L)),
                    slab::ld_word(is + 4 * (it.y == 0 ? LL - L : -L)),
                    slab::ld_word(is + 4 * LL),
                    slab::ld_word(is - 4 * LL)};
                const uint32_t rec = recs[pos];
                uint32_t neg[6], mask[6], one[6], two[6], c[4];
                mp::unit_signs(rec & 63u, neg);
#pragma unroll
                for (int k = 0; k < 6; ++k) neg[k] = mp::logic<mp::kXor3>(self, nb[k], neg[k]);  // satisfied
                mp::unit_signs((rec >> kRecOne) & 63u, mask);
#pragma unroll
                for (int k = 0; k < 6; ++k) one[k] = neg[k] & mask[k];
                mp::unit_signs((rec >> kRecTwo) & 63u, mask);
#pragma unroll
                for (int k = 0; k < 6; ++k) two[k] = neg[k] & mask[k];
                mp::satisfied_weight(one, two, c);
                const int M = (int)(rec >> kRecM);
                const uint32_t flip =
                    drawn ? mp::flips_general<true>(c, M, valid, sh.planes[b], sh.row[b], 0, A, site, (uint32_t)sw,
                                                    (uint32_t)word, key)
                          : mp::flips_general<false>(c, M, valid, sh.planes[b], sh.row[b], 0, A, site, (uint32_t)sw,
                                                     (uint32_t)word, key);
                const uint32_t v = self ^ flip;
                slab::st_word_if(1u, is, v);
                if (it.zl == 0) {  // to the upper halo of the block below
                    if (C == 1) slab::st_word_if(1u, is + dn_w, v);
                    else slab::push_word(is + dn_w, v, dn_bar + 8u * colour);
                }
                if (it.zl + 1 == zc) {  // to the lower halo of the block above
                    if (C == 1) slab::st_word_if(1u, is + up_w, v);
                    else slab::push_word(is + up_w, v, up_bar + 8u * colour);
                }
            }
            // the draws of the thread's first pair in the next half sweep, while the faces travel
            if (colour == 1) draws.set_sweep((uint32_t)sw + 1u, (uint32_t)word);
            if (tid < pairs) draws.planes(site_of(item(tid, colour ^ 1)), A);
            __syncthreads();
            if (C > 1) {
                const bool lost = sh.fail[colour ^ 1] != 0;  // set before this barrier, the same for every thread
                if (!slab::mbar_wait<false>(&sh.bar[colour], (phase >> colour) & 1u, a.wait_limit)) sh.fail[colour] = 1;
                phase ^= 1u << colour;
                if (lost) {  // (only now: no face may be on its way when the block leaves)
                    ok = false;
                    break;
                }
            }
        }
    }
    __syncthreads();
    ok = ok && !sh.fail[0] && !sh.fail[1];
    if (!ok && tid == 0) atomicExch(a.status, SG_ETIMEOUT);
    if (ok)
        for (int q = tid; q < sites; q += threads) g[(size_t)(z0 * LL + q) * a.Wn] = w[q];
    // no block leaves while another may still push to it
    if (C > 1) cluster.sync();
}

int block_threads(int L, int C)
{
    return (int)std::min<int64_t>(kThreads, (slab::pairs_of(L, C) + 31) / 32 * 32);
}
size_t dyn_smem(int L, int C) { return 4 * (slab::Geometry::words(L, C) + slab::Geometry::sites(L, C)); }

}  // namespace

// Blocks per cluster, or 0 when the row kernels should run it: the least estimated cycles of a
// half sweep, fitted to measurements on a GB300 (us at 2.07 GHz),
//   clusters     1700 + 670 per warp of pairs an SM partition holds (L = 8 on C = 4 1.1, L = 24 on
//                C = 12 2.5 and on C = 2 9.4)
//   row kernels  6600 + 1100 per warp of items over the whole GPU (L = 8 3.5, 12 words of L = 32 8.7)
// Clusters that are not resident at once run in waves.
int sa_general_cluster_blocks(int I, int L, int Wn, bool force)
{
    int dev = 0, smem = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t clusters = (int64_t)I * Wn;
    const char* e = getenv("SG_SA_CLUSTER_C");
    const int forced = e ? atoi(e) : 0;
    double best = 1e300;
    if (!force && !forced) best = 0.95 * (6600.0 + 1100.0 * (double)clusters * L * L * (L / 2) / 32.0 / (4.0 * sms));
    int bestC = 0;
    for (int C = 1; C <= slab::kMaxC; ++C) {
        if (forced ? C != forced || C > L : !slab::worth(L, C)) continue;
        if (dyn_smem(L, C) + sizeof(Shared) > (size_t)smem) continue;
        const int64_t active = resident_clusters((const void*)sa_general_cluster_kernel, C, dyn_smem(L, C), block_threads(L, C));
        if (active < 1) continue;
        const int64_t waves = (clusters + active - 1) / active;
        const int64_t per_sm = (std::min(clusters, active) * C + sms - 1) / sms;  // blocks on the busiest SM
        const double warps = std::max(1.0, (double)per_sm * (double)((slab::pairs_of(L, C) + 31) / 32) / 4.0);
        const double cost = waves * (1700.0 + 670.0 * warps);
        if (cost < best) {
            best = cost;
            bestC = C;
        }
    }
    return bestC;
}

int32_t launch_sa_general_cluster(int8_t* spins, const uint2* const* j6_ptrs, const RunKeys* keys, const uint32_t* thr,
                                  int* status, int I, int L, int Wn, int R, int S, int C, cudaStream_t st)
{
    GeneralArgs a{};
    a.spins = reinterpret_cast<uint32_t*>(spins);
    a.j6_ptrs = j6_ptrs;
    a.keys = keys;
    a.thr = thr;
    a.status = status;
    a.L = L;
    a.Wn = Wn;
    a.R = R;
    a.C = C;
    a.S = S;
    a.wait_limit = wait_limit_cycles();
    const int H = L / 2;
    a.Hmagic = H == 1 ? 0u : (uint32_t)((0x100000000ull + (uint64_t)H - 1) / (uint64_t)H);
    const void* const fn = (const void*)sa_general_cluster_kernel;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(C, Wn, I);
    cfg.blockDim = dim3(block_threads(L, C), 1, 1);
    cfg.dynamicSmemBytes = dyn_smem(L, C);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[] = {&a};
    cudaError_t e = allow_shared(fn) ? cudaLaunchKernelExC(&cfg, fn, args) : cudaErrorInvalidValue;
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("sa_general_cluster_kernel launch failed: %s", cudaGetErrorString(e));
        return SG_ECUDA;
    }
    return SG_OK;
}

}  // namespace sg
