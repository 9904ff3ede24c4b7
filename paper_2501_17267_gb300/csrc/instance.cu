// instance.cu -- tile-planting instance generator (host) and instance handles.
//
// Tile planting (arXiv:2501.17267, Sec. II): the periodic lattice is cut into unit
// cubes ("tiles") whose origins have all-even or all-odd coordinates; these N/4
// cubes share no edge and cover every edge once.  Each tile takes the couplings of
// a class template placed under a random cube symmetry.  Each template has the
// all-+1 corner state among its ground states, so the global all-+1 state is a
// ground state of the whole lattice and E_gs is the sum of the template minima.
// A random gauge tau then hides it: J'_ij = J_ij tau_i tau_j, planted state tau.
//
// The class templates are ferromagnetic cubes (J = -1) with a few antiferromagnetic
// (J = +1) edges that frustrate the faces the class is named after:
//   F22: x-edge at corner (0,0,0)                               -> 2 adjacent faces
//   F42: x-edges at (0,0,0) and (0,1,1)                         -> 4 faces, x-faces free
//   F6 : x-edge at (0,0,0), y-edge at (0,0,1), z-edge at (1,1,0) -> all 6 faces
// with minima -10, -8, -6 (one, two, three unsatisfiable edges).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <array>

#include "philox.cuh"
#include "sg_internal.h"

namespace sg {
namespace {

struct TemplateEdge {
    int corner[3];  // lower corner of the edge inside the unit cube
    int axis;       // 0 = x, 1 = y, 2 = z
    int8_t J;
};

// The twelve edges of a class template, each with its coupling.
std::array<TemplateEdge, 12> class_template(int cls)
{
    std::array<TemplateEdge, 12> t{};
    int n = 0;
    for (int axis = 0; axis < 3; ++axis)
        for (int hi = 0; hi < 2; ++hi)
            for (int lo = 0; lo < 2; ++lo) {
                // the two coordinates other than `axis`, lower axis first
                int c[3] = {0, 0, 0};
                int oa = axis == 0 ? 1 : 0;
                int ob = axis == 2 ? 1 : 2;
                c[oa] = lo;
                c[ob] = hi;
                t[n].corner[0] = c[0];
                t[n].corner[1] = c[1];
                t[n].corner[2] = c[2];
                t[n].axis = axis;
                t[n].J = -1;
                ++n;
            }
    auto flip = [&](int axis, int x, int y, int z) {
        for (auto& e : t)
            if (e.axis == axis && e.corner[0] == x && e.corner[1] == y && e.corner[2] == z)
                e.J = +1;
    };
    flip(0, 0, 0, 0);
    if (cls == 1) flip(0, 0, 1, 1);
    if (cls == 2) {
        flip(1, 0, 0, 1);
        flip(2, 1, 1, 0);
    }
    return t;
}

constexpr int kTemplateMin[3] = {-10, -8, -6};

// Cube symmetry g = 8 p + r: axis permutation p (lexicographic order over the six
// permutations of (x, y, z)) and reflection bits r.  The image of a corner has, on
// axis a, the original coordinate on axis perm[a], mirrored when bit a of r is set.
struct CubeSymmetry {
    int perm[3];
    int refl;
    void apply(const int in[3], int out[3]) const
    {
        for (int a = 0; a < 3; ++a) out[a] = in[perm[a]] ^ ((refl >> a) & 1);
    }
};

CubeSymmetry cube_symmetry(int g)
{
    int perms[6][3];
    int order[3] = {0, 1, 2};
    int n = 0;
    do {
        perms[n][0] = order[0];
        perms[n][1] = order[1];
        perms[n][2] = order[2];
        ++n;
    } while (std::next_permutation(order, order + 3));
    CubeSymmetry s;
    for (int a = 0; a < 3; ++a) s.perm[a] = perms[g / 8][a];
    s.refl = g % 8;
    return s;
}

struct PlacedEdge {  // tile-relative lower corner and axis of an image edge
    int dx, dy, dz, axis;
    int8_t J;
};
using Placements = std::array<std::array<std::array<PlacedEdge, 12>, 48>, 3>;

// All (class, symmetry) placements.
const Placements& placements()
{
    static const Placements placed = [] {
        Placements P{};
        for (int cls = 0; cls < 3; ++cls) {
            auto t = class_template(cls);
            for (int g = 0; g < 48; ++g) {
                CubeSymmetry s = cube_symmetry(g);
                for (int e = 0; e < 12; ++e) {
                    int a[3] = {t[e].corner[0], t[e].corner[1], t[e].corner[2]};
                    int b[3] = {a[0], a[1], a[2]};
                    b[t[e].axis] = 1;
                    int ga[3], gb[3];
                    s.apply(a, ga);
                    s.apply(b, gb);
                    int axis = 0;
                    while (ga[axis] == gb[axis]) ++axis;
                    const int* lo = ga[axis] < gb[axis] ? ga : gb;
                    P[cls][g][e] = PlacedEdge{lo[0], lo[1], lo[2], axis, t[e].J};
                }
            }
        }
        return P;
    }();
    return placed;
}

// Inverse CDF of a 32-bit uniform word: the cumulative class weights in 2^32 fixed point.
struct ClassCuts {
    uint64_t cut0, cut1;
};
ClassCuts class_cuts(const double class_prob[3])
{
    const double w0 = class_prob[0], w1 = class_prob[1], total = w0 + w1 + class_prob[2];
    return ClassCuts{(uint64_t)floor(ldexp(w0 / total, 32)), (uint64_t)floor(ldexp((w0 + w1) / total, 32))};
}

// ---- the same generator on the device, for instances whose couplings the host never reads ----

// A placed edge in a byte: lower corner (3 bits), axis (2), negative (1).
struct PackedPlacements {
    uint8_t e[3][48][12];
};

// One thread a tile: its class and symmetry, the couplings of its twelve edges (each edge
// belongs to one tile), the sum of the tiles' minima.
__global__ void generate_tiles_kernel(const PackedPlacements placed, int L, uint32_t k0, uint32_t k1, uint64_t cut0,
                                      uint64_t cut1, int8_t* __restrict__ J3, unsigned long long* __restrict__ e_gs)
{
    const int H = L >> 1, half = H * H * H;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    int E = 0;
    if (t < 2 * half) {
        const Philox4 r = philox4x32_10((uint32_t)t, 0, 0, kDomainGenerate, k0, k1);
        const int cls = r.v[0] < cut0 ? 0 : r.v[0] < cut1 ? 1 : 2;
        const int g = (int)__umulhi(r.v[1], 48u);
        constexpr int m0 = kTemplateMin[0], m1 = kTemplateMin[1], m2 = kTemplateMin[2];
        E = cls == 0 ? m0 : cls == 1 ? m1 : m2;
        const int parity = t >= half, q = t - parity * half;
        const int ox = 2 * (q % H) + parity, oy = 2 * (q / H % H) + parity, oz = 2 * (q / (H * H)) + parity;
#pragma unroll
        for (int e = 0; e < 12; ++e) {
            const int b = placed.e[cls][g][e];
            int x = ox + (b & 1), y = oy + ((b >> 1) & 1), z = oz + ((b >> 2) & 1);
            x = x >= L ? x - L : x, y = y >= L ? y - L : y, z = z >= L ? z - L : z;
            J3[3 * (x + L * (y + L * z)) + ((b >> 3) & 3)] = (b & 32) ? (int8_t)-1 : (int8_t)1;
        }
    }
    E = __reduce_add_sync(0xFFFFFFFFu, E);
    if ((threadIdx.x & 31) == 0 && E) atomicAdd(e_gs, (unsigned long long)(long long)E);
}

// Gauge of every site: 1 where tau = -1.
__global__ void generate_gauge_kernel(int N, int gauge, uint32_t k0, uint32_t k1, uint8_t* __restrict__ tau)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) tau[i] = gauge ? (uint8_t)(philox4x32_10((uint32_t)i, 0, 0, kDomainGauge, k0, k1).v[0] >> 31) : (uint8_t)0;
}

// The per-site records of the gauged couplings J tau tau' (kernels.cu: bytes +x, -x, +y, -y,
// +z, -z; sign bits).
__global__ void generate_records_kernel(const int8_t* __restrict__ J3, const uint8_t* __restrict__ tau, int L,
                                        uint2* __restrict__ j6, uint8_t* __restrict__ j1)
{
    const int LL = L * L, i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= LL * L) return;
    const int x = i % L, y = i / L % L, z = i / LL;
    const int xp = i + (x + 1 == L ? 1 - L : 1), xm = i + (x == 0 ? L - 1 : -1);
    const int yp = i + (y + 1 == L ? L - LL : L), ym = i + (y == 0 ? LL - L : -L);
    const int zp = i + (z + 1 == L ? LL - LL * L : LL), zm = i + (z == 0 ? LL * L - LL : -LL);
    const uint32_t t = tau[i];
    const uint32_t n = ((uint32_t)(J3[3 * i] < 0) ^ t ^ tau[xp]) | ((uint32_t)(J3[3 * xm] < 0) ^ t ^ tau[xm]) << 1 |
                       ((uint32_t)(J3[3 * i + 1] < 0) ^ t ^ tau[yp]) << 2 | ((uint32_t)(J3[3 * ym + 1] < 0) ^ t ^ tau[ym]) << 3 |
                       ((uint32_t)(J3[3 * i + 2] < 0) ^ t ^ tau[zp]) << 4 | ((uint32_t)(J3[3 * zm + 2] < 0) ^ t ^ tau[zm]) << 5;
    auto coupling = [&](int q) { return (n >> q) & 1u ? 0xFFu : 0x01u; };
    j6[i] = make_uint2(coupling(0) | coupling(1) << 8 | coupling(2) << 16 | coupling(3) << 24, coupling(4) | coupling(5) << 8);
    j1[i] = (uint8_t)n;
}

}  // namespace

int32_t launch_generate_instance(const sg_instance_desc& d, int8_t* J3, uint8_t* tau, unsigned long long* e_gs,
                                 uint2* j6, uint8_t* j1, cudaStream_t st)
{
    PackedPlacements packed;
    const Placements& P = placements();
    for (int c = 0; c < 3; ++c)
        for (int g = 0; g < 48; ++g)
            for (int e = 0; e < 12; ++e) {
                const PlacedEdge& q = P[c][g][e];
                packed.e[c][g][e] = (uint8_t)(q.dx | q.dy << 1 | q.dz << 2 | q.axis << 3 | (q.J < 0 ? 32 : 0));
            }
    const ClassCuts cuts = class_cuts(d.class_prob);
    const uint32_t k0 = (uint32_t)d.seed, k1 = (uint32_t)(d.seed >> 32);
    const int L = d.L, N = L * L * L, threads = 256;
    SG_TRY_CUDA(cudaMemsetAsync(e_gs, 0, sizeof(*e_gs), st));
    generate_tiles_kernel<<<(N / 4 + threads - 1) / threads, threads, 0, st>>>(packed, L, k0, k1, cuts.cut0, cuts.cut1,
                                                                              J3, e_gs);
    generate_gauge_kernel<<<(N + threads - 1) / threads, threads, 0, st>>>(N, d.gauge, k0, k1, tau);
    generate_records_kernel<<<(N + threads - 1) / threads, threads, 0, st>>>(J3, tau, L, j6, j1);
    SG_TRY_CUDA(cudaGetLastError());
    return SG_OK;
}

int64_t planted_energy(const sg_instance_desc& d)
{
    const ClassCuts cuts = class_cuts(d.class_prob);
    const uint32_t k0 = (uint32_t)d.seed, k1 = (uint32_t)(d.seed >> 32);
    const int64_t tiles = (int64_t)d.L * d.L * d.L / 4;
    int64_t E = 0;
    for (int64_t t = 0; t < tiles; ++t) {
        const uint32_t r = philox4x32_10((uint32_t)t, 0, 0, kDomainGenerate, k0, k1).v[0];
        E += kTemplateMin[r < cuts.cut0 ? 0 : r < cuts.cut1 ? 1 : 2];
    }
    return E;
}

int32_t generate_instance(int L, uint64_t seed, const double class_prob[3], int gauge,
                          int8_t* J3, int8_t* planted, int64_t* e_gs)
{
    if (L < 2 || L > SG_LMAX || (L & 1)) {
        set_error("L must be even with 2 <= L <= %d (got %d)", SG_LMAX, L);
        return SG_EINVAL;
    }
    const double w0 = class_prob[0], w1 = class_prob[1], w2 = class_prob[2];
    if (!(w0 >= 0 && w1 >= 0 && w2 >= 0) || !(w0 + w1 + w2 > 0)) {
        set_error("class_prob must be non-negative with a positive sum");
        return SG_EINVAL;
    }
    const auto [cut0, cut1] = class_cuts(class_prob);
    const Placements& placed = placements();

    const int64_t N = (int64_t)L * L * L;
    const int H = L / 2;
    const int64_t half = (int64_t)H * H * H;
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    auto wrap = [L](int v) { return v >= L ? v - L : v; };
    int64_t E = 0;
    for (int parity = 0; parity < 2; ++parity)
        for (int c = 0; c < H; ++c)
            for (int b = 0; b < H; ++b)
                for (int a = 0; a < H; ++a) {
                    const int64_t t = parity * half + a + (int64_t)H * (b + (int64_t)H * c);
                    const Philox4 r = philox4x32_10((uint32_t)t, 0, 0, kDomainGenerate, k0, k1);
                    const int cls = r.v[0] < cut0 ? 0 : (r.v[0] < cut1 ? 1 : 2);
                    const int g = (int)(((uint64_t)r.v[1] * 48u) >> 32);
                    E += kTemplateMin[cls];
                    const int ox = 2 * a + parity, oy = 2 * b + parity, oz = 2 * c + parity;
                    for (const PlacedEdge& pe : placed[cls][g]) {
                        const int64_t i = wrap(ox + pe.dx) +
                                          (int64_t)L * (wrap(oy + pe.dy) + (int64_t)L * wrap(oz + pe.dz));
                        J3[3 * i + pe.axis] = pe.J;
                    }
                }
    for (int64_t i = 0; i < N; ++i) {
        const Philox4 r = philox4x32_10((uint32_t)i, 0, 0, kDomainGauge, k0, k1);
        planted[i] = (gauge && (r.v[0] >> 31)) ? -1 : 1;
    }
    if (gauge) {
        for (int z = 0; z < L; ++z)
            for (int y = 0; y < L; ++y)
                for (int x = 0; x < L; ++x) {
                    const int64_t i = x + (int64_t)L * (y + (int64_t)L * z);
                    const int64_t nb[3] = {wrap(x + 1) + (int64_t)L * (y + (int64_t)L * z),
                                           x + (int64_t)L * (wrap(y + 1) + (int64_t)L * z),
                                           x + (int64_t)L * (y + (int64_t)L * wrap(z + 1))};
                    for (int d = 0; d < 3; ++d)
                        J3[3 * i + d] = (int8_t)(J3[3 * i + d] * planted[i] * planted[nb[d]]);
                }
    }
    *e_gs = E;
    return SG_OK;
}

// Upload J3 and build the per-site six-coupling records on the current device
// (once per device; later calls reuse the copy).
int32_t instance_device_j6(sg_instance* inst, cudaStream_t stream, const uint2** j6,
                           const uint8_t** j1)
{
    int dev = 0;
    SG_TRY_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(inst->mu);
    for (auto& d : inst->dev)
        if (d.device == dev) {
            *j6 = d.j6;
            if (j1) *j1 = d.j1;
            return SG_OK;
        }
    DeviceCopy dc;
    dc.device = dev;
    int8_t* J3d = nullptr;
    const size_t N = (size_t)inst->N;
    // one allocation: [N] uint2 records, then [N] sign bytes
    cudaError_t e = cudaMalloc(&dc.j6, sizeof(uint2) * N + N);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("cudaMalloc: %s", cudaGetErrorString(e));
        return SG_ENOMEM;
    }
    dc.j1 = reinterpret_cast<uint8_t*>(dc.j6 + N);
    e = cudaMalloc(&J3d, 3 * N);
    if (e != cudaSuccess) {
        cudaGetLastError();
        cudaFree(dc.j6);
        set_error("cudaMalloc: %s", cudaGetErrorString(e));
        return SG_ENOMEM;
    }
    e = cudaMemcpyAsync(J3d, inst->J3.data(), 3 * N, cudaMemcpyHostToDevice, stream);
    int32_t rc = e == cudaSuccess ? launch_prepare_j6(J3d, dc.j6, dc.j1, inst->L, stream) : SG_ECUDA;
    if (rc == SG_OK) {
        e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) rc = SG_ECUDA;
    }
    cudaFree(J3d);
    if (rc != SG_OK) {
        cudaFree(dc.j6);
        set_error("uploading couplings failed: %s", cudaGetErrorString(e));
        return rc;
    }
    inst->dev.push_back(dc);
    *j6 = dc.j6;
    if (j1) *j1 = dc.j1;
    return SG_OK;
}

}  // namespace sg

using namespace sg;

static int32_t finish_instance(sg_instance* inst)
{
    int64_t s = 0;
    bool unit = true;
    for (int8_t j : inst->J3) {
        s += j < 0 ? -j : j;
        unit &= (j == 1 || j == -1);
    }
    inst->abs_sum = (int32_t)s;
    inst->unit_couplings = unit;
    return SG_OK;
}

extern "C" int32_t sg_instance_create(const sg_instance_desc* d, sg_instance** out)
{
    clear_error();
    if (!d || !out) {
        set_error("NULL argument");
        return SG_EINVAL;
    }
    if (d->L < 2 || d->L > SG_LMAX || (d->L & 1)) {
        set_error("L must be even with 2 <= L <= %d (got %d)", SG_LMAX, d->L);
        return SG_EINVAL;
    }
    sg_instance* inst = new (std::nothrow) sg_instance;
    if (!inst) return SG_ENOMEM;
    inst->L = d->L;
    inst->N = (int64_t)d->L * d->L * d->L;
    try {
        inst->J3.assign((size_t)(3 * inst->N), 0);
        inst->planted.assign((size_t)inst->N, 1);
    } catch (...) {
        delete inst;
        set_error("host allocation failed");
        return SG_ENOMEM;
    }
    int32_t rc = generate_instance(d->L, d->seed, d->class_prob, d->gauge, inst->J3.data(),
                                   inst->planted.data(), &inst->e_gs);
    if (rc != SG_OK) {
        delete inst;
        return rc;
    }
    finish_instance(inst);
    *out = inst;
    return SG_OK;
}

extern "C" int32_t sg_instance_create_from_couplings(int32_t L, const int8_t* J3, int32_t mem_kind,
                                                     int64_t e_gs, sg_instance** out)
{
    clear_error();
    if (!J3 || !out || (mem_kind != SG_MEM_HOST && mem_kind != SG_MEM_DEVICE)) {
        set_error("NULL argument or bad mem_kind");
        return SG_EINVAL;
    }
    if (L < 2 || L > SG_LMAX || (L & 1)) {
        set_error("L must be even with 2 <= L <= %d (got %d)", SG_LMAX, L);
        return SG_EINVAL;
    }
    sg_instance* inst = new (std::nothrow) sg_instance;
    if (!inst) return SG_ENOMEM;
    inst->L = L;
    inst->N = (int64_t)L * L * L;
    inst->e_gs = e_gs;
    try {
        inst->J3.resize((size_t)(3 * inst->N));
        inst->planted.assign((size_t)inst->N, 1);
    } catch (...) {
        delete inst;
        set_error("host allocation failed");
        return SG_ENOMEM;
    }
    if (mem_kind == SG_MEM_DEVICE) {
        cudaError_t e = cudaMemcpy(inst->J3.data(), J3, inst->J3.size(), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) {
            delete inst;
            set_error("cudaMemcpy: %s", cudaGetErrorString(e));
            return SG_ECUDA;
        }
    } else {
        memcpy(inst->J3.data(), J3, inst->J3.size());
    }
    for (int8_t j : inst->J3)
        if (j > SG_JMAX || j < -SG_JMAX) {
            delete inst;
            set_error("coupling %d exceeds |J| <= %d", (int)j, SG_JMAX);
            return SG_EINVAL;
        }
    finish_instance(inst);
    *out = inst;
    return SG_OK;
}

extern "C" int32_t sg_instance_get(const sg_instance* inst, int32_t* L_out, int8_t* J3_out,
                                   int8_t* planted_out, int64_t* e_gs_out)
{
    clear_error();
    if (!inst) {
        set_error("NULL instance");
        return SG_EINVAL;
    }
    if (L_out) *L_out = inst->L;
    if (J3_out) memcpy(J3_out, inst->J3.data(), inst->J3.size());
    if (planted_out) memcpy(planted_out, inst->planted.data(), inst->planted.size());
    if (e_gs_out) *e_gs_out = inst->e_gs;
    return SG_OK;
}

extern "C" int32_t sg_instance_destroy(sg_instance* inst)
{
    clear_error();
    if (!inst) return SG_OK;
    int cur = 0;
    cudaGetDevice(&cur);
    for (auto& d : inst->dev) {
        cudaSetDevice(d.device);
        cudaFree(d.j6);
    }
    if (!inst->dev.empty()) cudaSetDevice(cur);
    delete inst;
    return SG_OK;
}
