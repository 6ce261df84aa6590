// Friends-of-friends halo finder (Sec. 2.1: FoF, linking length b = 0.2 mean
// inter-particle spacings; Sec. 2.5: halos of more than 100
// particles, Warren et al. 2006 masses M = m_p N (1 - N^-0.6)) and the halo
// mass function.
//
// Positions are taken in units of the mean spacing, u = q + d nq / L wrapped
// into [0, nq), in FP32 with every operation rounded once (the __f*_rn
// intrinsics are never contracted), so the friendship test r^2 <= b^2 gives
// the same answer bit for bit wherever it is evaluated.
//
// Cell list: one cell per mean spacing (nq^3 cells, cell = floor(u); b < 1/2
// keeps every friend in the 27 cells around a particle), built by counting
// sort: a histogram, an exclusive scan, and a scatter of (u, p) into cell
// order.
//
// Linking: a union-find over the sorted slots, so that the parents of particles
// that are near each other are near each other in memory.  A pair of friends is
// taken by the thread with the larger slot.  k_fof_hook hooks every particle
// under its first friend in slot order and stops there; k_fof_compress shortens
// the trees; k_fof_link then unites the pairs whose roots still differ, which
// after the first two steps one load per pair shows for most of them, and
// particles without a smaller friend are done before it.  (Uniting every pair
// with two finds over particle-indexed parents took 23.0 ms at 512^3, the hook
// and the link take 4.9 ms each; both wait on the loads of their candidates.)
// Where hardly any particle has a friend, hook and link find little to do and the
// passes over the parents count: the particle of a slot is kept apart from the record
// for them (512^3, L = 1536, node 3, b = 0.1: 6.75 ms for 6.70 in that form, b = 0.2:
// 7.14 for 7.30).  Calls of up to 64^3 such particles pay for three launches more
// (81 us for 65 at 32^3, 82 for 75 at 64^3; clustered ones take half the time).  Roots only
// ever hook under smaller slots, in lock-free steps; a group's label is the smallest
// particle index in it, so the labels do not depend on the order of anything.
#include "cola_common.cuh"

namespace cola {
namespace {

constexpr int kUnionCap = 1 << 20;  // default bound on the retries of one find or union
int g_union_cap = kUnionCap;        // the bound in use (cola_fof_set_retry_cap)
constexpr double kRhoCrit = 2.77536627e11;  // 3 H0^2 / (8 pi G) in h^2 Msun Mpc^-3

constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct FofLayout {
    size_t status, sorted, start, cursor, sums, total;
};

FofLayout fof_layout(long long np) {
    FofLayout L;
    size_t o = 0;
    L.status = o;
    o += 256;
    L.sorted = o;
    o = align256(o + (size_t)np * sizeof(float4));
    L.start = o;
    o = align256(o + (size_t)(np + 1) * sizeof(int));
    L.cursor = o;
    o = align256(o + (size_t)np * sizeof(int));
    L.sums = o;
    o = align256(o + scan_sums_bytes(np + 1));
    L.total = o;
    return L;
}

template <class T>
T* at(void* ws, size_t off) {
    return reinterpret_cast<T*>(static_cast<char*>(ws) + off);
}

// position along one axis in units of the mean spacing, wrapped into [0, nq)
__device__ __forceinline__ float wrap_pos(float q, float d, float inv, float nqf) {
    float u = __fadd_rn(q, __fmul_rn(d, inv));
    u = __fsub_rn(u, __fmul_rn(nqf, floorf(__fdiv_rn(u, nqf))));
    if (u < 0.f) u = __fadd_rn(u, nqf);
    if (u >= nqf) u = __fsub_rn(u, nqf);
    return u;
}

// u of particle p and its cell; false (cell 0, u NaN) for non-finite input
__device__ __forceinline__ bool particle_pos(const float* __restrict__ d, long long np, int nq, float inv, long long p,
                                             float u[3], int* cell) {
    const unsigned nqu = (unsigned)nq, pu = (unsigned)p;
    const unsigned q[3] = {pu / (nqu * nqu), (pu / nqu) % nqu, pu % nqu};
    const float nqf = (float)nq;
    bool ok = true;
    int c = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = wrap_pos((float)q[a], d[a * np + p], inv, nqf);
        ok = ok && (u[a] >= 0.f && u[a] < nqf);  // false for NaN
        int ca = (int)u[a];
        if (ca > nq - 1) ca = nq - 1;
        c = c * nq + ca;
    }
    if (!ok) {
        u[0] = u[1] = u[2] = __int_as_float(0x7fc00000);
        c = 0;
    }
    *cell = c;
    return ok;
}

__global__ void k_fof_count(const float* __restrict__ d, long long np, int nq, float inv, int* count, int* status) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    float u[3];
    int c;
    if (!particle_pos(d, np, nq, inv, p, u, &c)) set_status(status, COLA_ENONFINITE);
    atomicAdd(count + c, 1);
}

__global__ void k_fof_scatter(const float* __restrict__ d, long long np, int nq, float inv, int* cursor,
                              float4* sorted) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    float u[3];
    int c;
    particle_pos(d, np, nq, inv, p, u, &c);
    const int slot = atomicAdd(cursor + c, 1);
    sorted[slot] = make_float4(u[0], u[1], u[2], __int_as_float((int)p));
}


// ---------------------------------------------------------------------------
// union-find over sorted slots; parent[x] <= x always holds
// ---------------------------------------------------------------------------
__device__ __forceinline__ int fof_find(int* parent, int x, int* status, int cap) {
    for (int it = 0; it < cap; ++it) {
        const int px = __ldcg(parent + x);
        if (px == x) return x;
        const int gp = __ldcg(parent + px);
        if (gp != px) parent[x] = gp;  // path halving: gp is an ancestor of x, so gp <= px
        x = gp;
    }
    set_status(status, COLA_ETIMEOUT);
    return x;
}

// unites the trees of a and b; returns their root
__device__ __forceinline__ int fof_unite(int* parent, int a, int b, int* status, int cap) {
    for (int it = 0; it < cap; ++it) {
        a = fof_find(parent, a, status, cap);
        b = fof_find(parent, b, status, cap);
        if (a == b) return a;
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(parent + b, b, a) == b) return a;  // the larger root hooks under the smaller
    }
    set_status(status, COLA_ETIMEOUT);
    return a;
}

__device__ __forceinline__ float min_image(float x, float nqf, float half) {
    if (x > half) x = __fsub_rn(x, nqf);
    if (x < -half) x = __fadd_rn(x, nqf);
    return x;
}

__device__ __forceinline__ int wrap_cell(int c, int nq) { return c < 0 ? c + nq : (c >= nq ? c - nq : c); }

// the friendship test; the same for (a, o) and (o, a): negation is exact
__device__ __forceinline__ bool is_friend(const float4& a, const float4& o, float nqf, float half, float b2) {
    const float dx = min_image(__fsub_rn(a.x, o.x), nqf, half);
    const float dy = min_image(__fsub_rn(a.y, o.y), nqf, half);
    const float dz = min_image(__fsub_rn(a.z, o.z), nqf, half);
    const float r2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
    return r2 <= b2;
}

// Calls f(i) for every friend i < k of slot k, in ascending order except across
// the box's faces, until f returns true.  The candidates are the slots below k
// in the neighbour cells that the position reaches within `reach`; any superset
// also works (the distance test decides).  Cells along z are consecutive, so a
// neighbour row (x, y) is one range of slots, and rows of later cells hold no
// slot below k.
template <class F>
__device__ __forceinline__ void smaller_friends(const float4* __restrict__ sorted, const int* __restrict__ start,
                                                int k, const float4& a, int nq, float b2, float reach, const F& f) {
    const float nqf = (float)nq, half = (float)(nq / 2.0);
    const float pos[3] = {a.x, a.y, a.z};
    int c[3], lo[3], hi[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        c[e] = (int)pos[e];
        if (c[e] > nq - 1) c[e] = nq - 1;
        const float t = pos[e] - (float)c[e];  // exact
        lo[e] = t <= reach ? -1 : 0;
        hi[e] = 1.f - t <= reach ? 1 : 0;
    }
    const int own = (c[0] * nq + c[1]) * nq + c[2];
    const int z0 = c[2] + lo[2], z1 = c[2] + hi[2];
    auto range = [&](int row, int za, int zb) -> bool {
        if (row + za > own) return false;
        const int j1 = min(__ldg(start + row + zb + 1), k);
        for (int i = __ldg(start + row + za); i < j1; ++i)
            if (is_friend(a, __ldg(sorted + i), nqf, half, b2) && f(i)) return true;
        return false;
    };
    for (int ox = lo[0]; ox <= hi[0]; ++ox) {
        const int cx = wrap_cell(c[0] + ox, nq);
        for (int oy = lo[1]; oy <= hi[1]; ++oy) {
            const int row = (cx * nq + wrap_cell(c[1] + oy, nq)) * nq;
            if (z1 >= nq && range(row, 0, 0)) return;
            if (range(row, max(z0, 0), min(z1, nq - 1))) return;
            if (z0 < 0 && range(row, nq - 1, nq - 1)) return;
        }
    }
}

__device__ __forceinline__ bool finite_pos(const float4& a) { return a.x == a.x && a.y == a.y && a.z == a.z; }

// parent = the first friend below, or itself (non-finite input links to nothing);
// part[k] = the particle of slot k, so that k_fof_roots need not read the records again
__global__ void __launch_bounds__(256) k_fof_hook(const float4* __restrict__ sorted, const int* __restrict__ start,
                                                  int np, int nq, float b2, float reach, int* __restrict__ parent,
                                                  int* __restrict__ part) {
    const unsigned k = blockIdx.x * 256u + threadIdx.x;
    if (k >= (unsigned)np) return;
    const float4 a = __ldg(sorted + k);
    int first = (int)k;
    if (finite_pos(a))
        smaller_friends(sorted, start, (int)k, a, nq, b2, reach, [&](int i) {
            first = i;
            return true;
        });
    parent[k] = first;
    part[k] = __float_as_int(a.w);
}

// every parent becomes (at least) the root its tree has now; four slots per
// thread (np is a multiple of eight), as most parents are roots already in a
// hardly clustered state and the pass is then one read of the parents
__global__ void __launch_bounds__(256) k_fof_compress(int* parent, int np, int* status, int cap) {
    const unsigned k0 = (blockIdx.x * 256u + threadIdx.x) * 4u;
    if (k0 >= (unsigned)np) return;
    const int4 v = __ldcg(reinterpret_cast<const int4*>(parent + k0));
    const int first[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int k = (int)k0 + q;
        int x = first[q];
        if (x == k) continue;
        int it = 1;
        for (; it < cap; ++it) {
            const int px = __ldcg(parent + x);
            if (px == x) break;
            x = px;
        }
        if (it >= cap)
            set_status(status, COLA_ETIMEOUT);
        else if (x != first[q])
            parent[k] = x;
    }
}

__global__ void __launch_bounds__(256) k_fof_link(const float4* __restrict__ sorted, const int* __restrict__ start,
                                                  int np, int nq, float b2, float reach, int* parent, int* status,
                                                  int cap) {
    const unsigned k = blockIdx.x * 256u + threadIdx.x;
    if (k >= (unsigned)np) return;
    int root = __ldcg(parent + k);
    if (root == (int)k) return;  // no friend below it
    const float4 a = __ldg(sorted + k);
    smaller_friends(sorted, start, (int)k, a, nq, b2, reach, [&](int i) {
        const int pi = __ldcg(parent + i);
        if (pi != root) root = fof_unite(parent, root, pi, status, cap);
        return false;
    });
}

// root of every slot; least[k] = the slot's particle, to be lowered by k_fof_least
__global__ void __launch_bounds__(256) k_fof_roots(const int* __restrict__ part, int* parent, int np,
                                                   int* __restrict__ least, int* status, int cap) {
    const unsigned k = blockIdx.x * 256u + threadIdx.x;
    if (k >= (unsigned)np) return;
    least[k] = __ldg(part + k);
    int x = (int)k;
    for (int it = 0; it < cap; ++it) {
        const int px = __ldcg(parent + x);
        if (px == x) {
            if (x != (int)k) parent[k] = x;
            return;
        }
        x = px;
    }
    set_status(status, COLA_ETIMEOUT);
}

// least[root] = the smallest particle index of the group; a warp of one group takes
// one atomic.  least[k] is the particle of slot k unless k is a root, whose own index
// is in least[root] already, so neither needs the sorted records.
__global__ void __launch_bounds__(256) k_fof_least(const int* __restrict__ parent, int np, int* least) {
    const unsigned k = blockIdx.x * 256u + threadIdx.x;
    const bool in = k < (unsigned)np;
    const int root = in ? __ldg(parent + k) : -1;
    const bool adds = in && root != (int)k;
    const int p = adds ? __ldcg(least + k) : 0x7fffffff;
    const unsigned full = 0xffffffffu;
    if (__all_sync(full, root == __shfl_sync(full, root, 0))) {
        const int m = __reduce_min_sync(full, p);
        if ((threadIdx.x & 31) == 0 && root >= 0) atomicMin(least + root, m);
    } else if (adds) {
        atomicMin(least + root, p);
    }
}

__global__ void __launch_bounds__(256) k_fof_label(const float4* __restrict__ sorted, const int* __restrict__ parent,
                                                   const int* __restrict__ least, int np, int* __restrict__ group) {
    const unsigned k = blockIdx.x * 256u + threadIdx.x;
    if (k < (unsigned)np) group[__float_as_int(__ldg(&sorted[k].w))] = __ldg(least + __ldg(parent + k));
}

__global__ void k_fof_sizes(const int* __restrict__ group, long long np, int* size) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < np) atomicAdd(size + group[p], 1);
}

__global__ void k_fof_flags(const int* __restrict__ group, const int* __restrict__ size, long long np, int nmin,
                            int* flag) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < np) flag[p] = (group[p] == (int)p && size[p] >= nmin) ? 1 : 0;
}

// off: exclusive scan of the flags (np + 1 entries, off[np] = halo count)
__global__ void k_fof_emit(const int* __restrict__ off, const int* __restrict__ size, long long np, int* halo_root,
                           int* halo_size, long long* n_halos) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p == 0) *n_halos = off[np];
    if (p >= np) return;
    const int o = off[p];
    if (off[p + 1] != o) {
        halo_root[o] = (int)p;
        halo_size[o] = size[p];
    }
}

__global__ void k_mass_function(const int* __restrict__ halo_size, const long long* __restrict__ n_halos,
                                long long max_halos, double m_p, double lo, double dlog, int nbins,
                                unsigned long long* counts) {
    const long long n = min(*n_halos, max_halos);
    for (long long h = (long long)blockIdx.x * blockDim.x + threadIdx.x; h < n; h += (long long)gridDim.x * blockDim.x) {
        const double N = (double)halo_size[h];
        const double lm = log10(m_p * N * (1.0 - pow(N, -0.6)));
        const double t = floor((lm - lo) / dlog);
        if (t >= 0.0 && t < (double)nbins) atomicAdd(counts + (int)t, 1ull);
    }
}

unsigned blocks_for(long long n, int t) { return (unsigned)((n + t - 1) / t); }

int check_fof_args(const cola_config* cfg, long long* np) {
    size_t ignored = 0;
    if (!cfg) return COLA_EINVAL;
    if (int rc = cola_workspace_size(cfg, &ignored)) return rc;
    const long long n = (long long)cfg->nq * cfg->nq * cfg->nq;
    if (n + 1 > 0x7fffffffll) return COLA_EUNSUPPORTED_SIZE;  // int32 particle indices and scans
    *np = n;
    return COLA_OK;
}

int read_status(const int* dev_status, cudaStream_t s) {
    int h = 0;
    if (cudaMemcpyAsync(&h, dev_status, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess) return COLA_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return COLA_ECUDA;
    return h;
}

}  // namespace
}  // namespace cola

extern "C" {

int cola_fof_set_retry_cap(int32_t cap) {
    if (cap < 0 || cap > (1 << 30)) return COLA_EINVAL;
    cola::g_union_cap = cap ? cap : cola::kUnionCap;
    return COLA_OK;
}

int cola_fof_workspace_size(const cola_config* cfg, size_t* bytes) {
    long long np = 0;
    if (!bytes) return COLA_EINVAL;
    if (int rc = cola::check_fof_args(cfg, &np)) return rc;
    *bytes = cola::fof_layout(np).total;
    return COLA_OK;
}

int cola_fof(const cola_config* cfg, const cola_state* st, double b, int32_t* group, void* fws, size_t fws_bytes,
             void* stream) {
    using namespace cola;
    long long np = 0;
    if (int rc = check_fof_args(cfg, &np)) return rc;
    if (!st || !st->d || !group || !fws || !(b > 0.0 && b < 0.5)) return COLA_EINVAL;
    const FofLayout L = fof_layout(np);
    if (fws_bytes < L.total) return COLA_EWORKSPACE;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int* status = at<int>(fws, L.status);
    int* start = at<int>(fws, L.start);
    int* cursor = at<int>(fws, L.cursor);
    float4* sorted = at<float4>(fws, L.sorted);
    const float inv = (float)((double)cfg->nq / cfg->box);
    const int T = 256;
    const unsigned nb = blocks_for(np, T);
    if (cudaMemsetAsync(status, 0, sizeof(int), s) != cudaSuccess ||
        cudaMemsetAsync(start, 0, (size_t)(np + 1) * sizeof(int), s) != cudaSuccess)
        return COLA_ECUDA;
    k_fof_count<<<nb, T, 0, s>>>(st->d, np, cfg->nq, inv, start, status);
    if (int rc = check_launch()) return rc;
    if (int rc = exclusive_scan(start, np, at<int>(fws, L.sums), s)) return rc;
    if (cudaMemcpyAsync(cursor, start, (size_t)np * sizeof(int), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return COLA_ECUDA;
    k_fof_scatter<<<nb, T, 0, s>>>(st->d, np, cfg->nq, inv, cursor, sorted);
    // the cursor array becomes the parents, the cell offsets (once the pairs are linked) the groups' least members
    int* parent = cursor;
    int* least = start;
    const int n = (int)np, nq = cfg->nq, cap = g_union_cap;
    const float b2 = (float)(b * b), reach = (float)b + 0.01f;  // wider than b by far more than FP32 rounding
    k_fof_hook<<<nb, T, 0, s>>>(sorted, start, n, nq, b2, reach, parent, group);  // (group: scratch until the labels)
    k_fof_compress<<<blocks_for(np, 4 * T), T, 0, s>>>(parent, n, status, cap);
    k_fof_link<<<nb, T, 0, s>>>(sorted, start, n, nq, b2, reach, parent, status, cap);
    k_fof_roots<<<nb, T, 0, s>>>(group, parent, n, least, status, cap);
    k_fof_least<<<nb, T, 0, s>>>(parent, n, least);
    k_fof_label<<<nb, T, 0, s>>>(sorted, parent, least, n, group);
    if (int rc = check_launch()) return rc;
    return read_status(status, s);
}

int cola_fof_halos(const cola_config* cfg, const int32_t* group, int32_t min_members, int32_t* halo_root,
                   int32_t* halo_size, int64_t* n_halos, void* fws, size_t fws_bytes, void* stream) {
    using namespace cola;
    long long np = 0;
    if (int rc = check_fof_args(cfg, &np)) return rc;
    if (!group || !halo_root || !halo_size || !n_halos || !fws || min_members < 1) return COLA_EINVAL;
    const FofLayout L = fof_layout(np);
    if (fws_bytes < L.total) return COLA_EWORKSPACE;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int* size = at<int>(fws, L.cursor);
    int* off = at<int>(fws, L.start);
    const int T = 256;
    const unsigned nb = blocks_for(np, T);
    if (cudaMemsetAsync(size, 0, (size_t)np * sizeof(int), s) != cudaSuccess) return COLA_ECUDA;
    k_fof_sizes<<<nb, T, 0, s>>>(group, np, size);
    k_fof_flags<<<nb, T, 0, s>>>(group, size, np, min_members, off);
    if (int rc = check_launch()) return rc;
    if (int rc = exclusive_scan(off, np, at<int>(fws, L.sums), s)) return rc;
    k_fof_emit<<<nb, T, 0, s>>>(off, size, np, halo_root, halo_size, reinterpret_cast<long long*>(n_halos));
    return check_launch();
}

int cola_mass_function(const cola_config* cfg, const int32_t* halo_size, const int64_t* n_halos, int64_t max_halos,
                       double log10m_lo, double dlog10m, int32_t nbins, int64_t* counts, void* stream) {
    using namespace cola;
    long long np = 0;
    if (int rc = check_fof_args(cfg, &np)) return rc;
    if (!halo_size || !n_halos || !counts || max_halos < 0 || nbins < 1 || !(dlog10m > 0.0)) return COLA_EINVAL;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(counts, 0, (size_t)nbins * sizeof(int64_t), s) != cudaSuccess) return COLA_ECUDA;
    if (max_halos == 0) return COLA_OK;
    const double m_p = kRhoCrit * cfg->cosmo.omega_m * std::pow(cfg->box / cfg->nq, 3);
    const int T = 256;
    long long blocks = (max_halos + T - 1) / T;
    if (blocks > 4096) blocks = 4096;
    k_mass_function<<<(unsigned)blocks, T, 0, s>>>(halo_size, reinterpret_cast<const long long*>(n_halos), max_halos,
                                                   m_p, log10m_lo, dlog10m, nbins,
                                                   reinterpret_cast<unsigned long long*>(counts));
    return check_launch();
}

}  // extern "C"
