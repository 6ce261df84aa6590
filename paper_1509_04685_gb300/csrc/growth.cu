// FP64 time tables: growth factors and the COLA kick/drift integrals (Eqs. 2-3).
//
// The growth ODEs in y = ln a for D1 = a u and D2 = a^2 w (Sec. 2.2's 2LPT
// growth factors; the same equations as D1'' + (2 + dlnE/dy) D1' = 3/2 Om(a) D1
// and D2'' + (2 + dlnE/dy) D2' = 3/2 Om(a) (D2 - D1^2)), started on the
// Einstein-de Sitter modes (D1 = a, D2 = -3/7 a^2) at a = 1e-5 and normalised to
// D1(1) = 1.  u and w are constant in the matter era, so RK4 in these variables
// is accurate with far fewer steps than in D1, D2 themselves.  The integrals
// K = int dy / E and Dr = int dy a^kn / (a^2 E) go along (kn = 0: the standard
// drift; kn = n_LPT: the modified drift's integral).
//
// One RK4 step is a map that does not depend on the state it is applied to:
// (u, u') goes through a 2 x 2 matrix, (w, w') through another plus a term
// quadratic in (u, u') (the source -3/2 Om u^2 at the four stages), K and Dr get
// constants added.  Such maps compose to maps of the same form, so a warp
// takes up to 32 steps at once, one per lane, and reduces them in order; the
// chain that is left is one map per time node.  The steps, the stages and the
// formulas are those of the serial integration, one thread walking ~1400 steps
// of four right-hand sides: 21.4 ms per table (40 nodes) and 18.8 ms per
// snapshot that way, 0.15 ms and 61 us this way (two launches each).  What bounds
// it now is FP64 issue (about two lanes per clock and SM), hence one warp per
// block, spread over the SMs.
#include <cmath>

#include "cosmo.cuh"

namespace cola {

namespace {

// (u, u') -> m (u, u');  (w, w') -> a (w, w') + c (u^2, u u', u'^2)
struct GrowthMap {
    double m[4], a[4], c[6];
};
constexpr int kMapDoubles = 14;

__device__ __forceinline__ void map_identity(GrowthMap& g) {
#pragma unroll
    for (int i = 0; i < 4; ++i) g.m[i] = g.a[i] = (i == 0 || i == 3) ? 1.0 : 0.0;
#pragma unroll
    for (int i = 0; i < 6; ++i) g.c[i] = 0.0;
}

// g after f: x -> g(f(x))
__device__ __forceinline__ GrowthMap map_after(const GrowthMap& g, const GrowthMap& f) {
    GrowthMap r;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            r.m[2 * i + j] = g.m[2 * i] * f.m[j] + g.m[2 * i + 1] * f.m[2 + j];
            r.a[2 * i + j] = g.a[2 * i] * f.a[j] + g.a[2 * i + 1] * f.a[2 + j];
        }
    // quadratic monomials of f's output in those of its input
    const double p = f.m[0], q = f.m[1], s = f.m[2], t = f.m[3];
    const double sq[3][3] = {{p * p, 2.0 * p * q, q * q}, {p * s, p * t + q * s, q * t}, {s * s, 2.0 * s * t, t * t}};
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            r.c[3 * i + j] = g.a[2 * i] * f.c[j] + g.a[2 * i + 1] * f.c[3 + j] + g.c[3 * i] * sq[0][j] +
                             g.c[3 * i + 1] * sq[1][j] + g.c[3 * i + 2] * sq[2][j];
    return r;
}

// the map applied to the state s = (u, u', w, w')
__device__ __forceinline__ void map_apply(const double* g, double s[4]) {
    const double uu = s[0] * s[0], uv = s[0] * s[1], vv = s[1] * s[1];
    const double u = g[0] * s[0] + g[1] * s[1], v = g[2] * s[0] + g[3] * s[1];
    const double w = g[4] * s[2] + g[5] * s[3] + (g[8] * uu + g[9] * uv + g[10] * vv);
    const double x = g[6] * s[2] + g[7] * s[3] + (g[11] * uu + g[12] * uv + g[13] * vv);
    s[0] = u;
    s[1] = v;
    s[2] = w;
    s[3] = x;
}

// coefficients of the ODEs at y: u'' = -p u' - q u, w'' = -(p + 2) w' - r w - so u^2
struct GrowthCoef {
    double p, q, r, so, ik, idr;  // ik, idr: integrands of K and Dr
};

__device__ GrowthCoef growth_coef(double y, const CosmoD& c, double kn) {
    const double a = exp(y);
    const double a2 = a * a, a3 = a2 * a;
    const double E2 = c.om / a3 + c.ok / a2 + c.ol;
    const double E = sqrt(E2);
    const double oma = c.om / a3 / E2;
    const double fr = 2.0 + (-3.0 * c.om / a3 - 2.0 * c.ok / a2) / (2.0 * E2);
    GrowthCoef g;
    g.p = 2.0 + fr;
    g.q = 1.0 + fr - 1.5 * oma;
    g.r = 4.0 + 2.0 * fr - 1.5 * oma;
    g.so = 1.5 * oma;
    g.ik = 1.0 / E;
    g.idr = (kn != 0.0 ? exp(kn * y) : 1.0) / (a2 * E);
    return g;
}

__device__ __forceinline__ void growth_rhs(const GrowthCoef& g, const double* s, double* ds) {
    ds[0] = s[1];
    ds[1] = -g.p * s[1] - g.q * s[0];
    ds[2] = s[3];
    ds[3] = -(g.p + 2.0) * s[3] - g.r * s[2] - g.so * s[0] * s[0];
}

// one RK4 step of length h with the coefficients at its start, middle and end
__device__ void rk4_step(const GrowthCoef& g0, const GrowthCoef& g1, const GrowthCoef& g2, double h, double* s) {
    double k1[4], k2[4], k3[4], k4[4], t[4];
    growth_rhs(g0, s, k1);
#pragma unroll
    for (int q = 0; q < 4; ++q) t[q] = s[q] + 0.5 * h * k1[q];
    growth_rhs(g1, t, k2);
#pragma unroll
    for (int q = 0; q < 4; ++q) t[q] = s[q] + 0.5 * h * k2[q];
    growth_rhs(g1, t, k3);
#pragma unroll
    for (int q = 0; q < 4; ++q) t[q] = s[q] + h * k3[q];
    growth_rhs(g2, t, k4);
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] += h / 6.0 * (k1[q] + 2.0 * k2[q] + 2.0 * k3[q] + k4[q]);
}

// the step as a map: its action on basis states
__device__ GrowthMap step_map(const GrowthCoef& g0, const GrowthCoef& g1, const GrowthCoef& g2, double h) {
    GrowthMap r;
    double e[5][4] = {{1, 0, 0, 0}, {0, 1, 0, 0}, {1, 1, 0, 0}, {0, 0, 1, 0}, {0, 0, 0, 1}};
#pragma unroll
    for (int b = 0; b < 5; ++b) rk4_step(g0, g1, g2, h, e[b]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        r.m[2 * i] = e[0][i];
        r.m[2 * i + 1] = e[1][i];
        r.a[2 * i] = e[3][2 + i];
        r.a[2 * i + 1] = e[4][2 + i];
        r.c[3 * i] = e[0][2 + i];
        r.c[3 * i + 2] = e[1][2 + i];
        r.c[3 * i + 1] = e[2][2 + i] - e[0][2 + i] - e[1][2 + i];
    }
    return r;
}

// steps in y: from the start to the first output, and between outputs
constexpr double kHEarly = 1.0 / 64.0;
constexpr double kHSeg = 1.0 / 256.0;
constexpr double kAEarly = 1e-5;
constexpr double kNLpt = -2.5;  // n_LPT of the modified kick and drift (Tassev et al. 2013)

// n equal steps from y0 to y1
struct Span {
    double y0, y1;
    int n;
};
__host__ __device__ inline Span make_span(double y0, double y1, double hmax) {
    const double d = y1 - y0;
    return Span{y0, y1, d > 0.0 ? (int)ceil(d / hmax) : 0};
}

// Steps [lo, hi) of the spans s0, s1 taken one after the other (s1 may be
// empty), composed by the warp in order: every lane returns the map of its own
// and the later lanes' steps, lane 0 the whole one; k0, k1 and dr (lane 0) are
// the integrals K over s0's and s1's steps and Dr over both.
__device__ GrowthMap warp_map(const Span& s0, const Span& s1, int lo, int hi, const CosmoD& c, double kn, double* k0,
                              double* k1, double* dr) {
    const int lane = threadIdx.x & 31, n = hi - lo, per = (n + 31) / 32;
    GrowthMap r;
    map_identity(r);
    double a0 = 0.0, a1 = 0.0, ad = 0.0;
    const int b = lo + lane * per, e = b + per < hi ? b + per : hi;
    for (int i = b; i < e; ++i) {
        const bool second = i >= s0.n;
        const Span& s = second ? s1 : s0;
        const int q = second ? i - s0.n : i;
        const double h = (s.y1 - s.y0) / s.n;
        const double y = s.y0 + q * h;
        const GrowthCoef g0 = growth_coef(y, c, kn), g1 = growth_coef(y + 0.5 * h, c, kn),
                         g2 = growth_coef(q + 1 == s.n ? s.y1 : y + h, c, kn);
        const GrowthMap f = step_map(g0, g1, g2, h);
        r = i == b ? f : map_after(f, r);
        const double dk = h / 6.0 * (g0.ik + 4.0 * g1.ik + g2.ik);
        a0 += second ? 0.0 : dk;
        a1 += second ? dk : 0.0;
        ad += h / 6.0 * (g0.idr + 4.0 * g1.idr + g2.idr);
    }
    const unsigned full = 0xffffffffu;
    for (int o = 1; o < 32; o <<= 1) {
        GrowthMap f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f.m[i] = __shfl_down_sync(full, r.m[i], o);
            f.a[i] = __shfl_down_sync(full, r.a[i], o);
        }
#pragma unroll
        for (int i = 0; i < 6; ++i) f.c[i] = __shfl_down_sync(full, r.c[i], o);
        const double b0 = __shfl_down_sync(full, a0, o), b1 = __shfl_down_sync(full, a1, o),
                     bd = __shfl_down_sync(full, ad, o);
        if ((lane & (2 * o - 1)) == 0 && lane + o < 32 && (lane + o) * per < n) {
            r = map_after(f, r);
            a0 += b0;
            a1 += b1;
            ad += bd;
        }
    }
    *k0 = a0;
    *k1 = a1;
    *dr = ad;
    return r;
}

__device__ __forceinline__ void store_map(double* o, const GrowthMap& g) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        o[i] = g.m[i];
        o[4 + i] = g.a[i];
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) o[8 + i] = g.c[i];
}

// a span is cut into chunks of 32 steps, at most kMaxChunks of them
constexpr int kMaxChunks = 64;
__host__ __device__ inline int chunks_of(const Span& s) {
    const int c = (s.n + 31) / 32;
    return c < kMaxChunks ? c : kMaxChunks;
}
// steps [lo, hi) of chunk i of nc
__device__ __forceinline__ void chunk_range(const Span& s, int i, int nc, int* lo, int* hi) {
    const int per = (s.n + nc - 1) / nc;
    *lo = i * per < s.n ? i * per : s.n;
    *hi = *lo + per < s.n ? *lo + per : s.n;
}

// the Einstein-de Sitter modes at a = kAEarly
__device__ __forceinline__ void growth_init(double s[4]) {
    s[0] = 1.0;
    s[1] = 0.0;
    s[2] = -3.0 / 7.0;
    s[3] = 0.0;
}

__host__ __device__ inline double node_a(int j, int n, double ai, double af, int sampling, double p) {
    const double t = (double)j / (double)(n - 1);
    if (sampling == COLA_SAMPLING_LOG) return exp(log(ai) + t * (log(af) - log(ai)));
    if (sampling == COLA_SAMPLING_POW) return pow(pow(ai, p) + t * (pow(af, p) - pow(ai, p)), 1.0 / p);
    return ai + t * (af - ai);
}

struct Nodes {
    int n;
    double ai, af;
    int sampling;
    double sp;
    __device__ double a(int j) const { return node_a(j, n, ai, af, sampling, sp); }
};

// Scratch of the growth kernels (kHdrGrowth, stream-ordered like the rest of
// the workspace): the quadratic parts of the interval maps, then the maps of
// the chunks of up to four spans.
constexpr size_t kScrChunks = (size_t)kMaxSteps * 6;  // in doubles
static_assert((kScrChunks + 4 * kMaxChunks * kMapDoubles + 4 * kMaxChunks) * 8 <= kHdrBytes - kHdrGrowth,
              "growth scratch must fit in the header");

// One warp per block.  Blocks 0 .. n-2: interval j, [a_j, mid] and [mid, a_{j+1}]
// (arithmetic midpoint): row j of the table takes the linear parts of its map
// and K(a_j, mid), K(mid, a_{j+1}), Dr(a_j, a_{j+1}), the scratch the rest.
// The next ne blocks: the chunks of the early span; the last nt: those of the
// span from the last node to a = 1.
__global__ void __launch_bounds__(32) k_table_maps(double* tab, double* scr, Nodes nd, CosmoD c, double kn, Span early,
                                                   int ne, Span tail, int nt) {
    const int j = blockIdx.x;
    double k0, k1, dr;
    if (j < nd.n - 1) {
        const double aj = nd.a(j), an = nd.a(j + 1);
        const double ym = log(0.5 * (aj + an));
        const Span s0 = make_span(log(aj), ym, kHSeg), s1 = make_span(ym, log(an), kHSeg);
        const GrowthMap g = warp_map(s0, s1, 0, s0.n + s1.n, c, kn, &k0, &k1, &dr);
        if (threadIdx.x) return;
        double* r = tab + (size_t)j * kTableCols;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            r[i] = g.m[i];
            r[4 + i] = g.a[i];
        }
        r[8] = k0;
        r[9] = k1;
        r[10] = dr;
#pragma unroll
        for (int i = 0; i < 6; ++i) scr[6 * (size_t)j + i] = g.c[i];
        return;
    }
    const int q = j - (nd.n - 1);
    const bool first = q < ne;
    const Span& s = first ? early : tail;
    int lo, hi;
    chunk_range(s, first ? q : q - ne, first ? ne : nt, &lo, &hi);
    const GrowthMap g = warp_map(s, Span{0.0, 0.0, 0}, lo, hi, c, 0.0, &k0, &k1, &dr);
    if (threadIdx.x == 0) store_map(scr + kScrChunks + (size_t)q * kMapDoubles, g);
}

// Table row j (12 doubles): a, green, c1, c2, kick, drift, dD1, dD2, D1, D2, dD1/da, dD2/da.
// kn = 0: the standard kick and drift factors, kick = int da / (a E) over
// [a_{j-1/2}, a_{j+1/2}] and drift = int da / (a^3 E) over [a_j, a_{j+1}].
// kn = n_LPT: the modified factors of Tassev et al. (2013), the residual
// momentum varying as a power a^n of the scale factor about the reference time:
// kick = (a_{j+1/2}^n - a_{j-1/2}^n) / (n a_j^n E(a_j)) (force at the node),
// drift = a_{j+1/2}^-n int da a^n / (a^3 E) over [a_j, a_{j+1}] (momentum at the midpoint).
// One block: thread 0 walks the chunk and interval maps (staged through
// shared memory, 64 at a time) and leaves the state of every node in its row;
// then the rows are finished in parallel.
constexpr int kRowThreads = 256;
constexpr int kMapTile = 64;
__global__ void __launch_bounds__(kRowThreads) k_table_rows(double* tab, const double* scr, Nodes nd, CosmoD c,
                                                            int pm_only, double kn, int ne, int nt) {
    __shared__ double maps[kMapTile * kMapDoubles], st[kMapTile][4], norm, k_before;
    const int tid = threadIdx.x, n = nd.n;
    double s[4];
    growth_init(s);
    // chunk maps [q0, q1) applied in order
    auto walk = [&](int q0, int q1) {
        for (int q = q0; q < q1; q += kMapTile) {
            const int m = q1 - q < kMapTile ? q1 - q : kMapTile;
            __syncthreads();
            for (int e = tid; e < m * kMapDoubles; e += kRowThreads)
                maps[e] = scr[kScrChunks + (size_t)q * kMapDoubles + e];
            __syncthreads();
            if (tid == 0)
                for (int i = 0; i < m; ++i) map_apply(maps + i * kMapDoubles, s);
        }
    };
    walk(0, ne);
    for (int j0 = 0; j0 < n; j0 += kMapTile) {
        const int m = n - j0 < kMapTile ? n - j0 : kMapTile;
        __syncthreads();
        for (int e = tid; e < m * kMapDoubles; e += kRowThreads) {
            const int i = e / kMapDoubles, q = e - i * kMapDoubles;
            if (j0 + i < n - 1)
                maps[e] = q < 8 ? tab[(size_t)(j0 + i) * kTableCols + q] : scr[6 * (size_t)(j0 + i) + q - 8];
        }
        __syncthreads();
        if (tid == 0)
            for (int i = 0; i < m; ++i) {
#pragma unroll
                for (int q = 0; q < 4; ++q) st[i][q] = s[q];
                if (j0 + i < n - 1) map_apply(maps + i * kMapDoubles, s);
            }
        __syncthreads();
        for (int e = tid; e < 4 * m; e += kRowThreads) tab[(size_t)(j0 + e / 4) * kTableCols + e % 4] = st[e / 4][e % 4];
    }
    walk(ne, ne + nt);
    if (tid == 0) {
        norm = s[0];  // D1(1) = u at a = 1
        k_before = 0.0;
    }
    __syncthreads();
    const double nrm = norm;
    for (int j0 = 0; j0 < n; j0 += kRowThreads) {
        const int j = j0 + tid;
        double o[kTableCols], k_mine = 0.0;
        if (j < n) {
            const double* r = tab + (size_t)j * kTableCols;
            const bool last = j + 1 == n;
            const double aj = nd.a(j), an = last ? aj : nd.a(j + 1);
            const double D1 = aj * r[0] / nrm, D2 = aj * aj * r[2] / (nrm * nrm);
            const double green = 1.5 * c.om / aj;
            const double k_prev = j == j0 ? k_before : r[9 - kTableCols];  // K(mid_{j-1}, a_j)
            o[0] = aj;
            o[1] = green;
            o[2] = green * D1;
            o[3] = green * (D2 - D1 * D1);
            o[4] = k_prev + (last ? 0.0 : r[8]);
            o[5] = last ? 0.0 : r[10];
            o[6] = o[7] = 0.0;
            if (!last) {
                const double* q = r + kTableCols;
                o[6] = an * q[0] / nrm - D1;
                o[7] = an * an * q[2] / (nrm * nrm) - D2;
                k_mine = r[9];
            }
            o[8] = D1;
            o[9] = D2;
            o[10] = (r[0] + r[1]) / nrm;
            o[11] = aj * (2.0 * r[2] + r[3]) / (nrm * nrm);
            if (pm_only) o[2] = o[3] = o[6] = o[7] = 0.0;
            if (kn != 0.0) {
                const double ajn = pow(aj, kn);
                double k = 0.0;
                if (j > 0) k += ajn - pow(0.5 * (nd.a(j - 1) + aj), kn);
                if (!last) {
                    const double amn = pow(0.5 * (aj + an), kn);
                    k += amn - ajn;
                    o[5] /= amn;
                }
                o[4] = k / (kn * ajn * E_of(aj, c));
            }
        }
        __syncthreads();  // every row of this batch has been read
        if (j < n) {
            double* r = tab + (size_t)j * kTableCols;
#pragma unroll
            for (int q = 0; q < kTableCols; ++q) r[q] = o[q];
        }
        if (tid == kRowThreads - 1) k_before = k_mine;
        __syncthreads();
    }
}

// Snapshot drift from a_node to a_out: the spans start -> lo, lo -> hi,
// lo -> 1 (start -> 1 if lo > 1) and start -> a_out, lo and hi the smaller and
// the larger of the two; one warp per chunk.
struct SnapSpans {
    Span s[4];
    int nc[4], first[5];
};
__global__ void __launch_bounds__(32) k_snapshot_maps(double* scr, SnapSpans sp, CosmoD c) {
    int w = 0;
    while (w < 3 && (int)blockIdx.x >= sp.first[w + 1]) ++w;
    int lo, hi;
    chunk_range(sp.s[w], blockIdx.x - sp.first[w], sp.nc[w], &lo, &hi);
    double k0, k1, dr;
    const GrowthMap g = warp_map(sp.s[w], Span{0.0, 0.0, 0}, lo, hi, c, 0.0, &k0, &k1, &dr);
    if (threadIdx.x) return;
    store_map(scr + kScrChunks + (size_t)blockIdx.x * kMapDoubles, g);
    scr[kScrChunks + 4 * kMaxChunks * kMapDoubles + blockIdx.x] = dr;
}

// (Dr(a_node, a_out), D1(a_out) - D1(a_node), D2(a_out) - D2(a_node)), then the
// redshift-space coefficients at a_out (1 / (a^2 E), a D1'(a), a D2'(a)).
__global__ void __launch_bounds__(256) k_snapshot(double* snap, const double* scr, SnapSpans sp, double a_node,
                                                  double a_out, CosmoD c, int pm_only) {
    extern __shared__ double maps[];
    const int total = sp.first[4];
    for (int e = threadIdx.x; e < total * kMapDoubles; e += blockDim.x) maps[e] = scr[kScrChunks + e];
    for (int e = threadIdx.x; e < total; e += blockDim.x)
        maps[total * kMapDoubles + e] = scr[kScrChunks + 4 * kMaxChunks * kMapDoubles + e];
    __shared__ double fin[3][4];
    __syncthreads();
    // warps 0, 1, 2 walk start -> lo -> hi, (start -> lo ->) 1 and start -> a_out at the same time
    const int w = threadIdx.x >> 5;
    const double lo = fmin(a_node, a_out), hi = fmax(a_node, a_out);
    if ((threadIdx.x & 31) == 0 && w < 3) {
        double s[4];
        growth_init(s);
        auto walk = [&](int q) {
            for (int i = sp.first[q]; i < sp.first[q + 1]; ++i) map_apply(maps + i * kMapDoubles, s);
        };
        if (w == 2) {
            walk(3);
        } else {
            if (w == 0 || lo <= 1.0) walk(0);
            if (w == 0) {
                fin[1][2] = lo * s[0];       // D1 at lo, raw
                fin[1][3] = lo * lo * s[2];  // D2
                walk(1);
            } else {
                walk(2);
            }
        }
        if (w == 1) {
            fin[1][0] = s[0];  // D1(1)
        } else {
            for (int q = 0; q < 4; ++q) fin[w][q] = s[q];
        }
    }
    __syncthreads();
    if (threadIdx.x) return;
    double dr = 0.0;
    for (int i = sp.first[1]; i < sp.first[2]; ++i) dr += maps[total * kMapDoubles + i];
    const double nrm = fin[1][0], sign = (a_out >= a_node) ? 1.0 : -1.0;
    snap[0] = sign * dr;
    snap[1] = pm_only ? 0.0 : sign * (hi * fin[0][0] - fin[1][2]) / nrm;
    snap[2] = pm_only ? 0.0 : sign * (hi * hi * fin[0][2] - fin[1][3]) / (nrm * nrm);
    // redshift-space shift along the line of sight at a_out: p_z / (a^2 E) with the full
    // momentum p = v + a^3 E (D1' Psi1 + D2' Psi2), i.e. v_z / (a^2 E) + a (D1' Psi1_z + D2' Psi2_z)
    const double dD1 = (fin[2][0] + fin[2][1]) / nrm;                        // dD1/da at a_out
    const double dD2 = a_out * (2.0 * fin[2][2] + fin[2][3]) / (nrm * nrm);  // dD2/da at a_out
    snap[3] = 1.0 / (a_out * a_out * E_of(a_out, c));
    snap[4] = pm_only ? 0.0 : a_out * dD1;
    snap[5] = pm_only ? 0.0 : a_out * dD2;
}

}  // namespace

int launch_tables(const cola_config* cfg, double* table, double* scratch, cudaStream_t s) {
    ProfScope ps(kKSetup, s);
    const CosmoD c = cosmo_of(cfg);
    const double kn = (cfg->flags & COLA_FLAG_MODIFIED_KDK) ? kNLpt : 0.0;
    const Nodes nd{cfg->n_steps, cfg->a_init, cfg->a_final, cfg->sampling, cfg->sampling_p};
    const double y_first = std::log(node_a(0, nd.n, nd.ai, nd.af, nd.sampling, nd.sp));
    const double y_last = std::log(node_a(nd.n - 1, nd.n, nd.ai, nd.af, nd.sampling, nd.sp));
    const Span early = make_span(std::log(kAEarly), y_first, kHEarly), tail = make_span(y_last, 0.0, kHSeg);
    const int ne = chunks_of(early), nt = chunks_of(tail);
    k_table_maps<<<nd.n - 1 + ne + nt, 32, 0, s>>>(table, scratch, nd, c, kn, early, ne, tail, nt);
    if (int rc = check_launch()) return rc;
    k_table_rows<<<1, kRowThreads, 0, s>>>(table, scratch, nd, c, (cfg->flags & COLA_FLAG_PM_ONLY) ? 1 : 0, kn, ne,
                                           nt);
    return check_launch();
}

int launch_snapshot_coeffs(const cola_config* cfg, double a_node, double a_out, double* snap, double* scratch,
                           cudaStream_t s) {
    ProfScope ps(kKSetup, s);
    const CosmoD c = cosmo_of(cfg);
    const double lo = std::fmin(a_node, a_out), hi = std::fmax(a_node, a_out), y0 = std::log(kAEarly);
    SnapSpans sp;
    sp.s[0] = make_span(y0, std::log(lo), kHEarly);
    sp.s[1] = make_span(std::log(lo), std::log(hi), kHSeg);
    sp.s[2] = lo > 1.0 ? make_span(y0, 0.0, kHEarly) : make_span(std::log(lo), 0.0, kHSeg);
    sp.s[3] = make_span(y0, std::log(a_out), kHEarly);
    sp.first[0] = 0;
    for (int q = 0; q < 4; ++q) {
        sp.nc[q] = chunks_of(sp.s[q]);
        sp.first[q + 1] = sp.first[q] + sp.nc[q];
    }
    const int total = sp.first[4];
    if (total > 0) {
        k_snapshot_maps<<<total, 32, 0, s>>>(scratch, sp, c);
        if (int rc = check_launch()) return rc;
    }
    const size_t smem = (size_t)total * (kMapDoubles + 1) * sizeof(double);  // at most 30 KB
    k_snapshot<<<1, 256, smem, s>>>(snap, scratch, sp, a_node, a_out, c, (cfg->flags & COLA_FLAG_PM_ONLY) ? 1 : 0);
    return check_launch();
}

}  // namespace cola
