// 2LPT initial conditions (Sec. 2.2: Gaussian field + 2LPT): Philox-4x32-10
// white noise (Salmon et al. 2011) with a 53-bit Box-Muller draw in FP64,
// the Eisenstein & Hu (1998) no-wiggle spectrum normalised to sigma8, and
// Psi1_k = i k delta_k/k^2, delta2 = sum_{i<j} phi_ii phi_jj - phi_ij^2,
// Psi2_k = -i k delta2_k / k^2 (Crocce et al. 2006 convention).
#include <cmath>

#include "cosmo.cuh"
#include "noise.cuh"

namespace cola {

// ---------------------------------------------------------------------------
// Eisenstein & Hu (1998) no-wiggle transfer function (their Eqs. 26, 28-31)
// ---------------------------------------------------------------------------
// what of it does not depend on k (host, once per set-up)
struct EhShape {
    double xs;          // 0.43 h s, s the sound horizon in Mpc
    double omh, al;     // Gamma_eff = omh (al + (1 - al) / (1 + (xs k)^4))
    double th2;         // (T_cmb / 2.7 K)^2
    double ns;
};

static EhShape eh_shape(const CosmoD& c) {
    const double omh2 = c.om * c.h * c.h, obh2 = c.ob * c.h * c.h, fb = c.ob / c.om, th = c.tcmb / 2.7;
    const double sh = 44.5 * std::log(9.83 / omh2) / std::sqrt(1.0 + 10.0 * std::pow(obh2, 0.75));
    const double al = 1.0 - 0.328 * std::log(431.0 * omh2) * fb + 0.38 * std::log(22.3 * omh2) * fb * fb;
    return EhShape{0.43 * c.h * sh, c.om * c.h, al, th * th, c.ns};
}

__device__ __forceinline__ double eh_nowiggle(double k, const EhShape& e) {
    const double x = e.xs * k;
    const double x2 = x * x;
    const double geff = e.omh * (e.al + (1.0 - e.al) / (1.0 + x2 * x2));
    const double q = k * e.th2 / geff;
    const double L0 = log(2.0 * 2.718281828459045235 + 1.8 * q);
    const double C0 = 14.2 + 731.0 / (1.0 + 62.5 * q);
    return L0 / (L0 + C0 * q * q);
}

__device__ double tophat(double x) {
    if (fabs(x) < 0.1) {
        const double x2 = x * x;
        return 1.0 - x2 / 10.0 + x2 * x2 / 280.0 - x2 * x2 * x2 / 15120.0;
    }
    double sn, cs;
    sincos(x, &sn, &cs);
    return 3.0 * (sn - x * cs) / (x * x * x);
}

// sigma8 normalisation: A = sigma8^2 / sigma_8,unnormalised^2 by composite
// Simpson in ln k over [1e-7, 250] h/Mpc with 2^17 intervals.  One point per
// thread, a partial sum per block; the blocks of k_ic_amp add the partials in
// one fixed order.  FP64-bound (about 250 FP64 operations a point): one block
// took 15.5 ms, all SMs take 67 us.
constexpr int kSigPoints = 1 << 17;
constexpr int kSigBlocks = kSigPoints / 256;

// sum over the block of one value per thread, in a fixed order; every thread receives it
__device__ __forceinline__ double block_sum256(double v, double* red) {
    red[threadIdx.x] = v;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    return red[0];
}

__global__ void __launch_bounds__(256) k_sigma8(double* part, EhShape e) {
    __shared__ double red[256];
    const double lo = log(1e-7), hi = log(2e3 / 8.0);
    const double h = (hi - lo) / kSigPoints;
    double acc = 0.0;
    const int last = (blockIdx.x == kSigBlocks - 1 && threadIdx.x == 255) ? 2 : 1;  // the last thread takes both ends
    for (int q = 0; q < last; ++q) {
        const int i = blockIdx.x * 256 + threadIdx.x + q;
        const double lk = lo + i * h;
        const double k = exp(lk);
        const double T = eh_nowiggle(k, e);
        const double W = tophat(8.0 * k);
        const double f = exp((3.0 + e.ns) * lk) * T * T * W * W;
        acc += ((i == 0 || i == kSigPoints) ? 1.0 : ((i & 1) ? 4.0 : 2.0)) * f;
    }
    const double t = block_sum256(acc, red);
    if (threadIdx.x == 0) part[blockIdx.x] = t * h / 3.0 / (2.0 * 3.14159265358979323846 * 3.14159265358979323846);
}

// amp[m] = sqrt(A P_unnormalised(kf sqrt(m)) / dq3), 1 <= m < nm: the factor of
// the noise modes with |n|^2 = m.  Modes share it (3 (nq/2 - 1)^2 values of m
// against nq^3 / 2 modes), so the FP64 transfer function is evaluated once per m
// instead of once per mode (256^3: 48 thousand evaluations instead of 8.4
// million: 32 us against 5.6 ms).
__global__ void __launch_bounds__(256) k_ic_amp(const double* __restrict__ part, float* __restrict__ amp, int nm,
                                                double s8, double kf, double dq3, EhShape e) {
    __shared__ double red[256];
    double v = 0.0;
    for (int i = threadIdx.x; i < kSigBlocks; i += 256) v += part[i];
    const double A = s8 * s8 / block_sum256(v, red);
    const int m = blockIdx.x * 256 + threadIdx.x + 1;
    if (m >= nm) return;
    const double kk = kf * sqrt((double)m);
    const double T = eh_nowiggle(kk, e);
    const double pk = A * pow(kk, e.ns) * T * T;
    amp[m] = (float)sqrt(pk / dq3);
}

// ---------------------------------------------------------------------------
// white-noise field (noise.cuh)
// ---------------------------------------------------------------------------
// noise of Lagrangian cell (i, j, k) -> real view of an nq mesh (row pitch 2P floats)
__global__ void k_noise(float* mesh, int nq, long long P2, unsigned long long seed) {
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n3 = (long long)nq * nq * nq;
    if (n >= n3) return;
    const uint4 w = philox4x32_10(make_uint4((unsigned)n, (unsigned)(n >> 32), 0u, 0u),
                                  make_uint2((unsigned)seed, (unsigned)(seed >> 32)));
    const long long row = n / nq;
    const int k = (int)(n - row * nq);
    mesh[row * P2 + k] = (float)box_muller(w);
}

// ---------------------------------------------------------------------------
// spectral operations on the nq half-complex mesh
// ---------------------------------------------------------------------------
__device__ __forceinline__ int signed_index(int i, int n) { return i < n / 2 ? i : i - n; }

// Spectral kernels: a block of 32 x 8 threads takes 8 consecutive rows (ix, iy)
// and walks along kz, so no thread divides per mode; each source value is read
// once for all the fields made from it (bound by the mesh traffic).
// k = 0 and every mode with an index on a Nyquist plane are set to zero.
constexpr int kSpecRows = 8;

struct SpecMode {
    int n[3];
    bool zero;
};
__device__ __forceinline__ SpecMode spec_mode(int ix, int iy, int kz, int nq) {
    const int half = nq / 2;
    SpecMode m;
    m.zero = ix == half || iy == half || kz == half || (ix == 0 && iy == 0 && kz == 0);
    m.n[0] = signed_index(ix, nq);
    m.n[1] = signed_index(iy, nq);
    m.n[2] = kz;
    return m;
}

// in place: delta_k = w_k amp(|n|^2)
__global__ void __launch_bounds__(32 * kSpecRows) k_ic_delta(float2* mesh, int nq, int P,
                                                             const float* __restrict__ amp) {
    const int row = blockIdx.x * kSpecRows + threadIdx.y;
    if (row >= nq * nq) return;
    const int ix = row / nq, iy = row - ix * nq;
    float2* r = mesh + (long long)row * P;
    for (int kz = threadIdx.x; kz <= nq / 2; kz += 32) {
        const SpecMode m = spec_mode(ix, iy, kz, nq);
        const int n2 = m.n[0] * m.n[0] + m.n[1] * m.n[1] + m.n[2] * m.n[2];
        r[kz] = m.zero ? make_float2(0.f, 0.f) : cscale(r[kz], __ldg(amp + n2));
    }
}

// dst[a] = sign i k_a src / k^2 norm, a = x, y, z (meshes `pitch` apart)
__global__ void __launch_bounds__(32 * kSpecRows) k_ic_grad(const float2* __restrict__ src, float2* __restrict__ dst,
                                                            long long pitch, int nq, int P, float kf, float norm,
                                                            float sign) {
    const int row = blockIdx.x * kSpecRows + threadIdx.y;
    if (row >= nq * nq) return;
    const int ix = row / nq, iy = row - ix * nq;
    for (int kz = threadIdx.x; kz <= nq / 2; kz += 32) {
        const SpecMode m = spec_mode(ix, iy, kz, nq);
        const long long q = (long long)row * P + kz;
        const float k2 = kf * kf * (float)(m.n[0] * m.n[0] + m.n[1] * m.n[1] + m.n[2] * m.n[2]);
        const float2 v = src[q];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float f = sign * (kf * m.n[a]) / k2 * norm;
            dst[a * pitch + q] = m.zero ? make_float2(0.f, 0.f) : make_float2(-f * v.y, f * v.x);  // i f v
        }
    }
}

// dst[t] = k_a k_b src / k^2 norm for the pairs (a, b) = 00, 11, 22, 01, 02, 12
__global__ void __launch_bounds__(32 * kSpecRows) k_ic_hess(const float2* __restrict__ src, float2* __restrict__ dst,
                                                            long long pitch, int nq, int P, float kf, float norm) {
    const int row = blockIdx.x * kSpecRows + threadIdx.y;
    if (row >= nq * nq) return;
    const int ix = row / nq, iy = row - ix * nq;
    for (int kz = threadIdx.x; kz <= nq / 2; kz += 32) {
        const SpecMode m = spec_mode(ix, iy, kz, nq);
        const long long q = (long long)row * P + kz;
        const float k2 = kf * kf * (float)(m.n[0] * m.n[0] + m.n[1] * m.n[1] + m.n[2] * m.n[2]);
        const float2 v = src[q];
        const float k[3] = {kf * m.n[0], kf * m.n[1], kf * m.n[2]};
        constexpr int pa[6] = {0, 1, 2, 0, 0, 1}, pb[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
        for (int t = 0; t < 6; ++t)
            dst[t * pitch + q] = m.zero ? make_float2(0.f, 0.f) : cscale(v, k[pa[t]] * k[pb[t]] / k2 * norm);
    }
}

// delta2 = phi00 phi11 + phi00 phi22 + phi11 phi22 - phi01^2 - phi02^2 - phi12^2 (real views)
__global__ void k_ic_delta2(float* b00, const float* b11, const float* b22, const float* b01, const float* b02,
                            const float* b12, int nq, long long P2) {
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n3 = (long long)nq * nq * nq;
    if (n >= n3) return;
    const long long row = n / nq;
    const long long q = row * P2 + (n - row * nq);
    const float p00 = b00[q], p11 = b11[q], p22 = b22[q], p01 = b01[q], p02 = b02[q], p12 = b12[q];
    b00[q] = p00 * p11 + p00 * p22 + p11 * p22 - p01 * p01 - p02 * p02 - p12 * p12;
}

// d = D1 psi1 + D2 psi2; v = 0 (COLA) or the LPT momentum a^3 E (D1' psi1 + D2' psi2) (PM only)
__global__ void k_ic_finish(cola_state st, long long np3, const double* row0, CosmoD c, int pm_only) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= np3) return;
    const float D1 = (float)row0[8], D2 = (float)row0[9];
    const float s1 = st.psi1[q], s2 = st.psi2[q];
    st.d[q] = D1 * s1 + D2 * s2;
    if (pm_only) {
        const double a = row0[0];
        const double pref = a * a * a * E_of(a, c);
        st.v[q] = (float)(pref * row0[10]) * s1 + (float)(pref * row0[11]) * s2;
    } else {
        st.v[q] = 0.f;
    }
}

int launch_ic(const cola_config* cfg, uint64_t seed, cola_state st, void* ws, const Layout& L, cudaStream_t s) {
    const int nq = cfg->nq;
    const int P = fft_pitch(nq);
    const size_t Mq = mesh_bytes(nq);
    float2* b[7];
    for (int i = 0; i < 7; ++i) b[i] = reinterpret_cast<float2*>(wsp(ws, L.ic + i * Mq));
    const float2* tw = twiddle_ptr(ws, kTwLagr);
    const CosmoD c = cosmo_of(cfg);
    const EhShape eh = eh_shape(c);
    const long long n3 = (long long)nq * nq * nq, mesh = (long long)nq * nq * P;
    const float kf = (float)(2.0 * 3.14159265358979323846 / cfg->box);
    const double dq = cfg->box / nq;
    const float norm = (float)(1.0 / ((double)n3));
    const unsigned gr = (unsigned)((n3 + 255) / 256), gs = (unsigned)((nq * nq + kSpecRows - 1) / kSpecRows);
    const dim3 ts(32, kSpecRows);
    const long long nrows = (long long)nq * nq;
    int rc;
    // forward transform of mesh 0 or 1; inverse of nm consecutive meshes, real rows to `out` or in place
    auto forward = [&](float2* buf) -> int {
        int r;
        if ((r = fft_z_r2c(nullptr, buf, nq, 0.f, tw, s, P, nrows, FRow{nq, 0, 1}))) return r;
        if ((r = fft_strided(buf, nq, 1, -1, tw, s))) return r;
        return fft_strided(buf, nq, 0, -1, tw, s);
    };
    auto inverse = [&](float2* buf, int nm, float* out) -> int {
        int r;
        const LineGeom x{(long long)nq * P, nm * nq, nq, mesh, P}, y{P, nm * nq, 1, (long long)nq * P, 0};
        if ((r = fft_lines(buf, nq, +1, tw, s, x, kKXInv))) return r;
        if ((r = fft_lines(buf, nq, +1, tw, s, y, kKYInv))) return r;
        return fft_z_c2r(buf, nq, tw, s, out, nq, 1.f, P, nm * nrows);
    };
    auto launched = [&](auto&& launch) -> int {
        ProfScope ps(kKIc, s);
        launch();
        return check_launch();
    };

    // white noise -> delta_k; the partial sums and the amplitude table sit in the idle meshes
    double* part = reinterpret_cast<double*>(b[1]);
    float* amp = reinterpret_cast<float*>(part + kSigBlocks);
    const int nm = 3 * (nq / 2 - 1) * (nq / 2 - 1) + 1;
    if ((rc = launched([&] { k_sigma8<<<kSigBlocks, 256, 0, s>>>(part, eh); }))) return rc;
    if ((rc = launched([&] {
             k_ic_amp<<<(nm + 255) / 256, 256, 0, s>>>(part, amp, nm, c.s8, (double)kf, dq * dq * dq, eh);
         })))
        return rc;
    if ((rc = launched([&] { k_noise<<<gr, 256, 0, s>>>(reinterpret_cast<float*>(b[0]), nq, 2ll * P, seed); })))
        return rc;
    if ((rc = forward(b[0]))) return rc;
    if ((rc = launched([&] { k_ic_delta<<<gs, ts, 0, s>>>(b[0], nq, P, amp); }))) return rc;
    // Psi1
    if ((rc = launched([&] { k_ic_grad<<<gs, ts, 0, s>>>(b[0], b[1], mesh, nq, P, kf, norm, 1.f); }))) return rc;
    if ((rc = inverse(b[1], 3, st.psi1))) return rc;
    // phi_ij -> delta2
    if ((rc = launched([&] { k_ic_hess<<<gs, ts, 0, s>>>(b[0], b[1], mesh, nq, P, kf, norm); }))) return rc;
    if ((rc = inverse(b[1], 6, nullptr))) return rc;
    if ((rc = launched([&] {
             k_ic_delta2<<<gr, 256, 0, s>>>((float*)b[1], (const float*)b[2], (const float*)b[3], (const float*)b[4],
                                            (const float*)b[5], (const float*)b[6], nq, 2ll * P);
         })))
        return rc;
    if ((rc = forward(b[1]))) return rc;
    // Psi2
    if ((rc = launched([&] { k_ic_grad<<<gs, ts, 0, s>>>(b[1], b[2], mesh, nq, P, kf, norm, -1.f); }))) return rc;
    if ((rc = inverse(b[2], 3, st.psi2))) return rc;
    return launched([&] {
        k_ic_finish<<<(unsigned)((3 * n3 + 255) / 256), 256, 0, s>>>(st, 3 * n3, table_ptr(ws), c,
                                                                     (cfg->flags & COLA_FLAG_PM_ONLY) ? 1 : 0);
    });
}

}  // namespace cola
