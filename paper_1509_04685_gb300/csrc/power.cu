// Matter power spectrum shells (Sec. 2.5): P(k) = <|delta_k|^2> over the modes
// of each k-bin, with optional CIC deconvolution and the Jing (2005) CIC
// aliasing correction, closed form or iterated.
//
// Bin i (1 .. ng/2) holds the modes with (i - 1/2)^2 < |n|^2 < (i + 1/2)^2,
// decided in integer arithmetic.  Half-spectrum modes count twice except on
// the kz = 0 and kz = Nyquist planes.  P(k_n) = |delta_k|^2 L^3 / ng^6.
// A fixed grid of blocks each accumulates its share of the modes into FP32
// shared-memory bins; the per-block partials are then summed in FP64 in a
// fixed block order.  With MULTI the bins also take P L_2(mu) and P L_4(mu),
// mu = n_z / |n| (line of sight z): the redshift-space multipoles
// P_l = (2l + 1) <P L_l(mu)> of the paper's RSD study (Eq. 5).
#include "cola_common.cuh"

namespace cola {

constexpr int kPkBlocks = 608;  // 4 blocks per SM on a 152-SM GB300
constexpr int kPkThreads = 256;

// Iterated Jing (2005) correction of one mode m (flag COLA_PK_ALIAS_ITER): the
// raw power over C(m) = sum over the images |n_i| <= kJingImages of
// W^2(m + ng n) (|m + ng n| / |m|)^n_eff, W the CIC window, P taken as a power
// law of index n_eff (this mode's bin) around |m|.  sin(pi (m + ng n) / ng) =
// +-sin(pi m / ng), so each image's window factor is, per axis,
// sin^4(pi m / ng) / (pi (m + ng n) / ng)^4 (1 for m = n = 0, 0 for m = 0 != n).
constexpr int kJingImages = 2;
constexpr int kJingIterations = 3;
constexpr double kNeffClamp = 4.0;

__device__ __forceinline__ float jing_alias_sum(const int nn[3], int ng, float n_eff) {
    constexpr int NI = 2 * kJingImages + 1;
    const float inv_ng = 1.0f / (float)ng;
    float fa[3][NI], x[3][NI];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float s = sinpif((float)nn[a] * inv_ng);
        const float s4 = (s * s) * (s * s);
#pragma unroll
        for (int j = 0; j < NI; ++j) {
            const int n = j - kJingImages;
            x[a][j] = (float)(nn[a] + ng * n);
            if (nn[a] == 0) {
                fa[a][j] = n == 0 ? 1.f : 0.f;
            } else {
                const float t = 3.14159265358979f * x[a][j] * inv_ng;
                fa[a][j] = s4 / ((t * t) * (t * t));
            }
        }
    }
    const float lm2 = log2f((float)((long long)nn[0] * nn[0] + (long long)nn[1] * nn[1] + (long long)nn[2] * nn[2]));
    const float h = 0.5f * n_eff;
    float C = 0.f;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        if (fa[0][i] == 0.f) continue;
#pragma unroll
        for (int j = 0; j < NI; ++j) {
            const float wxy = fa[0][i] * fa[1][j];
            if (wxy == 0.f) continue;
            const float rxy = x[0][i] * x[0][i] + x[1][j] * x[1][j];
#pragma unroll
            for (int l = 0; l < NI; ++l) {
                const float w = wxy * fa[2][l];
                if (w != 0.f) C += w * exp2f(h * (log2f(rxy + x[2][l] * x[2][l]) - lm2));
            }
        }
    }
    return C;
}

// bin of a mode with |n|^2 = n2 >= 1 (n2 < 2^24): (i - 1/2)^2 < n2 < (i + 1/2)^2, from its FP32 root
__device__ __forceinline__ int shell_of(int n2, float root) {
    int i = (int)(root + 0.5f);
    while (i * i + i < n2) ++i;
    while (i * i - i + 1 > n2) --i;
    return i;
}

// C of the iterated correction for every mode shape: it depends on |n_x|, |n_y|
// and n_z in any order, so one entry serves up to 24 modes of the half
// spectrum (four signs of n_x, n_y, six orders): ctab[(a H + b) H + c], a >= b >= c.
// (Evaluated per mode, 125 logarithms and exponentials each, the three
// iterations took 27.4 ms at 512^3; the tables take 1.6 ms.)  The shells up to
// low = min(kJingLow, nbins) have few modes, and there the FP32 rounding of C
// shows in P: they get a table with an entry per signed mode behind the first,
// ((n_x + low) (2 low + 1) + n_y + low) (low + 1) + n_z.
constexpr int kJingLow = 32;
__global__ void __launch_bounds__(128) k_pk_jing(float* __restrict__ ctab, int ng, int nbins, int low,
                                                 const double* __restrict__ neff) {
    const int H = ng / 2 + 1;
    const int a = blockIdx.z, b = blockIdx.y, c = blockIdx.x * 128 + threadIdx.x;
    if (b > a || c > b || a == 0) return;
    const int n2 = a * a + b * b + c * c;
    const int i = shell_of(n2, sqrtf((float)n2));
    if (i > nbins || i <= low) return;
    const int nn[3] = {a, b, c};
    ctab[((size_t)a * H + b) * H + c] = jing_alias_sum(nn, ng, (float)neff[i - 1]);
}

__global__ void __launch_bounds__(64) k_pk_jing_low(float* __restrict__ clow, int ng, int low,
                                                    const double* __restrict__ neff) {
    const int nn[3] = {(int)blockIdx.y - low, (int)blockIdx.x - low, (int)threadIdx.x};
    if (nn[2] > low) return;
    const int n2 = nn[0] * nn[0] + nn[1] * nn[1] + nn[2] * nn[2];
    if (n2 == 0) return;
    const int i = shell_of(n2, sqrtf((float)n2));
    if (i > low) return;
    clow[(blockIdx.y * (2 * low + 1) + blockIdx.x) * (low + 1) + nn[2]] = jing_alias_sum(nn, ng, (float)neff[i - 1]);
}

// Shell sums: a block adds the modes blockIdx.x 256 + threadIdx.x, then every
// gridDim.x 256-th, into FP32 rows in shared memory (compare-and-swap loops, so
// lanes of one shell take turns: this bounds the kernel) and integer counts.
// The window factors per axis come from tables, the mode index is advanced
// without divisions and the next mode's value is read ahead.  (With divisions,
// three sines per window and FP32 counts per mode 6.4 ms at 1024^3, now 3.0 ms;
// lanes on modes 8 apart, which rarely share a shell, took 4.0 ms: eight index
// computations in flight cost more than the turns.)  ITER: a pass of the iterated correction, which only needs
// the sums of w P (the counts and sums of w k do not change).
template <bool MULTI, bool ITER>
__global__ void __launch_bounds__(kPkThreads) k_pk_shells(const float2* __restrict__ mk, int ng, int xbs, long long P,
                                                          float amp_scale, float kf, int flags, int nbins,
                                                          double* __restrict__ part, const float* __restrict__ ctab,
                                                          int low) {
    constexpr int NF = MULTI ? 4 : 2;  // sum w k, sum w P [, sum w P L2, sum w P L4]
    extern __shared__ float bins[];    // NF float rows of nbins, one of counts, then the axis tables
    unsigned* count = reinterpret_cast<unsigned*>(bins + NF * nbins);
    const int H = ng / 2 + 1, half = ng / 2;
    float* win = bins + (NF + 1) * nbins;  // CIC window sinc^2 per axis index
    float* jw = win + H;                   // closed-form alias factor per axis index
    for (int i = threadIdx.x; i < (NF + 1) * nbins; i += kPkThreads) bins[i] = 0.f;
    const float inv_ng = 1.0f / (float)ng;
    for (int n = threadIdx.x; n < H; n += kPkThreads) {
        const float x = (float)n * inv_ng, s = sinpif(x);
        const float sc = s / (3.14159265358979f * x);
        win[n] = n ? sc * sc : 1.f;
        jw[n] = 1.f - 2.f / 3.f * s * s;
    }
    __syncthreads();
    // (ix, iy, kz) of the first mode, and the step from one to the next
    const unsigned first = blockIdx.x * kPkThreads + threadIdx.x, stride = gridDim.x * kPkThreads;
    const unsigned dr = stride / H, dz = stride - dr * H, dx = dr / ng, dy = dr - dx * ng;
    int kz = (int)(first % H), iy = (int)(first / H % ng), ix = (int)(first / H / ng);
    const FRow fr{ng, xbs, 1};
    auto value = [&] { return ix < ng ? __ldg(mk + frow(ix, iy, 0, fr) * P + kz) : make_float2(0.f, 0.f); };
    float2 next = value();
    while (ix < ng) {
        const float2 d = next;
        const int mx = ix, my = iy, mz = kz;
        kz += (int)dz;
        iy += (int)dy;
        ix += (int)dx;
        if (kz >= H) {
            kz -= H;
            ++iy;
        }
        if (iy >= ng) {
            iy -= ng;
            ++ix;
        }
        next = value();
        const int nx = mx < half ? mx : ng - mx, ny = my < half ? my : ng - my;  // |n_x|, |n_y|
        const int n2 = nx * nx + ny * ny + mz * mz;
        if (n2 == 0) continue;
        const float root = sqrtf((float)n2);
        const int i = shell_of(n2, root);
        if (i > nbins) continue;
        const float re = d.x * amp_scale, im = d.y * amp_scale;
        float p = __fmaf_rn(re, re, __fmul_rn(im, im));  // rounded explicitly: one order for every variant
        if (ITER) {
            const float* c;
            if (i <= low) {
                const int sx = mx < half ? nx : -nx, sy = my < half ? ny : -ny;
                c = ctab + (size_t)H * H * H + ((sx + low) * (2 * low + 1) + sy + low) * (low + 1) + mz;
            } else {
                const int lo = min(nx, ny), hi = max(nx, ny);
                const int a = max(hi, mz), e = min(lo, mz), b = nx + ny + mz - a - e;
                c = ctab + ((size_t)a * H + b) * H + e;
            }
            p /= __ldg(c);
        }
        if (flags & COLA_PK_DECONV_CIC) {
            const float W = win[nx] * win[ny] * win[mz];
            p /= W * W;
        }
        if (flags & COLA_PK_ALIAS_JING) p /= jw[nx] * jw[ny] * jw[mz];
        const bool once = mz == 0 || mz == half;
        const float wt = once ? 1.f : 2.f;
        if (!ITER) {
            atomicAdd(&count[i - 1], once ? 1u : 2u);
            atomicAdd(&bins[i - 1], wt * (kf * root));
        }
        atomicAdd(&bins[nbins + i - 1], wt * p);
        if (MULTI) {
            const float mu2 = (float)(mz * mz) / (float)n2;
            const float l2 = 1.5f * mu2 - 0.5f;
            const float l4 = (35.f * mu2 * mu2 - 30.f * mu2 + 3.f) * 0.125f;
            atomicAdd(&bins[2 * nbins + i - 1], wt * p * l2);
            atomicAdd(&bins[3 * nbins + i - 1], wt * p * l4);
        }
    }
    __syncthreads();
    double* o = part + (size_t)blockIdx.x * (NF + 1) * nbins;
    for (int i = threadIdx.x; i < nbins; i += kPkThreads) {
        if (!ITER) o[i] = (double)count[i];
        for (int q = ITER ? 1 : 0; q < NF; ++q) o[(q + 1) * nbins + i] = (double)bins[q * nbins + i];
    }
}

// The closed-form pass that starts the iterated correction: the same sums with
// every index, window and count worked out per mode (0.8 ms at 512^3 against
// 0.4 ms).  The slopes of the iteration amplify the rounding of sum w k by up to
// 1e4 in single bins, and that rounding depends on the order in which the warps
// of a block reach its bins, hence on the pace of this loop; it stays as it is
// so that iterated spectra stay as near to earlier ones as two runs are.
__global__ void __launch_bounds__(kPkThreads) k_pk_shells_first(const float2* __restrict__ mk, int ng, int xbs, long long P,
                                                                float amp_scale, float kf, int nbins,
                                                                double* __restrict__ part) {
    extern __shared__ float bins[];
    for (int i = threadIdx.x; i < 3 * nbins; i += blockDim.x) bins[i] = 0.f;
    __syncthreads();
    const int H = ng / 2 + 1;
    const long long total = (long long)ng * ng * H;
    const int half = ng / 2;
    const float inv_ng = 1.0f / (float)ng;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const long long row = e / H;
        const int kz = (int)(e - row * H);
        const int ix = (int)(row / ng), iy = (int)(row - (long long)ix * ng);
        const int nn[3] = {ix < half ? ix : ix - ng, iy < half ? iy : iy - ng, kz};
        const long long n2 = (long long)nn[0] * nn[0] + (long long)nn[1] * nn[1] + (long long)kz * kz;
        if (n2 == 0) continue;
        int i = (int)(sqrtf((float)n2) + 0.5f);
        while ((long long)i * i + i < n2) ++i;
        while ((long long)i * i - i + 1 > n2) --i;
        if (i < 1 || i > nbins) continue;
        const float2 d = mk[frow(ix, iy, 0, FRow{ng, xbs, 1}) * P + kz];
        const float re = d.x * amp_scale, im = d.y * amp_scale;
        float p = __fmaf_rn(re, re, __fmul_rn(im, im));
        float W = 1.f, C = 1.f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (nn[a] != 0) {
                const float x = (float)nn[a] * inv_ng;
                const float sc = sinpif(x) / (3.14159265358979f * x);
                W *= sc * sc;
            }
        }
        p /= W * W;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float s = sinpif((float)nn[a] * inv_ng);
            C *= 1.f - 2.f / 3.f * s * s;
        }
        p /= C;
        const float w = (kz == 0 || kz == half) ? 1.f : 2.f;
        atomicAdd(&bins[i - 1], w);
        atomicAdd(&bins[nbins + i - 1], w * (kf * sqrtf((float)n2)));
        atomicAdd(&bins[2 * nbins + i - 1], w * p);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * nbins; i += blockDim.x)
        part[(size_t)blockIdx.x * 3 * nbins + i] = (double)bins[i];
}

// The blocks' partials summed in FP64 in a fixed order: 32 bins per block of 32
// x 16 threads, thread row y adding partials y, y + 16, ... (one thread per bin
// walking all 608 took 0.17 ms).
constexpr int kRedRows = 16;
__global__ void __launch_bounds__(32 * kRedRows) k_pk_reduce(const double* __restrict__ part, int nblocks, int nbins,
                                                             double* k, double* pk, double* nmodes, double* p2,
                                                             double* p4) {
    __shared__ double red[5][kRedRows][32];
    const int i = blockIdx.x * 32 + threadIdx.x;
    const int NA = p2 ? 5 : 3;
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (i < nbins)
        for (int b = threadIdx.y; b < nblocks; b += kRedRows) {
            const double* q = part + (size_t)b * NA * nbins + i;
#pragma unroll
            for (int a = 0; a < 5; ++a)
                if (a < NA) acc[a] += q[(size_t)a * nbins];
        }
#pragma unroll
    for (int a = 0; a < 5; ++a) red[a][threadIdx.y][threadIdx.x] = acc[a];
    __syncthreads();
    if (threadIdx.y || i >= nbins) return;
#pragma unroll
    for (int a = 0; a < 5; ++a)
        for (int y = 1; y < kRedRows; ++y) acc[a] += red[a][y][threadIdx.x];
    const double w = acc[0];
    nmodes[i] = w;
    k[i] = w > 0.0 ? acc[1] / w : 0.0;
    pk[i] = w > 0.0 ? acc[2] / w : 0.0;
    if (p2) {
        p2[i] = w > 0.0 ? 5.0 * acc[3] / w : 0.0;
        p4[i] = w > 0.0 ? 9.0 * acc[4] / w : 0.0;
    }
}

// n_eff per bin for the next Jing iteration: d ln P / d ln k over the
// neighbouring bins (one-sided at the ends; 0 where a power is not positive),
// clamped to [-kNeffClamp, kNeffClamp]
__global__ void k_pk_slopes(const double* __restrict__ k, const double* __restrict__ pk, int nbins, double* neff) {
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
        const int lo = b > 0 ? b - 1 : 0, hi = b + 1 < nbins ? b + 1 : nbins - 1;
        double n = 0.0;
        if (hi != lo && pk[lo] > 0.0 && pk[hi] > 0.0 && k[hi] > k[lo] && k[lo] > 0.0)
            n = fmin(fmax(log(pk[hi] / pk[lo]) / log(k[hi] / k[lo]), -kNeffClamp), kNeffClamp);
        neff[b] = n;
    }
}

int launch_power(const float2* mk, int ng, int xbs, long long rs, double box, int flags, double* part, float* ctab, double* k,
                 double* pk, double* nmodes, int nbins, cudaStream_t s, double* p2, double* p4) {
    const double ng3 = (double)ng * ng * ng;
    const float amp_scale = (float)(box * sqrt(box) / ng3);  // sqrt(L^3 / ng^6)
    const float kf = (float)(2.0 * 3.14159265358979323846 / box);
    const bool multi = p2 && p4;
    const int H = ng / 2 + 1;
    const size_t smem = ((size_t)(multi ? 5 : 3) * nbins + 2 * H) * sizeof(float);
    double* neff = part + (size_t)kPkBlocks * 5 * nbins;
    const int low = nbins < kJingLow ? nbins : kJingLow;
    auto reduce = [&]() -> int {
        if (int rc = check_launch()) return rc;
        ProfScope ps(kKPkReduce, s);
        k_pk_reduce<<<(nbins + 31) / 32, dim3(32, kRedRows), 0, s>>>(part, kPkBlocks, nbins, k, pk, nmodes,
                                                                    multi ? p2 : nullptr, multi ? p4 : nullptr);
        return check_launch();
    };
    auto estimate = [&](int fl) -> int {
        const bool iter = fl & COLA_PK_ALIAS_ITER;
        auto kern = multi ? k_pk_shells<true, false> : (iter ? k_pk_shells<false, true> : k_pk_shells<false, false>);
        if (!set_smem((const void*)kern, smem)) return COLA_ECUDA;
        {
            ProfScope ps(kKPkShells, s);
            kern<<<kPkBlocks, kPkThreads, smem, s>>>(mk, ng, xbs, rs, amp_scale, kf, fl, nbins, part, ctab, low);
        }
        return reduce();
    };
    if (!(flags & COLA_PK_ALIAS_ITER)) return estimate(flags);
    // closed-form start, then kJingIterations passes with slopes from the last estimate
    {
        ProfScope ps(kKPkShells, s);
        k_pk_shells_first<<<kPkBlocks, kPkThreads, 3 * (size_t)nbins * sizeof(float), s>>>(mk, ng, xbs, rs, amp_scale, kf,
                                                                                        nbins, part);
    }
    int rc = reduce();
    for (int it = 0; it < kJingIterations && !rc; ++it) {
        k_pk_slopes<<<1, 256, 0, s>>>(k, pk, nbins, neff);
        if ((rc = check_launch())) break;
        {
            ProfScope ps(kKPkShells, s);
            k_pk_jing<<<dim3((H + 127) / 128, H, H), 128, 0, s>>>(ctab, ng, nbins, low, neff);
            if ((rc = check_launch())) break;
            k_pk_jing_low<<<dim3(2 * low + 1, 2 * low + 1), 64, 0, s>>>(ctab + (size_t)H * H * H, ng, low, neff);
        }
        if ((rc = check_launch())) break;
        rc = estimate(COLA_PK_ALIAS_ITER);
    }
    return rc;
}

// per-block partial sums, then the n_eff table of the iterated Jing correction
size_t power_partial_bytes(int nbins) { return ((size_t)kPkBlocks * 5 + 1) * nbins * sizeof(double); }

}  // namespace cola
