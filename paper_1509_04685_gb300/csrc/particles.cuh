// Particle-side helpers shared by the particle kernels (pm.cu) and the fused
// mesh kernels that deposit or gather inside an FFT pass (fft_fused.cuh):
// the CIC corners and fractions of a particle (Sec. 2.2), its fixed-point
// deposit weights, and the row bins of the PM step.
//
// Particle p = (i*nq + j)*nq + k sits at mesh coordinate
//   u = (i, j, k) * ng/nq + 1/2 + d * ng/L      (periodic)
// The Lagrangian part is formed exactly in integers, (i*2ng + nq)/(2nq), and
// only the small displacement term is FP32, so the CIC fraction keeps FP32
// precision for any mesh size.
//
// Deposit determinism: each particle's eight CIC weights are turned into
// unsigned 64-bit fixed point with 2^40 per particle (the largest corner takes
// the remainder so the eight sum to exactly 2^40) and added with integer
// atomics, which commute: the mesh is bit-identical whatever the order.
#pragma once

#include "cola_common.cuh"

namespace cola {

constexpr float kFix = 1099511627776.0f;  // 2^40

struct Cic {
    int c0[3];    // lower corner cell (wrapped)
    int c1[3];    // upper corner cell (wrapped)
    float f[3];   // fraction towards the upper corner
};

// Lattice site of particle index p (p < 2^31: nq^3 <= 4096^3 / 8 in practice;
// every lattice the library accepts has nq^3 < 2^31 particles addressed by int)
__device__ __forceinline__ void lattice_site(long long p, int nq, int idx[3]) {
    const unsigned q = (unsigned)p, n = (unsigned)nq;
    const unsigned ij = q / n;
    idx[2] = (int)(q - ij * n);
    idx[0] = (int)(ij / n);
    idx[1] = (int)(ij - (unsigned)idx[0] * n);
}

// The Lagrangian part of a lattice index along one axis in cells, (i 2 ng + nq) /
// (2 nq) in integers: whole cells and the fraction left.  For ng a multiple of
// nq it is i m + 1/2 exactly; otherwise one 32-bit division (i 2 ng + nq < 2^26
// for the sizes the library accepts).
struct Site1 {
    int base;
    float frac;
};
__device__ __forceinline__ Site1 site1(int i, int nq, int ng) {
    const int m = ng / nq;
    if (m * nq == ng) return Site1{i * m, 0.5f};
    const int den = 2 * nq, num = i * 2 * ng + nq, base = num / den;
    return Site1{base, (float)(num - base * den) / (float)den};
}

__device__ __forceinline__ bool cic_at(const Site1 st[3], int ng, float inv_cell, const float dx[3], Cic& c) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        // rounded explicitly (no contraction into an FMA): the binning, the
        // fused passes and the kick, in different translation units, must find
        // the same corner for the same particle
        const float t = __fadd_rn(st[a].frac, __fmul_rn(dx[a], inv_cell));
        if (!(fabsf(t) < 1.0e7f)) return false;  // NaN, Inf or absurd displacement
        const float fl = floorf(t);
        c.f[a] = t - fl;
        int cell = st[a].base + (int)fl;  // |cell| < 1e7 + 4096
        if ((unsigned)cell >= (unsigned)ng) {
            cell += cell < 0 ? ng : -ng;  // within a period of the box, the usual case
            if ((unsigned)cell >= (unsigned)ng) {
                cell %= ng;
                if (cell < 0) cell += ng;
            }
        }
        c.c0[a] = cell;
        c.c1[a] = (cell + 1 == ng) ? 0 : cell + 1;
    }
    return true;
}

__device__ __forceinline__ bool particle_cic(const int idx[3], int nq, int ng, float inv_cell, const float dx[3],
                                             Cic& c) {
    const Site1 st[3] = {site1(idx[0], nq, ng), site1(idx[1], nq, ng), site1(idx[2], nq, ng)};
    return cic_at(st, ng, inv_cell, dx, c);
}

// The eight fixed-point weights w[4a + 2b + e] of corner (c_a x, c_b y, c_e z):
// each rounded from the FP32 product, the corner of the largest weight along
// every axis taking the remainder of 2^40.  Weight i is hi[i] 2^20 + lo[i],
// 0 <= hi <= 2^20, |lo| <= 2^19: v 2^-20 and what it leaves are rounded by adding 1.5 2^23,
// which puts the integer into the mantissa, so the rounding to nearest (ties to
// even: hi 2^20 is even) is that of a conversion to 64 bits, without any
// 64-bit conversion or sum.
__device__ __forceinline__ void cic_fix_split(const Cic& c, int hi[8], int lo[8]) {
    const float wx[2] = {1.f - c.f[0], c.f[0]};
    const float wy[2] = {1.f - c.f[1], c.f[1]};
    const float wz[2] = {1.f - c.f[2], c.f[2]};
    const int m = 4 * (c.f[0] >= 0.5f) + 2 * (c.f[1] >= 0.5f) + (c.f[2] >= 0.5f);
    constexpr float magic = 12582912.0f;  // 1.5 2^23
    const int mbits = 0x4b400000;         // its bits
    int sh = 0, sl = 0;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int i = 4 * a + 2 * b + e;
                const float v = __fmul_rn(__fmul_rn(__fmul_rn(wx[a], wy[b]), wz[e]), kFix);
                const float h = __fmaf_rn(v, 9.5367431640625e-7f, magic);  // v 2^-20 is exact
                const float r = __fmaf_rn(__fsub_rn(h, magic), -1048576.0f, v);
                hi[i] = i == m ? 0 : __float_as_int(h) - mbits;
                lo[i] = i == m ? 0 : __float_as_int(__fadd_rn(r, magic)) - mbits;
                sh += hi[i];
                sl += lo[i];
            }
    // integer sums: the remainder is exact whatever the order of the others
    const int carry = ((1 << 19) - sl) >> 20;  // back to |lo| <= 2^19
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        hi[i] = i == m ? (1 << 20) - sh + carry : hi[i];
        lo[i] = i == m ? -sl - carry * (1 << 20) : lo[i];
    }
}

// the weight as one 64-bit integer
__device__ __forceinline__ unsigned long long fix_join(unsigned hi, int lo) {
    return (unsigned long long)hi * 1048576ull + (unsigned long long)(long long)lo;
}

__device__ __forceinline__ void cic_fix_weights(const Cic& c, unsigned long long w[8]) {
    int hi[8], lo[8];
    cic_fix_split(c, hi, lo);
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = fix_join((unsigned)hi[i], lo[i]);
}

}  // namespace cola
