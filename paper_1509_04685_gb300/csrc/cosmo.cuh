// The cosmology of a configuration in FP64, and the pieces of it that the
// growth tables (growth.cu) and the initial conditions (ic.cu) share.
#pragma once

#include "cola_common.cuh"

namespace cola {

struct CosmoD {
    double om, ol, ok, ob, h, s8, ns, tcmb;
};

inline CosmoD cosmo_of(const cola_config* cfg) {
    const cola_cosmology& c = cfg->cosmo;
    return CosmoD{c.omega_m, c.omega_l, 1.0 - c.omega_m - c.omega_l, c.omega_b, c.h, c.sigma8, c.n_s, c.t_cmb};
}

__device__ __forceinline__ double E_of(double a, const CosmoD& c) {
    return sqrt(c.om / (a * a * a) + c.ok / (a * a) + c.ol);
}

}  // namespace cola
