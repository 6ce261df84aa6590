// Dynamic shared-memory limits of the kernels (smem.cu).
#pragma once

#include <cstddef>

namespace cola {

extern int g_last_cuda_error;  // the CUDA error behind the last COLA_ECUDA of a launch (cola_last_cuda_error)

// Raise kernel fn's dynamic shared-memory limit to at least `bytes`; false if CUDA refuses.
bool set_smem(const void* fn, size_t bytes);

}  // namespace cola
