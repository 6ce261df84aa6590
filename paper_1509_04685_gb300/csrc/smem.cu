// Dynamic shared-memory limits of the kernels.  A kernel's limit is set when a
// launch first needs it and again only for a larger launch: once a size has
// been used, launches of it (also those inside a stream capture) set nothing,
// and a launch captured earlier keeps the limit that it needs.  Every kernel of
// the library that any mesh needs has its entry, however many there are, and
// launches from several threads take turns.
#include <cuda_runtime.h>

#include <mutex>
#include <unordered_map>

#include "smem.h"

namespace cola {

bool set_smem(const void* fn, size_t bytes) {
    // the 48 KB a launch may take without the attribute covers static and
    // dynamic shared memory together; the kernels' static arrays stay far below 8 KB
    if (bytes + 8 * 1024 <= 48 * 1024) return true;
    static std::mutex mutex;
    static std::unordered_map<const void*, size_t> limit;
    const std::lock_guard<std::mutex> lock(mutex);
    size_t& have = limit[fn];
    if (have >= bytes) return true;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) {
        g_last_cuda_error = (int)e;
        cudaGetLastError();
        return false;
    }
    have = bytes;
    return true;
}

}  // namespace cola
