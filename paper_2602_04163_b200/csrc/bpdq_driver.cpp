// The one entry point the library takes from the driver (it does not link libcuda).
#include <cuda_runtime_api.h>

#include "bpdq_tma.cuh"

namespace bpdq {

// Handles may be created in several threads at once, each of which asks: the answer is looked up in the initialiser of a local
// static, which later callers wait for.
EncodeTiledFn encode_tiled_fn() {
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(ptr);
        cudaGetLastError();
        return nullptr;
    }();
    return fn;
}

}  // namespace bpdq
