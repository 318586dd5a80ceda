// The bulk update's instances for FP16 storage.
#include "bulk.cuh"

namespace lbm {
template cudaError_t launch_bulk_t<__half>(const Lattice &, const __half *, __half *, const uint8_t *, int *, cudaStream_t, int,
                                        const int *, const int *, int, int);
}  // namespace lbm
