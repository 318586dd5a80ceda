// The bulk update's instances for FP32 storage.
#include "bulk.cuh"

namespace lbm {
template cudaError_t launch_bulk_t<float>(const Lattice &, const float *, float *, const uint8_t *, int *, cudaStream_t, int,
                                        const int *, const int *, int, int);
}  // namespace lbm
