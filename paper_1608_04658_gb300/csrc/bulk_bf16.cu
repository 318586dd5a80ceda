// The bulk update's instances for BF16 storage.
#include "bulk.cuh"

namespace lbm {
template cudaError_t launch_bulk_t<__nv_bfloat16>(const Lattice &, const __nv_bfloat16 *, __nv_bfloat16 *, const uint8_t *, int *, cudaStream_t, int,
                                        const int *, const int *, int, int);
}  // namespace lbm
