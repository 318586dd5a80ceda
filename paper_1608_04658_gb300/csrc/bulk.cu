// Launcher of the bulk update for every storage form; FP64's instances (the
// other forms' have translation units of their own, to compile beside it).
#include "bulk.cuh"

namespace lbm {

extern template cudaError_t launch_bulk_t<float>(const Lattice &, const float *, float *, const uint8_t *, int *,
                                                 cudaStream_t, int, const int *, const int *, int, int);
extern template cudaError_t launch_bulk_t<__half>(const Lattice &, const __half *, __half *, const uint8_t *, int *,
                                                  cudaStream_t, int, const int *, const int *, int, int);
extern template cudaError_t launch_bulk_t<__nv_bfloat16>(const Lattice &, const __nv_bfloat16 *, __nv_bfloat16 *,
                                                         const uint8_t *, int *, cudaStream_t, int, const int *,
                                                         const int *, int, int);

cudaError_t launch_bulk(int storage, const Lattice &L, const void *fa, void *fb, const uint8_t *flags, int *status,
                        cudaStream_t s, int mode, const int *sweep, const int *cap, int z_lo, int z_n)
{
    if (mode != BULK_ALL && (!sweep || (mode == BULK_BAND && !cap))) return cudaErrorInvalidValue;
    if (z_n < 0) z_n = L.nz - z_lo;
    if (z_lo < 0 || z_lo + z_n > L.nz) return cudaErrorInvalidValue;
    if (z_n == 0 && mode != BULK_BAND) return cudaSuccess;
    return dispatch_storage(storage, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        return launch_bulk_t<S>(L, (const S *)fa, (S *)fb, flags, status, s, mode, sweep, cap, z_lo, z_n);
    });
}

}  // namespace lbm
