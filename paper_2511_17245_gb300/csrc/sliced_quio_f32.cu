// sliced_quio_f32.cu -- time-sliced sweep kernels for QUIO models with f32 fields.
#include "sweep_launch.cuh"

namespace sa {
int launch_sliced_quio_f32(const SweepArgs& a, int zbytes, int rule, int grid, int threads, size_t sh, void* stream,
                        int* bps) {
    return launch_sliced_family<float, KIND_QUIO>(a, zbytes, rule, grid, threads, sh, (cudaStream_t)stream, bps);
}
}  // namespace sa
