// sliced_quio_i64.cu -- time-sliced sweep kernels for QUIO models with i64 fields.
#include "sweep_launch.cuh"

namespace sa {
int launch_sliced_quio_i64(const SweepArgs& a, int zbytes, int rule, int grid, int threads, size_t sh, void* stream,
                        int* bps) {
    return launch_sliced_family<long long, KIND_QUIO>(a, zbytes, rule, grid, threads, sh, (cudaStream_t)stream, bps);
}
}  // namespace sa
