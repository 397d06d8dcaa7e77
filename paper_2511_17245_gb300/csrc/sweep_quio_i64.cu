// sweep_quio_i64.cu -- sweep kernels for QUIO models with i64 fields.
#include "sweep_launch.cuh"

namespace sa {
int launch_sweep_quio_i64(const SweepArgs& a, int zbytes, int rule, bool smem, int blocks, int threads,
                              size_t sh, void* stream) {
    return launch_family<long long, KIND_QUIO>(a, zbytes, rule, smem, blocks, threads, sh, (cudaStream_t)stream);
}
}  // namespace sa
