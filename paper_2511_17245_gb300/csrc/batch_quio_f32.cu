// batch_quio_f32.cu -- batch kernels for QUIO models with f32 fields.
#include "sweep_launch.cuh"

namespace sa {
int launch_batch_quio_f32(const BatchArgs& b, int zbytes, int rule, bool smem, int blocks, int threads,
                             size_t sh, void* stream, bool set_attr) {
    return launch_batch_family<float, KIND_QUIO>(b, zbytes, rule, smem, blocks, threads, sh, (cudaStream_t)stream, set_attr);
}
}  // namespace sa
