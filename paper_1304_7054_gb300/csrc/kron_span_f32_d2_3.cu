// General-layout kernels: FP32 storage, 2-D, operand extents 13 to 16.
#include "kron_span.cuh"

namespace kron {
template <>
kron_status span_group<float, 2, 3>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<float, 2, 3>(d, a, smem, st);
}
}  // namespace kron
