// General-layout kernels: FP32 storage, 3-D, operand extents 1 to 4.
#include "kron_span.cuh"

namespace kron {
template <>
kron_status span_group<float, 3, 0>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<float, 3, 0>(d, a, smem, st);
}
}  // namespace kron
