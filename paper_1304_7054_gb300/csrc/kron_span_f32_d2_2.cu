// General-layout kernels: FP32 storage, 2-D, operand extents 9 to 12.
#include "kron_span.cuh"

namespace kron {
template <>
kron_status span_group<float, 2, 2>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<float, 2, 2>(d, a, smem, st);
}
}  // namespace kron
