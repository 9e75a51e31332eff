// General-layout kernels: FP32 storage, 3-D (layout, dispatch, runtime extents).
#include "kron_span.cuh"

namespace kron {
template <>
kron_status span_group<float, 3, 0>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st);
template <>
kron_status span_group<float, 3, 1>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st);
template <>
kron_status span_group<float, 3, 2>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st);
template <>
kron_status span_group<float, 3, 3>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st);
kron_status launch_span_f32_d3(const KronDesc& d, cudaStream_t s) { return launch_span<float, 3>(d, s); }
}  // namespace kron
