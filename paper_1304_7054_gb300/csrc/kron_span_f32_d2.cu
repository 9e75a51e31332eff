// General-layout kernels: FP32 storage, 2-D (layout, dispatch, runtime extents).
#include "kron_span.cuh"

namespace kron {
template <>
kron_status span_group<float, 2, 0>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st);
template <>
kron_status span_group<float, 2, 1>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st);
template <>
kron_status span_group<float, 2, 2>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st);
template <>
kron_status span_group<float, 2, 3>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st);
kron_status launch_span_f32_d2(const KronDesc& d, cudaStream_t s) { return launch_span<float, 2>(d, s); }
}  // namespace kron
