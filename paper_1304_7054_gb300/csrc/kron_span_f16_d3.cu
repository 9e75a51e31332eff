// General-layout kernels: f16 storage, 3-D.
#include "kron_span.cuh"

namespace kron {
template <>
kron_status span_group<__half, 3, 0>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<__half, 3, 0>(d, a, smem, st);
}
template <>
kron_status span_group<__half, 3, 1>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<__half, 3, 1>(d, a, smem, st);
}
template <>
kron_status span_group<__half, 3, 2>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<__half, 3, 2>(d, a, smem, st);
}
template <>
kron_status span_group<__half, 3, 3>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<__half, 3, 3>(d, a, smem, st);
}
kron_status launch_span_f16_d3(const KronDesc& d, cudaStream_t s) { return launch_span<__half, 3>(d, s); }
}  // namespace kron
