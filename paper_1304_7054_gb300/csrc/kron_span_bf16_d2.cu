// General-layout kernels: bf16 storage, 2-D.
#include "kron_span.cuh"

namespace kron {
template <>
kron_status span_group<__nv_bfloat16, 2, 0>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<__nv_bfloat16, 2, 0>(d, a, smem, st);
}
template <>
kron_status span_group<__nv_bfloat16, 2, 1>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<__nv_bfloat16, 2, 1>(d, a, smem, st);
}
template <>
kron_status span_group<__nv_bfloat16, 2, 2>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<__nv_bfloat16, 2, 2>(d, a, smem, st);
}
template <>
kron_status span_group<__nv_bfloat16, 2, 3>(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    return launch_span_group<__nv_bfloat16, 2, 3>(d, a, smem, st);
}
kron_status launch_span_bf16_d2(const KronDesc& d, cudaStream_t s) { return launch_span<__nv_bfloat16, 2>(d, s); }
}  // namespace kron
