// Forward row pass, FP32 instantiation (see fftconv_rows.inl).
#include "fftconv_rows.inl"

namespace sgk {
template sg_status rows_fwd<float>(int, int, const row_fwd_args<float> &, int, const float2 *, cudaStream_t,
                                   const row_fwd_args<float> *, batch_shape, int, const edge_args<float> *,
                                   const edge_args<float> *);
}  // namespace sgk
