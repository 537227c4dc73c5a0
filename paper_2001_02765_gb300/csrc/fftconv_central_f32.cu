// Central-slope column pass and edge columns, FP32 instantiation (see fftconv_central.inl).
#include "fftconv_central.inl"

namespace sgk {
template sg_status cols_central<float>(int, int, int, const col_args<float> &, int, const float2 *, int *, cudaStream_t,
                                       const col_args<float> *, batch_shape);
template sg_status edge_cols<float>(int, const edge_args<float> &, const float2 *, cudaStream_t,
                                    const edge_args<float> *, batch_shape);
}  // namespace sgk
