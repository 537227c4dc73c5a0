// Central-slope column pass and edge columns, FP64 instantiation (see fftconv_central.inl).
#include "fftconv_central.inl"

namespace sgk {
template sg_status cols_central<double>(int, int, int, const col_args<double> &, int, const double2 *, int *, cudaStream_t,
                                        const col_args<double> *, batch_shape);
template sg_status edge_cols<double>(int, const edge_args<double> &, const double2 *, cudaStream_t,
                                     const edge_args<double> *, batch_shape);
}  // namespace sgk
