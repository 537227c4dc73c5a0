// Forward row pass, FP64 instantiation (see fftconv_rows.inl).
#include "fftconv_rows.inl"

namespace sgk {
template sg_status rows_fwd<double>(int, int, const row_fwd_args<double> &, int, const double2 *, cudaStream_t,
                                    const row_fwd_args<double> *, batch_shape, int, const edge_args<double> *,
                                    const edge_args<double> *);
}  // namespace sgk
