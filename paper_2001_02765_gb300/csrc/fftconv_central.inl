// Column pass of the central-slope convolution (slope spectra formed from
// sigma's, see fftconv.cuh) with its launch-shape variants, and the edge-column
// transforms it needs, for one solve or a batch of solves of one padded length.
#include "fftconv.cuh"

namespace sgk {
namespace {

template <typename T, int PY, int CB, int NOUT, bool BATCH>
sg_status launch_cols_central(const col_args<T> &one, const col_args<T> *many, batch_shape bs, int qx,
                              const cplx_t<T> *tw, int *err, cudaStream_t st)
{
    constexpr int THREADS = CB * PY / 8, NPL = NOUT == 3 ? 9 : (NOUT == 1 ? 3 : 6);
    const size_t smem = (size_t)col_smem_bytes<T, PY, CB, NPL, col_central_nbuf<T, PY, CB, NOUT, BATCH>()>();
    auto kern = k_col_conv_central<T, PY, CB, THREADS, NOUT, BATCH>;
    SG_TRY(smem_limit(kern, smem));
    dim3 grid((qx + CB - 1) / CB, 1, BATCH ? bs.nmem : 1);
    SG_CUDA_TRY(sg_launch_dep(kern, grid, dim3(THREADS), smem, st, one, many, qx, tw, err));
    SG_CUDA_TRY(cudaGetLastError());
    return SG_OK;
}

template <typename T, int PY, int CB>
sg_status launch_cols_central_any(const col_args<T> &one, const col_args<T> *many, batch_shape bs, int qx,
                                  const cplx_t<T> *tw, int *err, cudaStream_t st)
{
    if (many) return launch_cols_central<T, PY, CB, 2, true>(one, many, bs, qx, tw, err, st);
    return launch_cols_central<T, PY, CB, 2, false>(one, many, bs, qx, tw, err, st);
}

// the potential and off-plane passes (one and three outputs) have the default shape only
template <typename T, int PY>
sg_status cols_central_py(int cb, int nout, const col_args<T> &one, const col_args<T> *many, batch_shape bs, int qx,
                          const cplx_t<T> *tw, int *err, cudaStream_t st)
{
    constexpr int D = col_cb_default(PY);
    constexpr int A = shape_candidate(D, 0), C = shape_candidate(D, 2);
    if (nout != 2) {
        if (many) return SG_EINVAL;
        if (nout == 1) return launch_cols_central<T, PY, D, 1, false>(one, many, bs, qx, tw, err, st);
        return launch_cols_central<T, PY, D, 3, false>(one, many, bs, qx, tw, err, st);
    }
    if (cb == D) return launch_cols_central_any<T, PY, D>(one, many, bs, qx, tw, err, st);
    if constexpr (col_feasible_t<T, PY, A, 6>()) {
        if (cb == A) return launch_cols_central_any<T, PY, A>(one, many, bs, qx, tw, err, st);
    }
    if constexpr (col_feasible_t<T, PY, C, 6>()) {
        if (cb == C) return launch_cols_central_any<T, PY, C>(one, many, bs, qx, tw, err, st);
    }
    return SG_EINVAL;
}

template <typename T, int PY>
sg_status launch_edge_cols(const edge_args<T> &one, const edge_args<T> *many, batch_shape bs, const cplx_t<T> *tw,
                           cudaStream_t st)
{
    constexpr int THREADS = PY / 8 >= 64 ? (PY / 8 + 31) / 32 * 32 : 64;
    const size_t smem = (size_t)spad_size<cplx_t<T>>(PY) * sizeof(cplx_t<T>);
    // the first kernel of the solve; the row pass starts beside it (see k_edge_cols)
    if (many) {
        auto kern = k_edge_cols<T, PY, THREADS, true>;
        SG_TRY(smem_limit(kern, smem));
        SG_CUDA_TRY(sg_launch_dep(kern, dim3(1, 1, bs.nmem), dim3(THREADS), smem, st, one, many, tw));
    } else {
        auto kern = k_edge_cols<T, PY, THREADS, false>;
        SG_TRY(smem_limit(kern, smem));
        SG_CUDA_TRY(sg_launch_dep(kern, dim3(1), dim3(THREADS), smem, st, one, many, tw));
    }
    SG_CUDA_TRY(cudaGetLastError());
    return SG_OK;
}

}  // namespace

template <typename T>
sg_status cols_central(int py, int cb, int nout, const col_args<T> &one, int qx, const cplx_t<T> *tw, int *err, cudaStream_t st,
                       const col_args<T> *many, batch_shape bs)
{
    SG_PAD_SWITCH(py, return (cols_central_py<T, PP>(cb, nout, one, many, bs, qx, tw, err, st)));
    return SG_EINVAL;
}

template <typename T>
sg_status edge_cols(int py, const edge_args<T> &one, const cplx_t<T> *tw, cudaStream_t st, const edge_args<T> *many,
                    batch_shape bs)
{
    SG_PAD_SWITCH(py, return (launch_edge_cols<T, PP>(one, many, bs, tw, st)));
    return SG_EINVAL;
}

}  // namespace sgk
