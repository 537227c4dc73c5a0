// Forward row pass of the uniform-patch convolution (R2C with the fields
// formed) and its launch-shape variants, for one solve or a batch of solves of
// one padded length.
#include "fftconv.cuh"

namespace sgk {
namespace {

// EDGE_BEFORE: launched right after the edge-column transform of a central-slope
// solve, as a dependent launch that runs beside it and waits for it at its end
// (row_fwd_body with WAIT_AT_END); otherwise the first kernel of the solve, a
// dependent launch too (it waits for the stream's previous kernel at its start):
// launched normally, solves back to back started on a grid of 2.05 us steps.
template <typename T, int PX, int NB, bool BATCH, int EDGE>
sg_status launch_rows_fwd(const row_fwd_args<T> &one, const row_fwd_args<T> *many, const edge_args<T> *ed,
                          const edge_args<T> *ed_many, batch_shape bs, int nf, const cplx_t<T> *tw, cudaStream_t st)
{
    constexpr int THREADS = row_threads(PX, NB);
    const size_t smem = (size_t)row_smem_bytes<T>(PX, NB, THREADS);
    auto kern = k_row_fwd<T, PX, NB, THREADS, BATCH, EDGE>;
    SG_TRY(smem_limit(kern, smem));
    const int ny = BATCH ? bs.maxny : one.src.ny;
    dim3 grid((ny + 2 * NB - 1) / (2 * NB) + (EDGE == EDGE_INSIDE ? 1 : 0), nf, BATCH ? bs.nmem : 1);
    edge_args<T> e = {};
    if (EDGE == EDGE_INSIDE && ed) e = *ed;
    SG_CUDA_TRY(sg_launch_dep(kern, grid, dim3(THREADS), smem, st, one, many, e, ed_many, tw));
    SG_CUDA_TRY(cudaGetLastError());
    return SG_OK;
}

template <typename T, int PX, int NB>
sg_status launch_rows_fwd_any(const row_fwd_args<T> &one, const row_fwd_args<T> *many, const edge_args<T> *ed,
                              const edge_args<T> *ed_many, batch_shape bs, int nf, const cplx_t<T> *tw, cudaStream_t st,
                              int edge)
{
#define SG_ROWS(E)                                                                                       \
    return many ? launch_rows_fwd<T, PX, NB, true, E>(one, many, ed, ed_many, bs, nf, tw, st)            \
                : launch_rows_fwd<T, PX, NB, false, E>(one, many, ed, ed_many, bs, nf, tw, st)
    if constexpr (edge_inside(PX, PX)) {
        if (edge == EDGE_INSIDE) { SG_ROWS(EDGE_INSIDE); }
    }
    if (edge == EDGE_BEFORE) { SG_ROWS(EDGE_BEFORE); }
    SG_ROWS(EDGE_NONE);
#undef SG_ROWS
}

template <typename T, int PX>
sg_status rows_fwd_px(int nb, const row_fwd_args<T> &one, const row_fwd_args<T> *many, batch_shape bs, int nf,
                      const cplx_t<T> *tw, cudaStream_t st, int edge, const edge_args<T> *ed, const edge_args<T> *ed_many)
{
    constexpr int D = row_nb_default(PX);
    constexpr int A = shape_candidate(D, 0), C = shape_candidate(D, 2);
    if (nb == D) return launch_rows_fwd_any<T, PX, D>(one, many, ed, ed_many, bs, nf, tw, st, edge);
    if constexpr (row_feasible_t<T>(PX, A)) {
        if (nb == A) return launch_rows_fwd_any<T, PX, A>(one, many, ed, ed_many, bs, nf, tw, st, edge);
    }
    if constexpr (row_feasible_t<T>(PX, C)) {
        if (nb == C) return launch_rows_fwd_any<T, PX, C>(one, many, ed, ed_many, bs, nf, tw, st, edge);
    }
    return SG_EINVAL;
}

}  // namespace

template <typename T>
sg_status rows_fwd(int px, int nb, const row_fwd_args<T> &one, int nf, const cplx_t<T> *tw, cudaStream_t st,
                   const row_fwd_args<T> *many, batch_shape bs, int edge, const edge_args<T> *ed,
                   const edge_args<T> *ed_many)
{
    SG_PAD_SWITCH(px, return (rows_fwd_px<T, PP>(nb, one, many, bs, nf, tw, st, edge, ed, ed_many)));
    return SG_EINVAL;
}

}  // namespace sgk
