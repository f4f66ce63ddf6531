// Definitions of the general kernels' launches (general_launch.cuh).
#pragma once
#include "general_launch.cuh"

namespace gj {

template <typename R, class Pro> void gen_row_fwd_attr() { allow_max_smem(k_row_fwd<R, Pro>); }
template <typename R, class Epi> void gen_row_inv_attr() { allow_max_smem(k_row_inv<R, Epi>); }
template <typename R, class Epi> void gen_row_resid_attr() { allow_max_smem(k_row_resid<R, Epi>); }
template <typename R> void gen_col_attr() {
    allow_max_smem(k_col_fwd<R>);
    allow_max_smem(k_col_adj<R>);
}

// (every launch may start while the kernel before it drains: launch_after)
template <typename R, class Pro>
void gen_row_fwd(const gj_op *o, const OpView<R> &v, const PairMap &pm, int n_in, cpx<R> *out0, cpx<R> *out1,
                 const Pro &pro, const int *done, cudaStream_t st, int nf) {
    const int np = pm.joint ? pm.nlines : (pm.nlines + 1) / 2;
    const RowShape rs = row_shape(o, (long long)np * nf, sizeof(cpx<R>));
    launch_after(k_row_fwd<R, Pro>, dim3((np + rs.P - 1) / rs.P, nf), dim3(row_threads(o->px, rs.P, (long long)np * nf)),
                 row_smem(o->Nx, rs.pitch, sizeof(cpx<R>)), st, v, pm, n_in, rs, out0, out1, pro, done);
}
template <typename R, class Epi>
void gen_row_inv(const gj_op *o, const OpView<R> &v, const PairMap &pm, int n_out, const cpx<R> *in0,
                 const cpx<R> *in1, const Epi &epi, const int *done, cudaStream_t st, int nf) {
    const int np = pm.joint ? pm.nlines : (pm.nlines + 1) / 2;
    const RowShape rs = row_shape(o, (long long)np * nf, sizeof(cpx<R>));
    launch_after(k_row_inv<R, Epi>, dim3((np + rs.P - 1) / rs.P, nf), dim3(row_threads(o->px, rs.P, (long long)np * nf)),
                 row_smem(o->Nx, rs.pitch, sizeof(cpx<R>)), st, v, pm, n_out, rs, in0, in1, epi, done);
}
template <typename R, class Epi>
void gen_row_resid(const gj_op *o, const OpView<R> &v, const PairMap &pm, int n_out, const cpx<R> *in0,
                   const cpx<R> *in1, cpx<R> *out0, cpx<R> *out1, const Epi &epi, const int *done, cudaStream_t st,
                   int nf) {
    const int np = (pm.nlines + 1) / 2;
    const RowShape rs = row_shape(o, (long long)np * nf, sizeof(cpx<R>));
    launch_after(k_row_resid<R, Epi>, dim3((np + rs.P - 1) / rs.P, nf),
                 dim3(row_threads(o->px, rs.P, (long long)np * nf)), row_smem(o->Nx, rs.pitch, sizeof(cpx<R>)), st, v, pm, n_out, rs, in0, in1, out0, out1, epi, done);
}
template <typename R>
void gen_col_fwd(const gj_op *o, const OpView<R> &v0, const OpView<R> &v1, int nf, int layers, const int *done,
                 cudaStream_t st) {
    const ColShape s = col_shape(o, nf, layers, sizeof(cpx<R>), false);
    launch_after(k_col_fwd<R>, dim3((o->ncol + s.C - 1) / s.C, (layers + s.L - 1) / s.L, nf),
                 dim3(gen_threads(o->py.mmax, s.C * s.G)), col_smem(o->Ny, s.pitch, s.pitch, sizeof(cpx<R>)), st, v0, v1,
                 s, done);
}
template <typename R>
void gen_col_adj(const gj_op *o, const OpView<R> &v0, const OpView<R> &v1, int nf, int layers, const int *done,
                 cudaStream_t st) {
    const ColShape s = col_shape(o, nf, layers, sizeof(cpx<R>), true);
    launch_after(k_col_adj<R>, dim3((o->ncol + s.C - 1) / s.C, (layers + s.L - 1) / s.L, nf),
                 dim3(gen_threads(o->py.mmax, s.C * s.G)), col_smem(o->Ny, s.pitch, s.pitch1, sizeof(cpx<R>)), st, v0, v1,
                 s, done);
}
template <typename R> void gen_rec_attr() {
    allow_max_smem(k_col_rec_fwd<R>);
    allow_max_smem(k_col_rec_adj<R>);
    allow_max_smem(k_col_plane<R, false>);
    allow_max_smem(k_col_plane<R, true>);
}
template <typename R> void gen_rec_fwd(const gj_op *o, const OpView<R> &v, int r, cudaStream_t st) {
    const RecShape s = rec_shape(o->py, o->even_rows, sizeof(cpx<R>));
    launch_after(k_col_rec_fwd<R>, dim3((o->ncol + s.C - 1) / s.C), dim3(gen_threads(o->py.mmax, s.C)),
                 rec_smem(s, o->Ny, sizeof(cpx<R>)), st, v, s, recompute_rows_out(o), recompute_twy64(o), r);
}
template <typename R> void gen_rec_adj(const gj_op *o, const OpView<R> &v, int r, cudaStream_t st) {
    const RecShape s = rec_shape(o->py, o->even_rows, sizeof(cpx<R>));
    launch_after(k_col_rec_adj<R>, dim3((o->ncol + s.C - 1) / s.C), dim3(gen_threads(o->py.mmax, s.C)),
                 rec_smem(s, o->Ny, sizeof(cpx<R>)), st, v, s, recompute_rows_out(o), recompute_twy64(o), r);
}
template <typename R> void gen_rec_plane(const gj_op *o, const OpView<R> &v, bool inverse, cudaStream_t st) {
    const ColShape s = col_shape(o, 1, 1, sizeof(cpx<R>), true);
    launch_after(inverse ? k_col_plane<R, true> : k_col_plane<R, false>, dim3((o->ncol + s.C - 1) / s.C),
                 dim3(gen_threads(o->py.mmax, s.C)), (size_t)(2 * s.pitch1 + 1) * o->Ny * sizeof(cpx<R>), st, v, s);
}

}  // namespace gj

// Explicit instantiations.
#define GJ_ROW_FWD(R, PRO)                                                                                        \
    template void gen_row_fwd_attr<R, PRO>();                                                                     \
    template void gen_row_fwd<R, PRO>(const gj_op *, const OpView<R> &, const PairMap &, int, cpx<R> *, cpx<R> *, \
                                      const PRO &, const int *, cudaStream_t, int);
#define GJ_ROW_INV(R, EPI)                                                                                    \
    template void gen_row_inv_attr<R, EPI>();                                                                 \
    template void gen_row_inv<R, EPI>(const gj_op *, const OpView<R> &, const PairMap &, int, const cpx<R> *, \
                                      const cpx<R> *, const EPI &, const int *, cudaStream_t, int);
#define GJ_ROW_RESID(R, EPI)                                                                                    \
    template void gen_row_resid_attr<R, EPI>();                                                                 \
    template void gen_row_resid<R, EPI>(const gj_op *, const OpView<R> &, const PairMap &, int, const cpx<R> *, \
                                        const cpx<R> *, cpx<R> *, cpx<R> *, const EPI &, const int *, cudaStream_t, \
                                        int);
#define GJ_COLS(R)                                                                                               \
    template void gen_col_attr<R>();                                                                             \
    template void gen_col_fwd<R>(const gj_op *, const OpView<R> &, const OpView<R> &, int, int, const int *,     \
                                 cudaStream_t);                                                                  \
    template void gen_col_adj<R>(const gj_op *, const OpView<R> &, const OpView<R> &, int, int, const int *,     \
                                 cudaStream_t);
#define GJ_RECOMPUTE(R)                                                                     \
    template void gen_rec_attr<R>();                                                        \
    template void gen_rec_fwd<R>(const gj_op *, const OpView<R> &, int, cudaStream_t);      \
    template void gen_rec_adj<R>(const gj_op *, const OpView<R> &, int, cudaStream_t);      \
    template void gen_rec_plane<R>(const gj_op *, const OpView<R> &, bool, cudaStream_t);
