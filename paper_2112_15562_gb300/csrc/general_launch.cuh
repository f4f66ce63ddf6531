// Launch shapes and launches of the general product kernels (any padded size).
#pragma once
#include <algorithm>

#include "view.cuh"

namespace gj {

constexpr int kGenThreads = 256;             // most threads of a CTA
constexpr size_t kGenSmem = 100 * 1024;      // shared memory up to which a shape may grow: two CTAs an SM
constexpr int kGenCtas = 304;                // CTAs worth having in flight: two an SM

inline int gen_threads(int mmax, int lines) {
    const int t = (mmax * lines + 31) / 32 * 32;
    return t < 64 ? 64 : (t > kGenThreads ? kGenThreads : t);
}

// the padded (odd) pitch where it fits the device's shared memory, else the plain one
inline int odd_pitch(int lines) { return lines | 1; }
constexpr size_t kGenSmemMax = 224 * 1024;

// Pairs per CTA of a row pass over npairs line pairs: as many as keep the widest stage
// within the CTA's threads, but not so many that the pass leaves SMs idle.
inline int pick_row_pairs(const FftPlanDev &pl, long long npairs, size_t cs) {
    int P = 1;
    while (P < 16 && 2 * P * pl.mmax <= kGenThreads && (npairs + 2 * P - 1) / (2 * P) >= kGenCtas &&
           row_smem(pl.N, odd_pitch(2 * P), cs) <= kGenSmem)
        P *= 2;
    return P;
}

inline RowShape row_shape_of(const FftPlanDev &pl, int P, size_t cs) {
    RowShape s;
    s.P = P;
    s.pitch = row_smem(pl.N, odd_pitch(P), cs) <= kGenSmemMax ? odd_pitch(P) : P;
    s.mP = div_magic(P);
    return s;
}
// of a pass over npairs line pairs: the operator's P_row when it was tuned or when the
// lines' elements lie apart (transposed intermediates, whose runs are the P lines)
inline RowShape row_shape(const gj_op *o, long long npairs, size_t cs) {
    const bool fixed = o->rows_tuned || o->fast1024;
    return row_shape_of(o->px, fixed ? o->P_row : pick_row_pairs(o->px, npairs, cs), cs);
}

// Layers taken at a time: as many as fill the CTA's threads and fit.
inline int pick_layer_lines(const FftPlanDev &pl, int C, int L, size_t cs) {
    int G = kGenThreads / (pl.mmax * C);
    if (G > L) G = L;
    while (G > 1 && col_smem(pl.N, odd_pitch(C * G), odd_pitch(C * G), cs) > kGenSmem) --G;
    return G < 1 ? 1 : G;
}

// Layers per CTA: all of them when the column tiles alone fill the GPU (the layer sum
// then never leaves the CTA), else so few that the CTAs do, but no fewer than a CTA takes
// at a time.
inline int pick_layers(const FftPlanDev &pl, int C, int tiles, int nz, size_t cs) {
    const int G = pick_layer_lines(pl, C, nz, cs);
    int groups = (kGenCtas + tiles - 1) / tiles;
    if (groups > (nz + G - 1) / G) groups = (nz + G - 1) / G;
    return (nz + groups - 1) / groups;
}

// Columns per CTA: a column tile's rows should fill 32-byte sectors (4 FP32 or 2 FP64
// columns) when there are enough tiles and layers to fill the GPU, one column when not.
inline int pick_col_tile(const FftPlanDev &pl, int ncol, int nz, int nf, size_t cs) {
    int C = 8;
    while (C > 1 && (C * pl.mmax > kGenThreads || col_smem(pl.N, odd_pitch(C), odd_pitch(C), cs) > kGenSmem)) C /= 2;
    while (C > 1) {
        const long long tiles = (long long)((ncol + C - 1) / C) * nf;
        const int G = pick_layer_lines(pl, C, nz, cs);
        if (tiles * ((nz + G - 1) / G) >= kGenCtas) break;
        C /= 2;
    }
    return C;
}

// layers: of the launch (1 in the recompute mode, whose launches share one sum)
inline ColShape col_shape(const gj_op *o, int nf, int layers, size_t cs, bool adjoint) {
    ColShape s;
    s.C = o->cols_tuned ? o->C_col : pick_col_tile(o->py, o->ncol, layers, nf, cs);
    const int tiles = (o->ncol + s.C - 1) / s.C * nf;
    s.L = o->layers_tuned ? std::min(o->L_grp, layers) : pick_layers(o->py, s.C, tiles, layers, cs);
    // the forward sums have room for gen_slots groups
    if (!adjoint && !o->recompute) s.L = std::max(s.L, (layers + o->gen_slots - 1) / o->gen_slots);
    s.G = pick_layer_lines(o->py, s.C, s.L, cs);
    const int B = s.C * s.G;
    const bool pad = col_smem(o->Ny, odd_pitch(B), adjoint ? odd_pitch(s.C) : odd_pitch(B), cs) <= kGenSmemMax;
    s.pitch = pad ? odd_pitch(B) : B;
    s.pitch1 = pad ? odd_pitch(s.C) : s.C;
    s.mB = div_magic(B);
    s.mC = div_magic(s.C);
    s.arrivals = (layers + s.L - 1) / s.L;
    s.serial = o->recompute ? 1 : 0;
    return s;
}

// Launches (general_impl.cuh; instantiated by general_*.cu, one translation unit per
// precision and pass, because a kernel holds every codelet).  The attribute calls are
// made once before a capture.  grid y of the rows: fields (LoadPlain2 / StorePlain2).
template <typename R, class Pro> void gen_row_fwd_attr();
template <typename R, class Pro>
void gen_row_fwd(const gj_op *o, const OpView<R> &v, const PairMap &pm, int n_in, cpx<R> *out0, cpx<R> *out1,
                 const Pro &pro, const int *done, cudaStream_t st, int nf = 1);
template <typename R, class Epi> void gen_row_inv_attr();
template <typename R, class Epi>
void gen_row_inv(const gj_op *o, const OpView<R> &v, const PairMap &pm, int n_out, const cpx<R> *in0,
                 const cpx<R> *in1, const Epi &epi, const int *done, cudaStream_t st, int nf = 1);
template <typename R, class Epi> void gen_row_resid_attr();
template <typename R, class Epi>
void gen_row_resid(const gj_op *o, const OpView<R> &v, const PairMap &pm, int n_out, const cpx<R> *in0,
                   const cpx<R> *in1, cpx<R> *out0, cpx<R> *out1, const Epi &epi, const int *done, cudaStream_t st);
template <typename R> void gen_col_attr();
template <typename R>
void gen_col_fwd(const gj_op *o, const OpView<R> &v0, const OpView<R> &v1, int nf, int layers, const int *done,
                 cudaStream_t st);
template <typename R>
void gen_col_adj(const gj_op *o, const OpView<R> &v0, const OpView<R> &v1, int nf, int layers, const int *done,
                 cudaStream_t st);

}  // namespace gj
