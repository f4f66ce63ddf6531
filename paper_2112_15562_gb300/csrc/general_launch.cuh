// Launch shapes and launches of the general product kernels (any padded size).
#pragma once
#include <algorithm>

#include "view.cuh"

namespace gj {

constexpr int kGenThreads = 256;             // most threads of a CTA
constexpr size_t kGenSmem = 110 * 1024;      // shared memory up to which a shape may grow: two CTAs an SM
constexpr int kGenCtas = 304;                // CTAs worth having in flight: two an SM
constexpr int kGenGroups = 10;               // most layer groups of a column tile (partial sums to keep and to add)

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

// Threads of a row pass: the widest stage's butterflies; when there are few CTAs, enough that
// the staging and epilogue loops are one or two elements long (each is a memory latency).
inline int row_threads(const FftPlanDev &pl, int P, long long npairs) {
    const int t = gen_threads(pl.mmax, P);
    return (npairs + P - 1) / P > kGenCtas ? t : std::max(t, gen_threads((pl.N + 1) / 2, P));
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

// Columns and layers per CTA of a column pass over nz layers of nf fields.  Fixed values
// (from gj_op_tune) are kept when positive.
//
// FP32 passes wait for latencies: four columns fill a 32-byte sector of the spectra and
// intermediates, and two CTAs an SM keep enough in flight; more layer groups only add partial
// sums.  Problems too small for that take one column a CTA.  (Forward / adjoint of both
// fields, us: 148x146x20 at 300x294 48 / 43 so, 53 / 40 with eight columns, 58 / 49 with one;
// 300x200x30 at 400x600 118 / 94, 121 / 103 and 168 / 126 (two).)
//
// FP64 passes are bound by the two FP64 lanes of an SM: the shape with the least work on the
// fullest SM, where a CTA costs its group transforms, one more for the residual (adjoint) or
// a share of the sums (forward), some 2 us of its own, and one or two CTAs of imbalance;
// single columns waste half of each sector.  (Forward of both fields, us: 200x180x20 at
// 360x400 463 with four columns and two layers, 591 with one and ten; 256x256x40 at 512x512
// 1007 with two and five, 1064 with one and twenty.)
struct ColPick { int C, L; };
// FP64 work of B lines relative to full warps on the four schedulers of an SM (half of what a
// CTA leaves idle is taken by the others).
inline double fp64_fill(const FftPlanDev &pl, int B) {
    double f = 0.0;
    for (int s = 0; s < pl.nst; ++s) {
        const int items = pl.st[s].M * B, warps = (items + 31) / 32;
        f += (warps + 3) / 4 * 128.0 / items / pl.nst;
    }
    return 0.5 + 0.5 * f;
}
inline ColPick pick_cols(const FftPlanDev &pl, int ncol, int nz, int nf, size_t cs, bool adjoint, int fixC = 0,
                         int fixL = 0) {
    const bool wide = cs == 16;  // complex doubles
    auto fits = [&](int C) { return col_smem(pl.N, odd_pitch(C), odd_pitch(C), cs) <= kGenSmem; };
    auto tiles_of = [&](int C) { return (ncol + C - 1) / C * nf; };
    ColPick best{fixC > 0 ? fixC : 1, nz};
    if (!wide) {
        if (fixC <= 0) {
            best.C = 4;
            while (best.C > 1 && !fits(best.C)) best.C /= 2;
            const int G = pick_layer_lines(pl, best.C, nz, cs);
            if (tiles_of(best.C) * ((nz + G - 1) / G) < kGenCtas / 2) best.C = 1;
        }
        const int tiles = tiles_of(best.C), G = pick_layer_lines(pl, best.C, nz, cs);
        int groups = std::max(1, (kGenCtas + tiles / 2) / tiles);
        groups = std::min(std::min(groups, kGenGroups), (nz + G - 1) / G);
        best.L = fixL > 0 ? std::min(fixL, nz) : (nz + groups - 1) / groups;
        return best;
    }
    double least = 1e300;
    for (int C = fixC > 0 ? fixC : 1; C <= (fixC > 0 ? fixC : 4); C *= 2) {
        if (fixC <= 0 && C > 1 && (C * pl.mmax > 2 * kGenThreads || C >= 2 * ncol || !fits(C))) break;
        const double waste = C == 1 ? 1.2 : 1.0;
        for (int groups = 1; groups <= nz && groups <= kGenGroups; ++groups) {
            const int L = fixL > 0 ? std::min(fixL, nz) : (nz + groups - 1) / groups;
            const int G = pick_layer_lines(pl, C, L, cs), n = (nz + L - 1) / L;
            const double work = (double)pl.N * C * G * 15.0 / 1900.0 * waste * fp64_fill(pl, C * G);  // microseconds
            const double ctas = tiles_of(C) * n / 152.0;
            const double t = ((L + G - 1) / G + (adjoint ? 1.0 : 0.3)) *
                                 std::max((ctas + (adjoint ? 1.0 : 2.0)) * work, 2.5) +
                             2.0 * ctas + (n > 1 && !adjoint ? 1.5 + 0.2 * n : 0.0);
            if (t < 0.98 * least) { least = t; best = ColPick{C, L}; }
            if (fixL > 0) break;
        }
    }
    return best;
}

inline ColShape col_shape(const gj_op *o, int nf, int layers, size_t cs, bool adjoint) {
    ColShape s;
    const ColPick pick =
        pick_cols(o->py, o->ncol, layers, nf, cs, adjoint, o->cols_tuned ? o->C_col : 0, o->layers_tuned ? o->L_grp : 0);
    s.C = pick.C;
    s.L = pick.L;
    // the forward sums have room for gen_slots groups
    if (!adjoint) s.L = std::max(s.L, (layers + o->gen_slots - 1) / o->gen_slots);
    s.G = pick_layer_lines(o->py, s.C, s.L, cs);
    const int B = s.C * s.G;
    // an odd pitch where it fits; an FP64 adjoint pass takes the space for another CTA instead
    // (256x256x40 at 512x512, both fields: 991 -> 952 us; the forward pass lost, 1007 -> 1045)
    const bool pad = !(adjoint && cs == 16) && col_smem(o->Ny, odd_pitch(B), adjoint ? odd_pitch(s.C) : odd_pitch(B), cs) <= kGenSmemMax;
    s.pitch = pad ? odd_pitch(B) : B;
    s.pitch1 = pad ? odd_pitch(s.C) : s.C;
    s.mB = div_magic(B);
    s.mC = div_magic(s.C);
    s.arrivals = (layers + s.L - 1) / s.L;
    return s;
}

// Launches (general_impl.cuh; instantiated by general_*.cu, one translation unit per
// precision and pass, because a kernel holds every codelet).  The attribute calls are
// made once before a capture.  grid y of the rows: fields (LoadPlain2 / StorePlain2, the
// solver's data-line epilogues).
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
                   const cpx<R> *in1, cpx<R> *out0, cpx<R> *out1, const Epi &epi, const int *done, cudaStream_t st,
                   int nf);
template <typename R> void gen_col_attr();
template <typename R>
void gen_col_fwd(const gj_op *o, const OpView<R> &v0, const OpView<R> &v1, int nf, int layers, const int *done,
                 cudaStream_t st);
template <typename R>
void gen_col_adj(const gj_op *o, const OpView<R> &v0, const OpView<R> &v1, int nf, int layers, const int *done,
                 cudaStream_t st);

// Columns per CTA of the recompute mode's column passes (RecShape): two FP64 lines where
// they fit two CTAs an SM.
inline size_t rec_smem(const RecShape &s, int N, size_t cs) {
    return 2 * (size_t)s.buf + (size_t)N * sizeof(double2) + (size_t)(s.C + 1) * N * cs;
}
inline RecShape rec_shape(const FftPlanDev &pl, bool even, size_t cs) {
    RecShape s;
    s.even = even ? 1 : 0;
    for (s.lines = 2;; s.lines = 1) {
        s.C = even ? 2 * s.lines : s.lines;
        s.buf = pl.N * (int)std::max(s.lines * sizeof(double2), s.C * cs);
        if (s.lines == 1 || (s.lines * pl.mmax <= kGenThreads && rec_smem(s, pl.N, cs) <= kGenSmem)) break;
    }
    s.mC = div_magic(s.C);
    s.mlines = div_magic(s.lines);
    return s;
}

// Recompute mode: layer r's launches after recompute_rows (FP64 rows of the layer's table in
// Zs), and the one transform per product of the residual's or the summed spectrum's columns.
template <typename R> void gen_rec_attr();
template <typename R> void gen_rec_fwd(const gj_op *o, const OpView<R> &v, int r, cudaStream_t st);
template <typename R> void gen_rec_adj(const gj_op *o, const OpView<R> &v, int r, cudaStream_t st);
template <typename R> void gen_rec_plane(const gj_op *o, const OpView<R> &v, bool inverse, cudaStream_t st);

}  // namespace gj
