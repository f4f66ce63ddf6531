// Solver state and the vector work of an RRCG iteration as functors of the row passes
// (prologues of the forward rows, epilogues of the inverse ones).
#pragma once
#include <math.h>
#include <stddef.h>

#include "fast512.cuh"

namespace gj {

struct SolverDev {
    int k, done, status, pending_update;
    int sat[2];
    int kmax, stop_on_chi2, per_field;
    int anchor;           // GJ_ANCHOR_*
    int gspace;           // GJ_GRAMIAN_*
    int p[2];
    double eps2;
    double alpha[2], q[2], alpha_min[2], lam[2], lo[2], hi[2];
    double chi2_target[2];
    double s[2], beta[2];
    double ll_prev[2];
    double phi_last[2], SG_last;
    // accumulators, zeroed after use
    double G[3];          // (m1,m1), (m2,m2), (m1,m2) of the current models
    double phi[2];        // ||r~||^2
    double ll[2];         // ||l||^2
    double pl[2], pp[2];  // (p,l), ||p||^2
    double qq[2];         // ||A~ p||^2
    gj_rrcg_hist *hist;
};

template <typename R>
struct FieldVecs {
    R *m[2];
    R *p[2];
    R *l[2];
    R *v[2];               // W_d r~ (s values)
    const R *wd[2];        // 1 / sigma
    const R *dobs[2];
    const R *mapr[2];      // may be null
    const R *wdep[2];      // nz values
    const R *iwdep[2];     // 1 / wdep, nz values
    const R *whard[2];     // may be null
    R *mtp[2];             // W_{k-1} m_{k-1} (previous-model anchor only), else null
};

// The L1 reweighting factor of Eq. WL and its reciprocal for p = 1 (1 for p = 2):
// ((m - m_apr)^2 + eps^2)^(-1/4) and ((m - m_apr)^2 + eps^2)^(1/4).
template <typename R> __device__ __forceinline__ void lp_factors(int p, R d, R eps2, R &wl, R &inv_wl);
// FP64: two reciprocal square roots, u = q^-2, q = (d^2 + eps^2) u, q^-1/2 (a square root, a
// reciprocal one and a division by the weight took twice the FP64 instructions)
template <>
__device__ __forceinline__ void lp_factors<double>(int p, double d, double eps2, double &wl, double &inv_wl) {
    if (p == 1) {
        const double x = d * d + eps2, q = x * rsqrt(x);
        wl = rsqrt(q);
        inv_wl = q * wl;
    } else {
        wl = 1.0;
        inv_wl = 1.0;
    }
}
// One hardware reciprocal square root (relative error about 1e-7; arguments below
// FLT_MIN flush to zero).  Its arguments here are d^2 + eps^2 and (d^2 + eps^2)^-1/2.
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// FP32: two reciprocal square roots, u = q^-1/2, q^1/4 = u^-1/2, q^-1/4 = u q^1/4
template <>
__device__ __forceinline__ void lp_factors<float>(int p, float d, float eps2, float &wl, float &inv_wl) {
    if (p == 1) {
        const float u = rsqrt_approx(d * d + eps2);
        inv_wl = rsqrt_approx(u);
        wl = u * inv_wl;
    } else {
        wl = 1.0f;
        inv_wl = 1.0f;
    }
}

// The general kernels' form: FP32 keeps the full range of eps^2 (no flush of small arguments).
template <typename R>
__device__ __forceinline__ void lp_factors_full(int p, R d, R eps2, R &wl, R &inv_wl) { lp_factors<R>(p, d, eps2, wl, inv_wl); }
template <>
__device__ __forceinline__ void lp_factors_full<float>(int p, float d, float eps2, float &wl, float &inv_wl) {
    if (p == 1) {
        const float q = sqrtf(d * d + eps2);
        wl = rsqrtf(q);
        inv_wl = sqrtf(q);
    } else {
        wl = 1.0f;
        inv_wl = 1.0f;
    }
}

// The solver scalars that a pass uses, in precision R, for every thread: lane i of one warp
// reads and converts scalar(i) (a conversion is FP64 work), the block shares them, and
// set() takes them.  Functors with NS scalars inherit init() from here (all threads call it);
// the general kernels take the steps apart, so that these loads overlap with the data's.
template <class Fn>
__device__ __forceinline__ void init_scalars(Fn &fn) {
    using R = typename Fn::Real;
    __shared__ R sh[Fn::NS > 0 ? Fn::NS : 1];
    if constexpr (Fn::NS > 0) {
        if (threadIdx.x < Fn::NS) sh[threadIdx.x] = fn.scalar((int)threadIdx.x);
        __syncthreads();
    }
    fn.set(sh);
}

// Forward of m with the pending model update (RRCG:7-8 and the bounds) and the
// Gramian sums of the updated models.
template <typename R, bool OPT = true>
struct ProModel {
    FieldVecs<R> F;
    SolverDev *S;
    int nx, ny;
    // per-thread
    int upd, pw[2], gsp;
    R s[2], lo[2], hi[2], eps2;
    R acc[3];
    using Real = R;
    static constexpr int NS = 7;
    __device__ __forceinline__ R scalar(int i) const {
        return (R)*(i < 2 ? S->s + i : i < 4 ? S->lo + (i - 2) : i < 6 ? S->hi + (i - 4) : &S->eps2);
    }
    __device__ __forceinline__ void begin() {  // what load() needs, and the other integers
        upd = S->pending_update;
        gsp = S->gspace;
        for (int i = 0; i < 2; ++i) pw[i] = S->p[i];
    }
    __device__ __forceinline__ void set(const R *v) {
        eps2 = v[6];
        for (int i = 0; i < 2; ++i) { s[i] = v[i]; lo[i] = v[2 + i]; hi[i] = v[4 + i]; }
        acc[0] = acc[1] = acc[2] = 0;
    }
    __device__ void init() {
        begin();
        init_scalars(*this);
    }
    // the general kernels' per-element form in two steps, so that the loads of several elements
    // are in flight before the first store
    struct Raw { R m[2], p[2], wh[2], ma[2]; };
    __device__ __forceinline__ Raw load(int la, int, bool, int j) const {
        const size_t c = (size_t)la * nx + j;
        Raw q;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            q.m[i] = F.m[i][c];
            q.p[i] = F.p[i][c];  // (zero before the first direction; unconditional, so that no load waits for upd)
            q.wh[i] = (OPT && F.whard[i]) ? F.whard[i][c] : R(1);
            q.ma[i] = (OPT && F.mapr[i]) ? F.mapr[i][c] : R(0);
        }
        return q;
    }
    __device__ __forceinline__ void apply(const Raw &q, int la, int, bool, int j, R &a, R &b) {
        const size_t c = (size_t)la * nx + j;
        const int r = la / ny;
        R mv[2], gv[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            R mi = q.m[i], wl, iwl;
            if (upd) {
                lp_factors_full<R>(pw[i], mi - q.ma[i], eps2, wl, iwl);
                R inv_w = iwl * F.iwdep[i][r];
                if (OPT && F.whard[i]) inv_w /= q.wh[i];
                if (OPT && F.mtp[i]) F.mtp[i][c] = F.wdep[i][r] * q.wh[i] * wl * mi;  // W_k m_k, the next anchor
                mi = mi - s[i] * q.p[i] * inv_w;
                mi = fmin(fmax(mi, lo[i]), hi[i]);
                F.m[i][c] = mi;
            }
            mv[i] = gv[i] = mi;
            if (gsp) {  // the Gramian of the weighted models
                lp_factors_full<R>(pw[i], mi - q.ma[i], eps2, wl, iwl);
                gv[i] = F.wdep[i][r] * q.wh[i] * wl * mi;
            }
        }
        acc[0] += gv[0] * gv[0];
        acc[1] += gv[1] * gv[1];
        acc[2] += gv[0] * gv[1];
        a = mv[0];
        b = mv[1];
    }
    __device__ __forceinline__ void fetch(int la, int lb, bool hb, int j, R &a, R &b) {
        apply(load(la, lb, hb, j), la, lb, hb, j, a, b);
    }
    // rows a line needs in every launch (m, p), staged ahead by the persistent row
    // pass as pre[a][field][j]; the optional rows are read in place
    static constexpr int NPRE = 2;
    __device__ const R *pre_src(int a, int i) const { return a == 0 ? F.m[i] : (upd ? F.p[i] : nullptr); }
    // batched form: every load of the K elements is issued before any store
    template <int K, bool PRE = false>
    __device__ __forceinline__ void fetch_batch(int la, int, bool, int j0, int stride, int n, R (&a)[K], R (&b)[K],
                                                const R *pre = nullptr) {
        const size_t c0 = (size_t)la * nx;
        const int r = la / ny;
        R mv[2][K], pv[2][K], wh[2][K], ma[2][K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = j0 + k * stride;
            const bool ok = j < n;
            const size_t c = c0 + j;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                mv[i][k] = ok ? (PRE ? pre[i * f512::H + j] : F.m[i][c]) : R(0);
                pv[i][k] = (ok && upd) ? (PRE ? pre[(2 + i) * f512::H + j] : F.p[i][c]) : R(0);
                wh[i][k] = (ok && OPT && F.whard[i]) ? F.whard[i][c] : R(1);
                ma[i][k] = (ok && OPT && F.mapr[i]) ? F.mapr[i][c] : R(0);
            }
        }
        R wd[2], iwd[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) { wd[i] = F.wdep[i][r]; iwd[i] = F.iwdep[i][r]; }
        if (upd) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int j = j0 + k * stride;
                if (j >= n) continue;
                const size_t c = c0 + j;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    R wl, iwl;
                    lp_factors<R>(pw[i], mv[i][k] - ma[i][k], eps2, wl, iwl);
                    R inv_w = iwl * iwd[i];
                    if (OPT && F.whard[i]) inv_w /= wh[i][k];
                    if (OPT && F.mtp[i]) F.mtp[i][c] = wd[i] * wh[i][k] * wl * mv[i][k];  // W_k m_k, the next anchor
                    R mi = mv[i][k] - s[i] * pv[i][k] * inv_w;
                    mi = fmin(fmax(mi, lo[i]), hi[i]);
                    F.m[i][c] = mi;
                    mv[i][k] = mi;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            R gv[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                gv[i] = mv[i][k];
                if (gsp) {  // the Gramian of the weighted models W(m) m
                    R wl, iwl;
                    lp_factors<R>(pw[i], mv[i][k] - ma[i][k], eps2, wl, iwl);
                    gv[i] = wd[i] * wh[i][k] * wl * mv[i][k];
                }
            }
            acc[0] += gv[0] * gv[0];
            acc[1] += gv[1] * gv[1];
            acc[2] += gv[0] * gv[1];
            a[k] = mv[0][k];
            b[k] = mv[1][k];
        }
    }
    __device__ void flush(double *red) { block_accumulate<3>(acc, S->G, red); }
};

// The data-line epilogues: a launch serves both fields (grid y), a transform two lines la
// and lb of one of them, which field_functor(epi, field) selects; hb: line lb exists.

// Residual epilogue: r~ = W_d (A m - d), v = W_d r~, Phi partials (RRCG:1).
template <typename R>
struct EpiResidual {
    FieldVecs<R> F;
    SolverDev *S;
    int sx;
    int fld;
    R acc;
    using Real = R;
    static constexpr int NS = 0;
    __device__ __forceinline__ R scalar(int) const { return R(0); }
    __device__ __forceinline__ void begin() {}
    __device__ __forceinline__ void set(const R *) { acc = 0; }
    __device__ void init() { set(nullptr); }
    __device__ __forceinline__ const R *wd() const { return fld ? F.wd[1] : F.wd[0]; }  // (selects, not indexed loads)
    __device__ __forceinline__ const R *dobs() const { return fld ? F.dobs[1] : F.dobs[0]; }
    // y of both lines in a, b becomes W_d r~ (two steps, as in ProModel)
    struct Raw { R w[2], d[2]; };
    __device__ __forceinline__ Raw load(int la, int lb, bool hb, int j) const {
        const size_t t = (size_t)la * sx + j, u = (size_t)(hb ? lb : la) * sx + j;
        return Raw{{wd()[t], wd()[u]}, {dobs()[t], dobs()[u]}};
    }
    __device__ __forceinline__ void residual(const Raw &q, bool hb, R &a, R &b) {
        const R r0 = q.w[0] * (a - q.d[0]), r1 = hb ? q.w[1] * (b - q.d[1]) : R(0);
        acc += r0 * r0;
        acc += r1 * r1;
        a = q.w[0] * r0;
        b = q.w[1] * r1;
    }
    __device__ __forceinline__ void store(int la, int lb, bool hb, int j, R a, R b) {
        residual(load(la, lb, hb, j), hb, a, b);
        R *v = fld ? F.v[1] : F.v[0];
        v[(size_t)la * sx + j] = a;
        if (hb) v[(size_t)lb * sx + j] = b;
    }
    // fused form, in two steps so that the loads can be issued before the transform:
    // resid_load fetches W_d and d (zero where there is no element); resid_apply takes y of
    // both lines in a, b and returns v = W_d r~
    template <int K>
    __device__ __forceinline__ void resid_load(int la, int lb, bool hb, int j0, int stride, int n, R (&w)[2][K],
                                               R (&d)[2][K]) const {
        const R *w0 = wd() + (size_t)la * sx, *w1 = wd() + (size_t)lb * sx;
        const R *d0 = dobs() + (size_t)la * sx, *d1 = dobs() + (size_t)lb * sx;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = j0 + k * stride;
            const bool ok = j < n;
            w[0][k] = ok ? w0[j] : R(0);
            d[0][k] = ok ? d0[j] : R(0);
            w[1][k] = ok && hb ? w1[j] : R(0);
            d[1][k] = ok && hb ? d1[j] : R(0);
        }
    }
    template <int K>
    __device__ __forceinline__ void resid_apply(int j0, int stride, int n, bool hb, const R (&w)[2][K], const R (&d)[2][K],
                                                R (&a)[K], R (&b)[K]) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = j0 + k * stride;
            const bool ok = j < n;
            const R r0 = w[0][k] * (a[k] - d[0][k]);
            const R r1 = w[1][k] * (b[k] - d[1][k]);
            if (ok) acc += r0 * r0;
            if (ok && hb) acc += r1 * r1;
            a[k] = ok ? w[0][k] * r0 : R(0);
            b[k] = ok && hb ? w[1][k] * r1 : R(0);
        }
    }
    __device__ void flush(double *red) { block_accumulate<1>(&acc, S->phi + fld, red); }
};
template <typename R>
__device__ __forceinline__ EpiResidual<R> &field_functor(EpiResidual<R> &p, int f) {
    p.fld = f;
    return p;
}

// Gradient epilogue (RRCG:2-4): l = W^-1 A^T v + alpha (W m - W m_apr) + lambda l_G.
template <typename R, bool OPT = true>
struct EpiGradient {
    FieldVecs<R> F;
    SolverDev *S;
    int nx, ny;
    R alpha[2], lam[2], eps2, g11, g22, g12;
    int pw[2], gsp, prev;
    R acc[2];
    using Real = R;
    static constexpr int NS = 8;
    __device__ __forceinline__ R scalar(int i) const {
        return (R)*(i < 2 ? S->alpha + i : i < 4 ? S->lam + (i - 2) : i < 7 ? S->G + (i - 4) : &S->eps2);
    }
    __device__ __forceinline__ void begin() {
        gsp = S->gspace;
        prev = S->anchor == GJ_ANCHOR_PREVIOUS && S->k > 0;  // W_{k-1} m_{k-1} exists from k = 1
        for (int i = 0; i < 2; ++i) pw[i] = S->p[i];
    }
    __device__ __forceinline__ void set(const R *v) {
        for (int i = 0; i < 2; ++i) { alpha[i] = v[i]; lam[i] = v[2 + i]; }
        eps2 = v[7];
        g11 = v[4]; g22 = v[5]; g12 = v[6];
        acc[0] = acc[1] = 0;
    }
    __device__ void init() {
        begin();
        init_scalars(*this);
    }
    struct Raw { R m[2], wh[2], ma[2], an[2]; };
    __device__ __forceinline__ Raw load(int la, int, bool, int j) const {
        const size_t c = (size_t)la * nx + j;
        Raw q;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            q.m[i] = F.m[i][c];
            q.wh[i] = (OPT && F.whard[i]) ? F.whard[i][c] : R(1);
            q.ma[i] = (OPT && F.mapr[i]) ? F.mapr[i][c] : R(0);
            q.an[i] = (OPT && prev) ? F.mtp[i][c] : R(0);
        }
        return q;
    }
    __device__ __forceinline__ void apply(const Raw &q, int la, int, bool, int j, R a, R b) {
        const size_t c = (size_t)la * nx + j;
        const int r = la / ny;
        R w[2], inv_w[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            R wl, iwl;
            lp_factors_full<R>(pw[i], q.m[i] - q.ma[i], eps2, wl, iwl);
            w[i] = F.wdep[i][r] * wl;
            inv_w[i] = iwl * F.iwdep[i][r];
            if (OPT && F.whard[i]) { w[i] *= q.wh[i]; inv_w[i] /= q.wh[i]; }
        }
        // ascent directions in the chosen space (RRCG:2-3 or Eq. steepestascenta/b)
        const R u0 = gsp ? w[0] * q.m[0] : q.m[0], u1 = gsp ? w[1] * q.m[1] : q.m[1];
        const R lG[2] = {g22 * u0 - g12 * u1, g11 * u1 - g12 * u0};
        const R g[2] = {a, b};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const R anchor = (OPT && prev) ? q.an[i] : w[i] * q.ma[i];
            const R li = g[i] * inv_w[i] + alpha[i] * (w[i] * q.m[i] - anchor) + lam[i] * lG[i];
            F.l[i][c] = li;
            acc[i] += li * li;
        }
    }
    __device__ __forceinline__ void store(int la, int lb, bool hb, int j, R a, R b) {
        apply(load(la, lb, hb, j), la, lb, hb, j, a, b);
    }
    static constexpr int NPRE = 1;  // m, staged ahead by the persistent row pass
    __device__ const R *pre_src(int, int i) const { return F.m[i]; }
    template <int K, bool PRE = false>
    __device__ __forceinline__ void store_batch(int la, int, bool, int j0, int stride, int n, const R (&a)[K],
                                                const R (&b)[K], const R *pre = nullptr) {
        const size_t c0 = (size_t)la * nx;
        const int r = la / ny;
        R mv[2][K], wh[2][K], ma[2][K], an[2][K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = j0 + k * stride;
            const bool ok = j < n;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                mv[i][k] = ok ? (PRE ? pre[i * f512::H + j] : F.m[i][c0 + j]) : R(0);
                wh[i][k] = (ok && OPT && F.whard[i]) ? F.whard[i][c0 + j] : R(1);
                ma[i][k] = (ok && OPT && F.mapr[i]) ? F.mapr[i][c0 + j] : R(0);
                an[i][k] = (ok && OPT && prev) ? F.mtp[i][c0 + j] : R(0);
            }
        }
        R wd[2], iwd[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) { wd[i] = F.wdep[i][r]; iwd[i] = F.iwdep[i][r]; }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = j0 + k * stride;
            if (j >= n) continue;
            R w[2], inv_w[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                R wl, iwl;
                lp_factors<R>(pw[i], mv[i][k] - ma[i][k], eps2, wl, iwl);
                w[i] = wd[i] * wl;
                inv_w[i] = iwl * iwd[i];
                if (OPT && F.whard[i]) { w[i] *= wh[i][k]; inv_w[i] /= wh[i][k]; }
            }
            const R u0 = gsp ? w[0] * mv[0][k] : mv[0][k], u1 = gsp ? w[1] * mv[1][k] : mv[1][k];
            const R lG[2] = {g22 * u0 - g12 * u1, g11 * u1 - g12 * u0};
            const R g[2] = {a[k], b[k]};
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const R anchor = (OPT && prev) ? an[i][k] : w[i] * ma[i][k];
                const R li = g[i] * inv_w[i] + alpha[i] * (w[i] * mv[i][k] - anchor) + lam[i] * lG[i];
                F.l[i][c0 + j] = li;
                acc[i] += li * li;
            }
        }
    }
    __device__ void flush(double *red) { block_accumulate<2>(acc, S->ll, red); }
};

// Search direction (RRCG:5) and the forward input W^-1 p.
template <typename R, bool OPT = true>
struct ProDirection {
    FieldVecs<R> F;
    SolverDev *S;
    int nx, ny;
    R beta[2], eps2;
    int first, pw[2];
    R acc[4];  // (p,l)_0, (p,l)_1, ||p||^2_0, ||p||^2_1
    using Real = R;
    static constexpr int NS = 3;
    __device__ __forceinline__ R scalar(int i) const {
        if (i == 2) return (R)S->eps2;
        const double num = S->per_field ? S->ll[i] : S->ll[0] + S->ll[1];
        const double den = S->per_field ? S->ll_prev[i] : S->ll_prev[0] + S->ll_prev[1];
        return den > 0 ? (R)(num / den) : R(0);
    }
    __device__ __forceinline__ void begin() {
        first = S->k == 0;
        for (int i = 0; i < 2; ++i) pw[i] = S->p[i];
    }
    __device__ __forceinline__ void set(const R *v) {
        beta[0] = v[0];
        beta[1] = v[1];
        eps2 = v[2];
        acc[0] = acc[1] = acc[2] = acc[3] = 0;
    }
    __device__ void init() {
        begin();
        init_scalars(*this);
    }
    struct Raw { R l[2], p[2], m[2], wh[2], ma[2]; };
    __device__ __forceinline__ Raw load(int la, int, bool, int j) const {
        const size_t c = (size_t)la * nx + j;
        Raw q;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            q.l[i] = F.l[i][c];
            q.p[i] = F.p[i][c];
            q.m[i] = F.m[i][c];
            q.wh[i] = (OPT && F.whard[i]) ? F.whard[i][c] : R(1);
            q.ma[i] = (OPT && F.mapr[i]) ? F.mapr[i][c] : R(0);
        }
        return q;
    }
    __device__ __forceinline__ void apply(const Raw &q, int la, int, bool, int j, R &a, R &b) {
        const size_t c = (size_t)la * nx + j;
        const int r = la / ny;
        R x[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const R pi = first ? q.l[i] : q.l[i] + beta[i] * q.p[i];
            R wl, iwl;
            lp_factors_full<R>(pw[i], q.m[i] - q.ma[i], eps2, wl, iwl);
            R inv_w = iwl * F.iwdep[i][r];
            if (OPT && F.whard[i]) inv_w /= q.wh[i];
            F.p[i][c] = pi;
            acc[i] += pi * q.l[i];
            acc[2 + i] += pi * pi;
            x[i] = pi * inv_w;
        }
        a = x[0];
        b = x[1];
    }
    __device__ __forceinline__ void fetch(int la, int lb, bool hb, int j, R &a, R &b) {
        apply(load(la, lb, hb, j), la, lb, hb, j, a, b);
    }
    static constexpr int NPRE = 3;  // l, p, m, staged ahead by the persistent row pass
    __device__ const R *pre_src(int a, int i) const {
        return a == 0 ? F.l[i] : (a == 1 ? (first ? nullptr : F.p[i]) : F.m[i]);
    }
    template <int K, bool PRE = false>
    __device__ __forceinline__ void fetch_batch(int la, int, bool, int j0, int stride, int n, R (&a)[K], R (&b)[K],
                                                const R *pre = nullptr) {
        const size_t c0 = (size_t)la * nx;
        const int r = la / ny;
        R lv[2][K], pv[2][K], mv[2][K], wh[2][K], ma[2][K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = j0 + k * stride;
            const bool ok = j < n;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                lv[i][k] = ok ? (PRE ? pre[i * f512::H + j] : F.l[i][c0 + j]) : R(0);
                pv[i][k] = (ok && !first) ? (PRE ? pre[(2 + i) * f512::H + j] : F.p[i][c0 + j]) : R(0);
                mv[i][k] = ok ? (PRE ? pre[(4 + i) * f512::H + j] : F.m[i][c0 + j]) : R(0);
                wh[i][k] = (ok && OPT && F.whard[i]) ? F.whard[i][c0 + j] : R(1);
                ma[i][k] = (ok && OPT && F.mapr[i]) ? F.mapr[i][c0 + j] : R(0);
            }
        }
        R iwd[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) iwd[i] = F.iwdep[i][r];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = j0 + k * stride;
            const bool ok = j < n;
            R x[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const R pi = first ? lv[i][k] : lv[i][k] + beta[i] * pv[i][k];
                R wl, iwl;
                lp_factors<R>(pw[i], mv[i][k] - ma[i][k], eps2, wl, iwl);
                R inv_w = iwl * iwd[i];
                if (OPT && F.whard[i]) inv_w /= wh[i][k];
                if (ok) {
                    F.p[i][c0 + j] = pi;
                    acc[i] += pi * lv[i][k];
                    acc[2 + i] += pi * pi;
                }
                x[i] = ok ? pi * inv_w : R(0);
            }
            a[k] = x[0];
            b[k] = x[1];
        }
    }
    __device__ void flush(double *red) {
        // pl and pp are adjacent in SolverDev: one pass adds all four sums
        static_assert(offsetof(SolverDev, pp) == offsetof(SolverDev, pl) + 2 * sizeof(double), "layout");
        block_accumulate<4>(acc, S->pl, red);
    }
};

// ||A~ p||^2 = ||W_d A (W^-1 p)||^2 partials (RRCG:6).
template <typename R>
struct EpiQNorm {
    FieldVecs<R> F;
    SolverDev *S;
    int sx;
    int fld;
    R acc;
    using Real = R;
    static constexpr int NS = 0;
    __device__ __forceinline__ R scalar(int) const { return R(0); }
    __device__ __forceinline__ void begin() {}
    __device__ __forceinline__ void set(const R *) { acc = 0; }
    __device__ void init() { set(nullptr); }
    __device__ __forceinline__ const R *wd() const { return fld ? F.wd[1] : F.wd[0]; }
    struct Raw { R w[2]; };
    __device__ __forceinline__ Raw load(int la, int lb, bool hb, int j) const {
        return Raw{{wd()[(size_t)la * sx + j], wd()[(size_t)(hb ? lb : la) * sx + j]}};
    }
    __device__ __forceinline__ void apply(const Raw &q, int, int, bool hb, int, R a, R b) {
        const R q0 = q.w[0] * a, q1 = hb ? q.w[1] * b : R(0);
        acc += q0 * q0;
        acc += q1 * q1;
    }
    __device__ __forceinline__ void store(int la, int lb, bool hb, int j, R a, R b) {
        apply(load(la, lb, hb, j), la, lb, hb, j, a, b);
    }
    // batched form (the 512 kernels): prefetch loads W_d of lines la and lb, elements
    // lane + 32 k, before the transform; store_batch(j0 = lane or lane + 128) uses them
    R wq[2][8];
    __device__ __forceinline__ void prefetch(int la, int lb, bool hb, int lane, int n) {
        const R *w0 = wd() + (size_t)la * sx, *w1 = wd() + (size_t)lb * sx;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int j = lane + 32 * k;
            wq[0][k] = j < n ? w0[j] : R(0);
            wq[1][k] = j < n && hb ? w1[j] : R(0);
        }
    }
    template <int K>
    __device__ __forceinline__ void store_batch(int, int, bool hb, int j0, int stride, int n, const R (&a)[K],
                                                const R (&b)[K]) {
        const int o = (j0 - (int)(threadIdx.x & 31)) / 32;  // 0 or 4
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = j0 + k * stride;
            if (j >= n) continue;
            const R q0 = wq[0][o + k] * a[k];
            acc += q0 * q0;
            if (!hb) continue;
            const R q1 = wq[1][o + k] * b[k];
            acc += q1 * q1;
        }
    }
    __device__ void flush(double *red) { block_accumulate<1>(&acc, S->qq + fld, red); }
};
template <typename R>
__device__ __forceinline__ EpiQNorm<R> &field_functor(EpiQNorm<R> &p, int f) {
    p.fld = f;
    return p;
}

}  // namespace gj
