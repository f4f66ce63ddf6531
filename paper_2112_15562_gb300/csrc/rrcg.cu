// Regularised reweighted CG joint solve (Eq. RRCG:1-8) with Lp reweighting
// (Eq. W, Eq. WL), the Gramian coupling in the original space (RRCG:2-3),
// bounds (Sec. 2.5), the chi^2 stop (Eq. chi2) and the alpha schedule
// (Eq. regpara).  All vector work is fused into the prologues and epilogues of
// the FFT row passes; the scalars stay on the device.
//
// One loop body (iteration k -> k+1), both fields in every launch:
//   adjoint:  rows of v = W_d r~ -> columns -> conj-spectrum columns -> rows with
//             l = W^-1 A^T v + alpha (W m - W m_apr) + lambda l_G      (RRCG:4)
//   forward:  rows of p = l + beta p_prev, x = W^-1 p -> columns -> rows with
//             ||A~ p||^2                                              (RRCG:5-6)
//   scalars:  s = (p, l) / (||A~p||^2 + (alpha + lambda)||p||^2)
//   forward:  rows with m <- clip(m - s W^-1 p) and the Gramian sums -> columns
//             -> rows with r~ = W_d (A m - d), Phi = ||r~||^2          (RRCG:7-8, 1)
//   scalars:  chi^2 flags, alpha freeze/decay, stop flag
// The first forward of m_0 and its scalars run once when the solver is created.
#include <math.h>
#include <stddef.h>

#include <algorithm>
#include <new>
#include <type_traits>
#include <vector>

#include "fast_launch.cuh"
#include "general_launch.cuh"
#include "rrcg_functors.cuh"

namespace gj {

// The one-thread scalar steps run on a shared-memory copy of the solver state: a
// warp copies it in with one coalesced read (instead of a chain of dependent global
// loads), thread 0 takes the step, and the warp copies the state back.
static_assert(sizeof(SolverDev) % sizeof(unsigned long long) == 0 && alignof(SolverDev) == 8,
              "the state copies as 8-byte words");
constexpr int kStateWords = (int)(sizeof(SolverDev) / sizeof(unsigned long long));
__device__ __forceinline__ void state_copy(void *dst, const void *src) {
    for (int i = threadIdx.x; i < kStateWords; i += 32)
        static_cast<unsigned long long *>(dst)[i] = static_cast<const unsigned long long *>(src)[i];
}
template <void (*STEP)(SolverDev *)>
__device__ __forceinline__ void scalar_step_on_copy(SolverDev *S) {
    __shared__ SolverDev sh;
    state_copy(&sh, S);
    __syncwarp();
    if (threadIdx.x == 0) STEP(&sh);
    __syncwarp();
    state_copy(S, &sh);
}

// chi^2 test, alpha schedule and stop (Eq. chi2, Eq. regpara); one thread.
__device__ void scalars_after_residual(SolverDev *S) {
    if (S->done) return;
    const int k = S->k;
    for (int i = 0; i < 2; ++i)
        if (S->phi[i] <= S->chi2_target[i]) S->sat[i] = 1;
    if (k > 0)
        for (int i = 0; i < 2; ++i)
            if (!S->sat[i]) S->alpha[i] = fmax(S->q[i] * S->alpha[i], S->alpha_min[i]);
    const double SG = S->G[0] * S->G[1] - S->G[2] * S->G[2];
    S->phi_last[0] = S->phi[0];
    S->phi_last[1] = S->phi[1];
    S->SG_last = SG;
    if (S->hist) {
        gj_rrcg_hist &h = S->hist[k];
        h.phi[0] = S->phi[0]; h.phi[1] = S->phi[1];
        h.alpha[0] = S->alpha[0]; h.alpha[1] = S->alpha[1];
        h.S_G = SG;
        h.s[0] = h.s[1] = h.beta[0] = h.beta[1] = 0.0;
    }
    S->pending_update = 0;
    if (!isfinite(S->phi[0]) || !isfinite(S->phi[1])) {
        S->status = GJ_ERR_NONFINITE;
        S->done = 1;
        return;
    }
    if ((S->stop_on_chi2 && S->sat[0] && S->sat[1]) || k >= S->kmax) S->done = 1;
    S->phi[0] = S->phi[1] = 0.0;
}

// Step length s_k (RRCG:6); one thread.
__device__ void scalars_after_direction(SolverDev *S) {
    if (S->done) return;
    const int k = S->k;
    double den[2], beta[2];
    for (int i = 0; i < 2; ++i) den[i] = S->qq[i] + (S->alpha[i] + S->lam[i]) * S->pp[i];
    if (S->per_field) {
        for (int i = 0; i < 2; ++i) {
            S->s[i] = den[i] > 0 ? S->pl[i] / den[i] : 0.0;
            beta[i] = (k > 0 && S->ll_prev[i] > 0) ? S->ll[i] / S->ll_prev[i] : 0.0;
        }
    } else {
        const double d = den[0] + den[1];
        const double s = d > 0 ? (S->pl[0] + S->pl[1]) / d : 0.0;
        S->s[0] = S->s[1] = s;
        const double lp = S->ll_prev[0] + S->ll_prev[1];
        beta[0] = beta[1] = (k > 0 && lp > 0) ? (S->ll[0] + S->ll[1]) / lp : 0.0;
    }
    if (S->hist) {
        gj_rrcg_hist &h = S->hist[k];
        h.s[0] = S->s[0]; h.s[1] = S->s[1];
        h.beta[0] = beta[0]; h.beta[1] = beta[1];
    }
    if (!isfinite(S->s[0]) || !isfinite(S->s[1])) {
        S->status = GJ_ERR_NONFINITE;
        S->done = 1;
        return;
    }
    S->ll_prev[0] = S->ll[0];
    S->ll_prev[1] = S->ll[1];
    S->ll[0] = S->ll[1] = 0.0;
    S->pl[0] = S->pl[1] = S->pp[0] = S->pp[1] = 0.0;
    S->qq[0] = S->qq[1] = 0.0;
    S->G[0] = S->G[1] = S->G[2] = 0.0;
    S->pending_update = 1;
    S->k = k + 1;
}

// one warp each (launched as <<<1, 32>>>)
__global__ void k_scalars_after_residual(SolverDev *S) {
    pdl_go();
    pdl_wait();
    scalar_step_on_copy<scalars_after_residual>(S);
}
__global__ void k_scalars_after_direction(SolverDev *S) {
    pdl_go();
    pdl_wait();
    scalar_step_on_copy<scalars_after_direction>(S);
}

// The report of the solver state into device memory (one thread): the same fields
// as gj_rrcg_report_get, without a host round trip.
__global__ void k_report(const SolverDev *S, const int *err, gj_rrcg_report *rep) {
    rep->status = S->status;
    if (err && *err != 0 && rep->status == GJ_OK) rep->status = *err;
    rep->iterations = S->k;
    rep->converged = S->sat[0] && S->sat[1];
    rep->satisfied[0] = S->sat[0];
    rep->satisfied[1] = S->sat[1];
    rep->phi[0] = S->phi_last[0];
    rep->phi[1] = S->phi_last[1];
    rep->alpha[0] = S->alpha[0];
    rep->alpha[1] = S->alpha[1];
    rep->S_G = S->SG_last;
}

// W_d = 1 / sigma (s values, field blockIdx.y) and 1 / W_depth (nz values) of both fields.
template <typename R>
struct Reciprocals {
    const R *sigma[2], *wdep[2];
    R *wd[2], *iwdep[2];
    int s, nz;
};
template <typename R>
__global__ void k_reciprocals(Reciprocals<R> q) {
    const int f = blockIdx.y, i0 = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
    for (int i = i0; i < q.s; i += step) q.wd[f][i] = R(1) / q.sigma[f][i];
    for (int i = i0; i < q.nz; i += step) q.iwdep[f][i] = R(1) / q.wdep[f][i];
}
template <typename R>
static void launch_reciprocals(R *buf, size_t n, size_t s, int nz, const void *const sigma[2],
                               const void *const w_depth[2], cudaStream_t st) {
    Reciprocals<R> q;
    for (int i = 0; i < 2; ++i) {
        q.sigma[i] = static_cast<const R *>(sigma[i]);
        q.wdep[i] = static_cast<const R *>(w_depth[i]);
        q.wd[i] = buf + 4 * n + (2 + i) * s;
        q.iwdep[i] = buf + 4 * n + 4 * s + (size_t)i * nz;
    }
    q.s = (int)s;
    q.nz = nz;
    k_reciprocals<R><<<dim3(64, 2), 256, 0, st>>>(q);
}

}  // namespace gj

using namespace gj;

struct ProfilePair { cudaEvent_t a, b; };

struct gj_rrcg {
    const gj_op *op[2];
    gj_precision prec;
    int dev = 0;              // the device that the solver was made on
    cudaEvent_t used = nullptr;  // behind the last work enqueued on it
    bool in_a_graph = false;     // some of it into a caller's capture, to run whenever that is launched
    SolverDev *S = nullptr;   // device
    void *vhat = nullptr;     // spectra of the residual's rows, both fields (vhat_values)
    void *buf = nullptr;      // p, l (2 fields each, n), v (2 x s), wd (2 x s)
    const void *dobs[2], *mapr[2], *wdep[2], *whard[2];
    bool prev_anchor = false;
    void *m[2];
    gj_rrcg_hist *hist = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t graph_stream = nullptr;
    int profile = 0;
    std::vector<ProfilePair> eager_pairs;   // recorded since the last read
    std::vector<ProfilePair> graph_pairs;   // unused: events inside a graph cannot be timed
    std::vector<ProfilePair> free_pairs;
    bool capturing = false;
    // profiled graph form: the body captured as segments cut around each timed launch
    std::vector<cudaGraph_t> seg_graph;
    std::vector<cudaGraphExec_t> seg_exec;
    cudaStream_t cap_stream = nullptr;   // stream being captured while segmenting
    cudaError_t cap_err = cudaSuccess;
    int grid = 0;  // CTAs of the persistent fast-path launches (0: the operator's, one per SM)
};

namespace gj {

// Notes that work of the solver was enqueued on `st`: its destruction waits for that alone.
// (Calls on one solver are ordered, so the last event stands for all of them.  Waiting for the
// whole device instead fails, and breaks the capture, while any other thread captures a graph;
// the solver's pool memory then went back with its kernels still running.)
static cudaError_t mark_used(gj_rrcg *sv, cudaStream_t st) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess) return e;
    if (cap == cudaStreamCaptureStatusNone) return cudaEventRecord(sv->used, st);
    sv->in_a_graph = true;
    return cudaSuccess;
}

static ProfilePair take_pair(gj_rrcg *sv) {
    ProfilePair p;
    if (!sv->free_pairs.empty()) { p = sv->free_pairs.back(); sv->free_pairs.pop_back(); }
    else { cudaEventCreate(&p.a); cudaEventCreate(&p.b); }
    return p;
}

// Ends the capture in progress, keeps the captured segment, and begins the next.
static void cut_segment(gj_rrcg *sv, cudaStream_t st) {
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(st, &g);
    if (e == cudaSuccess) sv->seg_graph.push_back(g);
    else if (sv->cap_err == cudaSuccess) sv->cap_err = e;
    e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess && sv->cap_err == cudaSuccess) sv->cap_err = e;
}

// The residual's row spectra are written by the end of one iteration and read by the next, so
// they are the solver's own: an operator's workspace serves any other call in between (its
// products, another solver).  Complex values of one field, in the layout of the operator's
// column passes (transposed: rows beyond the stations stay zero); none where the rows are
// transformed from v at the start of an iteration.
static size_t vhat_values(const gj_op *o) {
    if (o->rows1024) return 0;
    return (size_t)o->ncol * (o->fast || o->fast1024 ? o->Ny / 2 : o->sy);
}

template <typename R>
struct SolverLaunch {
    gj_rrcg *sv;
    OpView<R> v0, v1;
    cpx<R> *vhat[2];
    f512::View2<R> V2;
    bool fast = false;
    bool fast1024 = false;  // general row kernels (transposed intermediates) + N_y = 1024 column kernels
    bool rows1024 = false;  // with the warp-FFT row kernels of fast1024.cuh
    FieldVecs<R> F;
    int grid;  // CTAs of the persistent fast-path launches

    void setup() {  // views and launch shapes only (no CUDA calls: safe during capture)
        const gj_op *o = sv->op[0];
        grid = sv->grid > 0 ? sv->grid : o->col_grid;
        v0 = view_of<R>(sv->op[0]);
        v1 = view_of<R>(sv->op[1]);
        if constexpr (std::is_same_v<R, float>) {
            fast = o->fast && sv->op[1]->fast;
            fast1024 = o->fast1024 && sv->op[1]->fast1024;
            rows1024 = fast1024 && o->rows1024;
            if (fast || fast1024) V2 = f512::make_view2<R>(sv->op[0], sv->op[1]);
        }
        vhat[0] = static_cast<cpx<R> *>(sv->vhat);
        vhat[1] = vhat[0] + vhat_values(o);
        if ((fast || fast1024) && !rows1024)
            for (int i = 0; i < 2; ++i) V2.op[i].V = vhat[i];
        const int n = o->nx * o->ny * o->nz, s = o->sx * o->sy;
        R *b = static_cast<R *>(sv->buf);
        for (int i = 0; i < 2; ++i) {
            F.m[i] = static_cast<R *>(sv->m[i]);
            F.p[i] = b + (size_t)i * n;
            F.l[i] = b + (size_t)(2 + i) * n;
            F.v[i] = b + (size_t)4 * n + (size_t)i * s;
            F.wd[i] = b + (size_t)4 * n + (size_t)(2 + i) * s;
            F.dobs[i] = static_cast<const R *>(sv->dobs[i]);
            F.mapr[i] = static_cast<const R *>(sv->mapr[i]);
            F.wdep[i] = static_cast<const R *>(sv->wdep[i]);
            F.iwdep[i] = b + (size_t)4 * n + (size_t)4 * s + (size_t)i * o->nz;
            F.mtp[i] = sv->prev_anchor ? b + (size_t)4 * n + (size_t)4 * s + (size_t)2 * o->nz + (size_t)i * n : nullptr;
            F.whard[i] = static_cast<const R *>(sv->whard[i]);
        }
    }

    // any optional row (hard weights, a-priori model, previous-model anchor) present:
    // the functors' variants without them skip those loads and factors entirely
    bool opt_rows() const {
        for (int i = 0; i < 2; ++i)
            if (F.whard[i] || F.mapr[i] || F.mtp[i]) return true;
        return false;
    }

    void set_attributes() {
        // Load every kernel of an iteration now: with lazy module loading, the first
        // launch of a kernel inside a stream capture would invalidate the capture.
        cudaFuncAttributes fa;
        cudaFuncGetAttributes(&fa, k_scalars_after_direction);
        cudaFuncGetAttributes(&fa, k_scalars_after_residual);
        if constexpr (std::is_same_v<R, float>) if (fast) {
            using namespace f512;
            set_row_fwd_t_attr<R, ProModel<R, true>>();
            set_row_fwd_t_attr<R, ProDirection<R, true>>();
            set_row_fwd_t_attr<R, ProModel<R, false>>();
            set_row_fwd_t_attr<R, ProDirection<R, false>>();
            set_row_resid_attr<R, EpiResidual<R>, kDataNW>();
            set_row_inv_t_attr<R, EpiGradient<R, true>>();
            set_row_inv_t_attr<R, EpiGradient<R, false>>();
            set_row_inv_attr<R, EpiQNorm<R>, kDataNW, kDataFPW>();
            set_col_attr<R>();
            return;
        }
        if constexpr (std::is_same_v<R, float>) if (fast1024) {
            f1024::set_col_attr<R>();
            f1024::set_row_fwd_attr<R, ProModel<R>>();
            f1024::set_row_fwd_attr<R, ProDirection<R>>();
            f1024::set_row_fwd_attr<R, LoadPlain2<R>>();
            f1024::set_row_inv_attr<R, EpiResidual<R>>();
            f1024::set_row_inv_attr<R, EpiGradient<R>>();
            f1024::set_row_inv_attr<R, EpiQNorm<R>>();
        }
        if constexpr (std::is_same_v<R, float>) if (rows1024) return;
        gen_row_fwd_attr<R, ProModel<R>>();
        gen_row_fwd_attr<R, ProDirection<R>>();
        gen_row_resid_attr<R, EpiResidual<R>>();
        gen_row_inv_attr<R, EpiGradient<R>>();
        gen_row_inv_attr<R, EpiQNorm<R>>();
        gen_col_attr<R>();
    }

    // Row passes of the general path over both fields (cell lines: a line of each field a
    // transform; data lines: nf = 2 and two lines of one field): the block FFT kernels, or
    // (rows1024) the warp-FFT row kernels that go with the N_y = 1024 columns.
    template <class Pro>
    void rows_fwd(const PairMap &pm, int n_in, cpx<R> *o0, cpx<R> *o1, const Pro &pro, const int *done,
                  cudaStream_t st) {
        if constexpr (std::is_same_v<R, float>) if (rows1024) {
            f1024::row_fwd<R>(v0, pm, n_in, o0, o1, sv->op[0]->twtab, pro, done, st);
            return;
        }
        gen_row_fwd<R>(sv->op[0], v0, pm, n_in, o0, o1, pro, done, st);
    }
    template <class Epi>
    void rows_inv(const PairMap &pm, int n_out, const cpx<R> *i0, const cpx<R> *i1, const Epi &epi, const int *done,
                  cudaStream_t st, int nf = 1) {
        if constexpr (std::is_same_v<R, float>) if (rows1024) {
            f1024::row_inv<R>(v0, pm, n_out, i0, i1, sv->op[0]->twtab, epi, done, st, nf);
            return;
        }
        gen_row_inv<R>(sv->op[0], v0, pm, n_out, i0, i1, epi, done, st, nf);
    }

    // Forward columns (Y = sum_r T^_r FFT_y(Z_r)) and inverse columns, both fields.
    void forward_columns(cudaStream_t st) {
        const gj_op *o = sv->op[0];
        if constexpr (std::is_same_v<R, float>) if (fast) {
            ProfilePair pp{};
            if (sv->profile && sv->capturing) {
                cut_segment(sv, st);  // the timed launch gets a segment of its own
            } else if (sv->profile) {
                pp = take_pair(sv);
                cudaEventRecord(pp.a, st);
            }
            f512::col_fwd<R>(V2, grid, &sv->S->done, st);
            if (sv->profile && sv->capturing) {
                cut_segment(sv, st);
            } else if (sv->profile) {
                cudaEventRecord(pp.b, st);
                sv->eager_pairs.push_back(pp);
            }
            return;
        }
        if constexpr (std::is_same_v<R, float>) if (fast1024) {
            ProfilePair pp{};
            if (sv->profile && !sv->capturing) {
                pp = take_pair(sv);
                cudaEventRecord(pp.a, st);
            }
            f1024::col_fwd<R>(V2, grid, &sv->S->done, st);
            if (sv->profile && !sv->capturing) {
                cudaEventRecord(pp.b, st);
                sv->eager_pairs.push_back(pp);
            }
            return;
        }
        ProfilePair pp{};
        if (sv->profile && !sv->capturing) {
            pp = take_pair(sv);
            cudaEventRecord(pp.a, st);
        }
        gen_col_fwd<R>(o, v0, v1, 2, o->nz, &sv->S->done, st);
        if (sv->profile && !sv->capturing) {
            cudaEventRecord(pp.b, st);
            sv->eager_pairs.push_back(pp);
        }
    }

    void head(cudaStream_t st) {  // forward of (updated) m, residual, chi^2 scalars
        const gj_op *o = sv->op[0];
        const int *done = &sv->S->done;
        if constexpr (std::is_same_v<R, float>) if (fast) {
            using namespace f512;
            if (opt_rows()) {
                ProModel<R, true> pm{F, sv->S, o->nx, o->ny};
                row_fwd_t<R>(V2, grid, o->nz, o->ny, o->nx, 0, pm, done, st);
            } else {
                ProModel<R, false> pm{F, sv->S, o->nx, o->ny};
                row_fwd_t<R>(V2, grid, o->nz, o->ny, o->nx, 0, pm, done, st);
            }
            forward_columns(st);
            // residual, Phi and the residual rows' spectra for the adjoint, in one pass
            EpiResidual<R> er{F, sv->S, o->sx};
            row_resid<R, kDataNW>(V2, o->sy, o->sx, er, done, st);
            launch_after(k_scalars_after_residual, dim3(1), dim3(32), 0, st, sv->S);
            return;
        }
        PairMap pc{o->nz * o->ny, 1, o->ny};
        ProModel<R> pm{F, sv->S, o->nx, o->ny};
        rows_fwd(pc, o->nx, v0.Z, v1.Z, pm, done, st);
        forward_columns(st);
        PairMap ps{o->sy, 0, o->sy};
        EpiResidual<R> er{F, sv->S, o->sx};
        // residual, Phi and the residual rows' spectra for the adjoint, in one pass
        if constexpr (std::is_same_v<R, float>)
            if (rows1024) f1024::row_inv<R>(v0, ps, o->sx, v0.W, v1.W, o->twtab, er, done, st, 2);
        if (!rows1024)
            gen_row_resid<R>(o, v0, ps, o->sx, v0.W, v1.W, vhat[0], vhat[1], er, done, st, 2);
        launch_after(k_scalars_after_residual, dim3(1), dim3(32), 0, st, sv->S);
    }

    void body(cudaStream_t st) {
        const gj_op *o = sv->op[0];
        const int *done = &sv->S->done;
        if constexpr (std::is_same_v<R, float>) if (fast) {
            using namespace f512;
            col_adj<R>(V2, grid, done, st);
            if (opt_rows()) {
                EpiGradient<R, true> eg{F, sv->S, o->nx, o->ny};
                row_inv_t<R>(V2, grid, o->nz, o->ny, o->nx, 0, eg, done, st);
                ProDirection<R, true> pd{F, sv->S, o->nx, o->ny};
                row_fwd_t<R>(V2, grid, o->nz, o->ny, o->nx, 0, pd, done, st);
            } else {
                EpiGradient<R, false> eg{F, sv->S, o->nx, o->ny};
                row_inv_t<R>(V2, grid, o->nz, o->ny, o->nx, 0, eg, done, st);
                ProDirection<R, false> pd{F, sv->S, o->nx, o->ny};
                row_fwd_t<R>(V2, grid, o->nz, o->ny, o->nx, 0, pd, done, st);
            }
            forward_columns(st);
            EpiQNorm<R> eq{F, sv->S, o->sx};
            row_inv<R, kDataNW, kDataFPW>(V2, 0, o->sy, o->sy, o->sx, 1, eq, done, st, 2);
            launch_after(k_scalars_after_direction, dim3(1), dim3(32), 0, st, sv->S);
            head(st);
            return;
        }
        PairMap ps{o->sy, 0, o->sy};
        PairMap pc{o->nz * o->ny, 1, o->ny};
        // adjoint: the residual rows' spectra (head) -> per-layer conj-spectrum columns -> Z
        if constexpr (std::is_same_v<R, float>) {
            if (rows1024)
                f1024::row_fwd<R>(v0, ps, o->sx, v0.V, v1.V, o->twtab, LoadPlain2<R>{{F.v[0], F.v[1]}, o->sx}, done, st,
                                  2);
            if (fast1024) f1024::col_adj<R>(V2, grid, done, st);
        }
        if (!fast1024) {
            OpView<R> a0 = v0, a1 = v1;
            a0.W = vhat[0];
            a1.W = vhat[1];
            gen_col_adj<R>(o, a0, a1, 2, o->nz, done, st);
        }
        EpiGradient<R> eg{F, sv->S, o->nx, o->ny};
        rows_inv(pc, o->nx, v0.Z, v1.Z, eg, done, st);
        // direction and its forward product
        ProDirection<R> pd{F, sv->S, o->nx, o->ny};
        rows_fwd(pc, o->nx, v0.Z, v1.Z, pd, done, st);
        forward_columns(st);
        EpiQNorm<R> eq{F, sv->S, o->sx};
        rows_inv(ps, o->sx, v0.W, v1.W, eq, done, st, 2);
        launch_after(k_scalars_after_direction, dim3(1), dim3(32), 0, st, sv->S);
        // model update, its forward product and the chi^2 scalars
        head(st);
    }
};

template <typename R>
static void run_head(gj_rrcg *sv, cudaStream_t st) {
    SolverLaunch<R> L{sv};
    L.setup();
    L.set_attributes();
    L.head(st);
}

template <typename R>
static void run_body(gj_rrcg *sv, cudaStream_t st) {
    SolverLaunch<R> L{sv};
    L.setup();
    L.body(st);
}

static gj_status check_ops(const gj_op *const ops[2]) {
    if (!ops || !ops[0] || !ops[1]) { set_error("rrcg: ops must be non-NULL"); return GJ_ERR_ARG; }
    const gj_op *a = ops[0], *b = ops[1];
    if (a->field != GJ_GRAVITY || b->field != GJ_MAGNETIC) {
        set_error("rrcg: ops[0] must be gravity and ops[1] magnetic"); return GJ_ERR_ARG;
    }
    if (a->sx != b->sx || a->sy != b->sy || a->nx != b->nx || a->ny != b->ny || a->nz != b->nz ||
        a->Nx != b->Nx || a->Ny != b->Ny || a->prec != b->prec) {
        set_error("rrcg: both operators must share grid sizes, padded sizes and precision"); return GJ_ERR_ARG;
    }
    if (a->recompute || b->recompute) {
        set_error("rrcg: operators that recompute their spectra per layer serve products only");
        return GJ_ERR_UNSUPPORTED;
    }
    return GJ_OK;
}

}  // namespace gj

// A solver is not made under stream capture: its memory would be a node of the graph.
static gj_status not_capturing(cudaStream_t st, const char *what) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    GJ_CUDA(cudaStreamIsCapturing(st, &cap));
    if (cap == cudaStreamCaptureStatusNone) return GJ_OK;
    set_error(std::string(what) + ": the stream is being captured");
    return GJ_ERR_CUDA;
}

// Creation was host time: two cudaMalloc, four small launches, and two cudaFree at the end (each a
// device-wide synchronisation).  One stream-ordered block of the library's pool and one launch
// for the reciprocals take their place: create and destroy of a 256 x 256 x 40 solver went from
// 258 + 110 to 157 + 28 us, six uneven ones from 1540 + 350 to 900 + 25 us.  wait: the solver is
// ready for any stream on return.  The one-shot solve stays in its stream and does not wait, so
// that its graph is captured while the first residual runs (70 us).
static gj_status rrcg_create(const gj_op *const ops[2], const gj_rrcg_params *P, const void *const dobs[2],
                             const void *const sigma[2], const void *const m_apr[2], const void *const w_depth[2],
                             const void *const w_hard[2], void *const m[2], gj_rrcg_hist *hist, gj_stream_t stream,
                             bool wait, gj_rrcg **out) {
    if (!out) { set_error("gj_rrcg_create: out is NULL"); return GJ_ERR_ARG; }
    *out = nullptr;
    gj_status rc = check_ops(ops);
    if (rc != GJ_OK) return rc;
    if (!P || !dobs || !sigma || !w_depth || !m) { set_error("gj_rrcg_create: NULL argument"); return GJ_ERR_ARG; }
    for (int i = 0; i < 2; ++i) {
        if (!dobs[i] || !sigma[i] || !w_depth[i] || !m[i]) { set_error("gj_rrcg_create: NULL vector"); return GJ_ERR_ARG; }
        if (P->p[i] != 1 && P->p[i] != 2) { set_error("gj_rrcg_create: p must be 1 or 2"); return GJ_ERR_ARG; }
        if (!(P->lo[i] <= P->hi[i])) { set_error("gj_rrcg_create: lo must not exceed hi"); return GJ_ERR_ARG; }
        if (!(P->alpha1[i] >= 0) || !(P->lambda[i] >= 0) || !(P->q[i] > 0)) {
            set_error("gj_rrcg_create: alpha1, lambda must be >= 0 and q > 0"); return GJ_ERR_ARG;
        }
    }
    if (P->kmax < 0) { set_error("gj_rrcg_create: kmax must be >= 0"); return GJ_ERR_ARG; }
    if (!(P->eps2 > 0)) { set_error("gj_rrcg_create: eps2 must be > 0"); return GJ_ERR_ARG; }
    if (P->scalars < 0 || P->scalars > 2) { set_error("gj_rrcg_create: bad scalars mode"); return GJ_ERR_ARG; }
    if (P->anchor != GJ_ANCHOR_APRIORI && P->anchor != GJ_ANCHOR_PREVIOUS) {
        set_error("gj_rrcg_create: bad anchor"); return GJ_ERR_ARG;
    }
    if (P->gramian_space != GJ_GRAMIAN_ORIGINAL && P->gramian_space != GJ_GRAMIAN_WEIGHTED) {
        set_error("gj_rrcg_create: bad gramian_space"); return GJ_ERR_ARG;
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if ((rc = not_capturing(st, "gj_rrcg_create")) != GJ_OK) return rc;
    gj_rrcg *sv = new (std::nothrow) gj_rrcg();
    if (!sv) { set_error("gj_rrcg_create: host allocation failed"); return GJ_ERR_OOM; }
    const gj_op *o = ops[0];
    sv->op[0] = ops[0]; sv->op[1] = ops[1];
    sv->prec = o->prec;
    cudaError_t e;
    if ((e = cudaGetDevice(&sv->dev)) != cudaSuccess) {
        delete sv;
        return cuda_fail(e, "gj_rrcg_create");
    }
    for (int i = 0; i < 2; ++i) {
        sv->dobs[i] = dobs[i];
        sv->mapr[i] = m_apr ? m_apr[i] : nullptr;
        sv->wdep[i] = w_depth[i];
        sv->whard[i] = w_hard ? w_hard[i] : nullptr;
        sv->m[i] = m[i];
    }
    sv->hist = hist;
    sv->prev_anchor = P->anchor == GJ_ANCHOR_PREVIOUS;
    const size_t es = elem_bytes(o->prec);
    const size_t n = (size_t)o->nx * o->ny * o->nz, s = (size_t)o->sx * o->sy;
    // one block: the state, the residual's row spectra, then the vectors
    const size_t vhat_bytes = (2 * vhat_values(o) * 2 * es + 255) / 256 * 256;
    const size_t nbuf = 4 * n + 4 * s + 2 * (size_t)o->nz + (sv->prev_anchor ? 2 * n : 0);
    constexpr size_t kStateBytes = (sizeof(SolverDev) + 255) / 256 * 256;
    void *blk = nullptr;
    if ((e = cudaEventCreateWithFlags(&sv->used, cudaEventDisableTiming)) != cudaSuccess ||
        (e = pool_alloc(&blk, kStateBytes + vhat_bytes + nbuf * es, st)) != cudaSuccess) {
        if (sv->used) cudaEventDestroy(sv->used);
        delete sv;
        return cuda_fail(e, "solver state and vectors");
    }
    sv->S = static_cast<SolverDev *>(blk);
    sv->vhat = static_cast<char *>(blk) + kStateBytes;
    sv->buf = static_cast<char *>(sv->vhat) + vhat_bytes;
    SolverDev h{};
    h.kmax = P->kmax;
    h.stop_on_chi2 = P->stop_on_chi2;
    const bool lam0 = P->lambda[0] == 0 && P->lambda[1] == 0;
    h.per_field = P->scalars == GJ_SCALARS_PER_FIELD || (P->scalars == GJ_SCALARS_AUTO && lam0);
    h.anchor = P->anchor;
    h.gspace = P->gramian_space;
    h.eps2 = P->eps2;
    for (int i = 0; i < 2; ++i) {
        h.p[i] = P->p[i];
        h.alpha[i] = P->alpha1[i]; h.q[i] = P->q[i]; h.alpha_min[i] = P->alpha_min[i];
        h.lam[i] = P->lambda[i]; h.lo[i] = P->lo[i]; h.hi[i] = P->hi[i];
        h.chi2_target[i] = (double)s + sqrt(2.0 * (double)s);
    }
    h.hist = hist;
    cudaMemcpyAsync(sv->S, &h, sizeof(h), cudaMemcpyHostToDevice, st);
    cudaMemsetAsync(sv->vhat, 0, vhat_bytes + 4 * n * es, st);
    if (o->prec == GJ_FP64) launch_reciprocals(static_cast<double *>(sv->buf), n, s, o->nz, sigma, w_depth, st);
    else launch_reciprocals(static_cast<float *>(sv->buf), n, s, o->nz, sigma, w_depth, st);
    if (o->prec == GJ_FP64) run_head<double>(sv, st); else run_head<float>(sv, st);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = mark_used(sv, st);
    if (e == cudaSuccess && wait) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaStreamSynchronize(st);  // (freeing pool memory does not wait for its kernels)
        cudaFree(sv->S);
        cudaEventDestroy(sv->used);
        delete sv;
        return cuda_fail(e, "gj_rrcg_create");
    }
    *out = sv;
    return GJ_OK;
}

extern "C" gj_status gj_rrcg_create(const gj_op *const ops[2], const gj_rrcg_params *P,
                                    const void *const dobs[2], const void *const sigma[2],
                                    const void *const m_apr[2], const void *const w_depth[2],
                                    const void *const w_hard[2], void *const m[2], gj_rrcg_hist *hist,
                                    gj_stream_t stream, gj_rrcg **out) {
    return rrcg_create(ops, P, dobs, sigma, m_apr, w_depth, w_hard, m, hist, stream, true, out);
}

static gj_status iterate_on(gj_rrcg *sv, int iters, int use_graph, cudaStream_t st) {
    if (use_graph && sv->profile && sv->prec == GJ_FP32_MIXED && sv->op[0]->fast) {
        // segments [.. | col | .. | col | ..] with stream events around the column launches
        if (sv->seg_exec.empty()) {
            cudaStream_t cap;
            GJ_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
            std::unique_lock<std::mutex> lock(capture_mutex());
            sv->capturing = true;
            sv->cap_err = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
            if (sv->cap_err == cudaSuccess) {
                run_body<float>(sv, cap);
                cudaGraph_t g = nullptr;
                cudaError_t e = cudaStreamEndCapture(cap, &g);
                if (e == cudaSuccess) sv->seg_graph.push_back(g);
                else if (sv->cap_err == cudaSuccess) sv->cap_err = e;
            }
            sv->capturing = false;
            lock.unlock();
            cudaStreamDestroy(cap);
            if (sv->cap_err != cudaSuccess || sv->seg_graph.size() != 5) {
                for (auto g : sv->seg_graph) cudaGraphDestroy(g);
                sv->seg_graph.clear();
                return cuda_fail(sv->cap_err != cudaSuccess ? sv->cap_err : cudaErrorUnknown, "rrcg segment capture");
            }
            for (auto g : sv->seg_graph) {
                cudaGraphExec_t x;
                GJ_CUDA(cudaGraphInstantiate(&x, g, 0));
                sv->seg_exec.push_back(x);
            }
        }
        for (int it = 0; it < iters; ++it) {
            for (int sgi = 0; sgi < 5; ++sgi) {
                ProfilePair pp{};
                if (sgi == 1 || sgi == 3) {
                    pp = take_pair(sv);
                    GJ_CUDA(cudaEventRecord(pp.a, st));
                }
                GJ_CUDA(cudaGraphLaunch(sv->seg_exec[sgi], st));
                if (sgi == 1 || sgi == 3) {
                    GJ_CUDA(cudaEventRecord(pp.b, st));
                    sv->eager_pairs.push_back(pp);
                }
            }
        }
        return GJ_OK;
    }
    if (use_graph) {
        if (!sv->exec) {
            cudaStream_t cap;
            GJ_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
            std::unique_lock<std::mutex> lock(capture_mutex());
            sv->capturing = true;
            cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
            if (e == cudaSuccess) {
                if (sv->prec == GJ_FP64) run_body<double>(sv, cap); else run_body<float>(sv, cap);
                e = cudaStreamEndCapture(cap, &sv->graph);
            }
            sv->capturing = false;
            lock.unlock();
            cudaStreamDestroy(cap);
            if (e != cudaSuccess) return cuda_fail(e, "rrcg graph capture");
            GJ_CUDA(cudaGraphInstantiate(&sv->exec, sv->graph, 0));
        }
        for (int it = 0; it < iters; ++it) GJ_CUDA(cudaGraphLaunch(sv->exec, st));
    } else {
        for (int it = 0; it < iters; ++it) {
            if (sv->prec == GJ_FP64) run_body<double>(sv, st); else run_body<float>(sv, st);
        }
        GJ_CUDA(cudaGetLastError());
    }
    return GJ_OK;
}

extern "C" gj_status gj_rrcg_iterate(gj_rrcg *sv, int iters, int use_graph, gj_stream_t stream) {
    if (!sv || iters < 0) { set_error("gj_rrcg_iterate: bad argument"); return GJ_ERR_ARG; }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    gj_status rc = iterate_on(sv, iters, use_graph, st);
    cudaError_t e = mark_used(sv, st);  // (a call that failed may have enqueued some of its work)
    return rc == GJ_OK && e != cudaSuccess ? cuda_fail(e, "gj_rrcg_iterate") : rc;
}

extern "C" gj_status gj_rrcg_report_get(gj_rrcg *sv, gj_rrcg_report *rep, gj_stream_t stream) {
    if (!sv || !rep) { set_error("gj_rrcg_report_get: NULL argument"); return GJ_ERR_ARG; }
    SolverDev h;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    GJ_CUDA(cudaMemcpyAsync(&h, sv->S, sizeof(h), cudaMemcpyDeviceToHost, st));
    GJ_CUDA(cudaStreamSynchronize(st));
    rep->status = h.status;
    rep->iterations = h.k;
    rep->converged = h.sat[0] && h.sat[1];
    rep->satisfied[0] = h.sat[0];
    rep->satisfied[1] = h.sat[1];
    rep->phi[0] = h.phi_last[0];
    rep->phi[1] = h.phi_last[1];
    rep->alpha[0] = h.alpha[0];
    rep->alpha[1] = h.alpha[1];
    rep->S_G = h.SG_last;
    if (sv->op[0]->err) {
        int e = 0;
        GJ_CUDA(cudaMemcpy(&e, sv->op[0]->err, sizeof(int), cudaMemcpyDeviceToHost));
        if (e != 0 && rep->status == GJ_OK) rep->status = e;
    }
    return GJ_OK;
}

extern "C" gj_status gj_rrcg_report_device(gj_rrcg *sv, gj_rrcg_report *rep, gj_stream_t stream) {
    if (!sv || !rep) { set_error("gj_rrcg_report_device: NULL argument"); return GJ_ERR_ARG; }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    k_report<<<1, 1, 0, st>>>(sv->S, sv->op[0]->err, rep);
    GJ_CUDA(cudaGetLastError());
    GJ_CUDA(mark_used(sv, st));
    return GJ_OK;
}

extern "C" int gj_rrcg_done(gj_rrcg *sv, gj_stream_t stream) {
    if (!sv) return -1;
    int d = 0;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(&d, &sv->S->done, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return -1;
    if (cudaStreamSynchronize(st) != cudaSuccess) return -1;
    return d;
}

extern "C" gj_status gj_rrcg_profile(gj_rrcg *sv, int enable) {
    if (!sv) { set_error("gj_rrcg_profile: NULL solver"); return GJ_ERR_ARG; }
    sv->profile = enable ? 1 : 0;
    return GJ_OK;
}

extern "C" gj_status gj_rrcg_profile_read(gj_rrcg *sv, int *launches, double *total_ms) {
    if (!sv || !launches || !total_ms) { set_error("gj_rrcg_profile_read: NULL argument"); return GJ_ERR_ARG; }
    GJ_CUDA(sync_device());
    double tot = 0.0;
    int cnt = 0;
    auto acc = [&](const std::vector<ProfilePair> &v) -> gj_status {
        for (const auto &p : v) {
            float ms = 0.f;
            cudaError_t e = cudaEventElapsedTime(&ms, p.a, p.b);
            if (e != cudaSuccess) return cuda_fail(e, "gj_rrcg_profile_read");
            tot += ms;
            ++cnt;
        }
        return GJ_OK;
    };
    gj_status rc = acc(sv->eager_pairs);
    if (rc != GJ_OK) return rc;
    for (auto &p : sv->eager_pairs) sv->free_pairs.push_back(p);
    sv->eager_pairs.clear();
    *launches = cnt;
    *total_ms = tot;
    return GJ_OK;
}

extern "C" void gj_rrcg_destroy(gj_rrcg *sv) {
    if (!sv) return;
    DeviceScope scope(sv->dev);  // whatever device is current: its kernels are the ones to wait for
    const cudaError_t e = sv->in_a_graph ? sync_device() : cudaEventSynchronize(sv->used);
    if (sv->exec) cudaGraphExecDestroy(sv->exec);
    if (sv->graph) cudaGraphDestroy(sv->graph);
    for (auto x : sv->seg_exec) cudaGraphExecDestroy(x);
    for (auto g : sv->seg_graph) cudaGraphDestroy(g);
    for (auto *v : {&sv->eager_pairs, &sv->graph_pairs, &sv->free_pairs})
        for (auto &p : *v) { cudaEventDestroy(p.a); cudaEventDestroy(p.b); }
    cudaEventDestroy(sv->used);
    // The state and the vectors, one block.  Memory whose work could not be waited for (in a
    // caller's graph, while somebody else captures) is not given back.
    if (e == cudaSuccess) cudaFree(sv->S);
    else cudaGetLastError();
    delete sv;
}

// Two page-locked ints per host thread for the one-shot solve's stop flags,
// allocated on first use and kept for the life of the process (portable: any
// device may write them).  NULL if page-locked memory is not available.
static int *pinned_flags() {
    thread_local int *p = nullptr;
    thread_local bool tried = false;
    if (!tried) {
        tried = true;
        if (cudaHostAlloc(reinterpret_cast<void **>(&p), 2 * sizeof(int), cudaHostAllocPortable) != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
    }
    return p;
}

extern "C" gj_status gj_rrcg_joint_solve(const gj_op *const ops[2], const gj_rrcg_params *P,
                                         const void *const dobs[2], const void *const sigma[2],
                                         const void *const m_apr[2], const void *const w_depth[2],
                                         const void *const w_hard[2], void *const m[2], gj_rrcg_hist *hist,
                                         gj_rrcg_report *rep, gj_stream_t stream) {
    if (!rep) { set_error("gj_rrcg_joint_solve: rep is NULL"); return GJ_ERR_ARG; }
    gj_rrcg *sv = nullptr;
    gj_status rc = rrcg_create(ops, P, dobs, sigma, m_apr, w_depth, w_hard, m, hist, stream, false, &sv);
    if (rc != GJ_OK) return rc;
    // Iterations go in chunks of eight graph replays.  The stop flag of chunk c - 1 is
    // copied into page-locked memory behind it and read while chunk c runs, so the
    // device never waits for the host; a chunk queued after the stop does no work
    // (every kernel returns at the flag).
    int left = P->kmax;
    const int chunk = 8;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int *flags = pinned_flags();
    cudaEvent_t ev[2] = {nullptr, nullptr};
    if (flags && (cudaEventCreateWithFlags(&ev[0], cudaEventDisableTiming) != cudaSuccess ||
                  cudaEventCreateWithFlags(&ev[1], cudaEventDisableTiming) != cudaSuccess))
        flags = nullptr;
    for (int c = 0; left > 0; ++c) {
        const int it = std::min(chunk, left);
        rc = gj_rrcg_iterate(sv, it, 1, stream);
        if (rc != GJ_OK) break;
        left -= it;
        if (!flags) {  // no page-locked flag: a synchronous check after each chunk
            const int d = gj_rrcg_done(sv, stream);
            if (d < 0) { rc = cuda_fail(cudaGetLastError(), "gj_rrcg_joint_solve"); break; }
            if (d) break;
            continue;
        }
        cudaError_t e = cudaMemcpyAsync(flags + (c & 1), &sv->S->done, sizeof(int), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaEventRecord(ev[c & 1], st);
        if (e == cudaSuccess && c > 0) e = cudaEventSynchronize(ev[(c - 1) & 1]);
        if (e != cudaSuccess) { rc = cuda_fail(e, "gj_rrcg_joint_solve: stop flag"); break; }
        if (c > 0 && flags[(c - 1) & 1]) break;
    }
    for (cudaEvent_t x : ev)
        if (x) cudaEventDestroy(x);
    if (rc == GJ_OK) rc = gj_rrcg_report_get(sv, rep, stream);
    gj_rrcg_destroy(sv);
    if (rc == GJ_OK && rep->status != GJ_OK) {
        set_error("gj_rrcg_joint_solve: non-finite scalar");
        return (gj_status)rep->status;
    }
    return rc;
}

// ---------------------------------------------------------------------------
// Batched form: several independent joint inversions (any sizes and precisions)
// advanced by one CUDA graph whose branches are the solvers' iterations.

struct gj_rrcg_batch {
    std::vector<gj_rrcg *> sv;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaEvent_t used = nullptr;  // behind the last step
};

extern "C" gj_status gj_rrcg_batch_create(gj_rrcg *const *solvers, int count, gj_stream_t stream,
                                          gj_rrcg_batch **out) {
    (void)stream;
    if (!out || !solvers || count < 1) { set_error("gj_rrcg_batch_create: bad argument"); return GJ_ERR_ARG; }
    *out = nullptr;
    for (int i = 0; i < count; ++i)
        if (!solvers[i]) { set_error("gj_rrcg_batch_create: NULL solver"); return GJ_ERR_ARG; }
    // the graph runs the solvers concurrently: an operator's workspace cannot be shared
    for (int i = 0; i < count; ++i)
        for (int j = 0; j < i; ++j)
            for (int a = 0; a < 2; ++a)
                for (int b2 = 0; b2 < 2; ++b2)
                    if (solvers[i]->op[a] == solvers[j]->op[b2]) {
                        set_error("gj_rrcg_batch_create: two solvers share an operator (give each its own)");
                        return GJ_ERR_ARG;
                    }
    gj_rrcg_batch *b = new (std::nothrow) gj_rrcg_batch();
    if (!b) { set_error("gj_rrcg_batch_create: host allocation failed"); return GJ_ERR_OOM; }
    b->sv.assign(solvers, solvers + count);
    // The branches run concurrently: the fast-path solvers get grids in proportion to
    // their work (column items, scaled by N_y, plus row lines per layer), so that their
    // persistent kernels (one CTA per SM each) can be resident at the same time.  Each
    // gets twice its proportional share: the branches finish at different times, and
    // grids that add up to one CTA per SM leave SMs idle once the smaller problems are
    // done.  A smaller grid never needs more layer-sum slots than the operator holds
    // (each warp's segment only grows); the check below keeps the full grid otherwise.
    {
        auto work = [](const gj_op *o) { return (double)o->nz * (2.0 * 257 * o->Ny / 512 + o->ny); };
        double tot = 0.0;
        int sms = 0;
        for (gj_rrcg *sv : b->sv)
            if (sv->op[0]->fast && sv->prec == GJ_FP32_MIXED) {
                tot += work(sv->op[0]);
                sms = sv->op[0]->col_grid;
            }
        for (gj_rrcg *sv : b->sv) {
            sv->grid = 0;
            const gj_op *o = sv->op[0];
            if (!(o->fast && sv->prec == GJ_FP32_MIXED) || tot <= 0.0) continue;
            const double share = work(o) / tot;
            const int g = std::max(1, std::min(o->col_grid, (int)(2.0 * sms * share)));
            const int ci = fast_col_items(o->Ny, o->nz);
            const long long warps = (long long)g * f512::CWARPS;
            if (g < o->col_grid && fast_slots(2, 257, ci, warps) <= o->slots && fast_slots(1, 257, ci, warps) <= o->slots)
                sv->grid = g;
        }
    }
    // streams and events exist before the capture begins
    cudaStream_t cap = nullptr;
    std::vector<cudaStream_t> br(count, nullptr);
    std::vector<cudaEvent_t> join(count, nullptr);
    cudaEvent_t fork = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->used, cudaEventDisableTiming);
    for (int i = 0; i < count && e == cudaSuccess; ++i) {
        e = cudaStreamCreateWithFlags(&br[i], cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join[i], cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
    std::unique_lock<std::mutex> lock(capture_mutex());
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        cudaError_t ce = cudaEventRecord(fork, cap);
        for (int i = 0; i < count && ce == cudaSuccess; ++i) {
            ce = cudaStreamWaitEvent(br[i], fork, 0);
            if (ce != cudaSuccess) break;
            gj_rrcg *sv = b->sv[i];
            sv->capturing = true;
            if (sv->prec == GJ_FP64) run_body<double>(sv, br[i]); else run_body<float>(sv, br[i]);
            sv->capturing = false;
            ce = cudaEventRecord(join[i], br[i]);
            if (ce == cudaSuccess) ce = cudaStreamWaitEvent(cap, join[i], 0);
        }
        cudaError_t ee = cudaStreamEndCapture(cap, &b->graph);
        e = ce != cudaSuccess ? ce : ee;
    }
    lock.unlock();
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
    for (gj_rrcg *sv : b->sv) sv->grid = 0;  // stepwise calls outside the batch use the full grid
    for (int i = 0; i < count; ++i) {
        if (br[i]) cudaStreamDestroy(br[i]);
        if (join[i]) cudaEventDestroy(join[i]);
    }
    if (fork) cudaEventDestroy(fork);
    if (cap) cudaStreamDestroy(cap);
    if (e != cudaSuccess) {
        if (b->graph) cudaGraphDestroy(b->graph);
        if (b->used) cudaEventDestroy(b->used);
        delete b;
        return cuda_fail(e, "gj_rrcg_batch_create");
    }
    *out = b;
    return GJ_OK;
}

extern "C" gj_status gj_rrcg_batch_step(gj_rrcg_batch *b, int iters, gj_stream_t stream) {
    if (!b || iters < 0) { set_error("gj_rrcg_batch_step: bad argument"); return GJ_ERR_ARG; }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    for (int it = 0; it < iters && e == cudaSuccess; ++it) e = cudaGraphLaunch(b->exec, st);
    cudaError_t e2 = cudaEventRecord(b->used, st);
    for (gj_rrcg *sv : b->sv)
        if (e2 == cudaSuccess) e2 = mark_used(sv, st);
    if (e == cudaSuccess) e = e2;
    return e == cudaSuccess ? GJ_OK : cuda_fail(e, "gj_rrcg_batch_step");
}

extern "C" void gj_rrcg_batch_destroy(gj_rrcg_batch *b) {
    if (!b) return;
    cudaEventSynchronize(b->used);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    cudaEventDestroy(b->used);
    delete b;
}

// ---------------------------------------------------------------------------
// Host-buffer form of the one-shot solve: the inputs are copied to the device,
// the solve runs as in gj_rrcg_joint_solve, and the models are copied back.

extern "C" gj_status gj_rrcg_joint_solve_host(const gj_op *const ops[2], const gj_rrcg_params *P,
                                              const void *const dobs[2], const void *const sigma[2],
                                              const void *const m_apr[2], const void *const w_depth[2],
                                              const void *const w_hard[2], void *const m[2], gj_rrcg_report *rep,
                                              gj_stream_t stream) {
    gj_status rc = check_ops(ops);
    if (rc != GJ_OK) return rc;
    if (!P || !dobs || !sigma || !w_depth || !m || !rep) {
        set_error("gj_rrcg_joint_solve_host: NULL argument");
        return GJ_ERR_ARG;
    }
    for (int i = 0; i < 2; ++i)
        if (!dobs[i] || !sigma[i] || !w_depth[i] || !m[i]) {
            set_error("gj_rrcg_joint_solve_host: NULL vector");
            return GJ_ERR_ARG;
        }
    const gj_op *o = ops[0];
    const size_t es = elem_bytes(o->prec);
    const size_t n = (size_t)o->nx * o->ny * o->nz, s = (size_t)o->sx * o->sy, nz = (size_t)o->nz;
    // one device block: dobs, sigma (s each), w_depth (nz), m, m_apr, w_hard (n each), per field
    size_t per = 2 * s + nz + n;
    if (m_apr && (m_apr[0] || m_apr[1])) per += n;
    if (w_hard && (w_hard[0] || w_hard[1])) per += n;
    char *blk = nullptr;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if ((rc = not_capturing(st, "gj_rrcg_joint_solve_host")) != GJ_OK) return rc;
    cudaError_t e = pool_alloc(reinterpret_cast<void **>(&blk), 2 * per * es, st);
    if (e != cudaSuccess) return cuda_fail(e, "gj_rrcg_joint_solve_host: device buffers");
    const void *d_dobs[2], *d_sig[2], *d_wdep[2], *d_mapr[2] = {nullptr, nullptr}, *d_wh[2] = {nullptr, nullptr};
    void *d_m[2];
    char *at = blk;
    auto put = [&](const void *src, size_t count) -> const void * {
        void *dst = at;
        at += count * es;
        if (src && e == cudaSuccess) e = cudaMemcpyAsync(dst, src, count * es, cudaMemcpyHostToDevice, st);
        return dst;
    };
    for (int i = 0; i < 2; ++i) {
        d_dobs[i] = put(dobs[i], s);
        d_sig[i] = put(sigma[i], s);
        d_wdep[i] = put(w_depth[i], nz);
        d_m[i] = const_cast<void *>(put(m[i], n));
        if (m_apr && (m_apr[0] || m_apr[1])) {
            const void *p = put(m_apr[i], n);
            d_mapr[i] = m_apr[i] ? p : nullptr;
        }
        if (w_hard && (w_hard[0] || w_hard[1])) {
            const void *p = put(w_hard[i], n);
            d_wh[i] = w_hard[i] ? p : nullptr;
        }
    }
    if (e != cudaSuccess) {
        cudaStreamSynchronize(st);  // (freeing pool memory does not wait for the copies)
        cudaFree(blk);
        return cuda_fail(e, "gj_rrcg_joint_solve_host: copies in");
    }
    rc = gj_rrcg_joint_solve(ops, P, d_dobs, d_sig, d_mapr, d_wdep, d_wh, d_m, nullptr, rep, stream);
    if (rc == GJ_OK || rc == GJ_ERR_NONFINITE) {
        for (int i = 0; i < 2 && e == cudaSuccess; ++i)
            e = cudaMemcpyAsync(m[i], d_m[i], n * es, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) {
            cudaStreamSynchronize(st);
            rc = cuda_fail(e, "gj_rrcg_joint_solve_host: copies out");
        }
    } else {
        cudaStreamSynchronize(st);  // a refused solve leaves the copies in behind
    }
    cudaFree(blk);
    return rc;
}
