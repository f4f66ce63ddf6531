// Kernels of the BTTB/BCCB sensitivity products (Sec. 2.7.1).
//
// A 2-D transform of an Ny x Nx layer is split into a row pass (length Nx, along x)
// and a column pass (length Ny, along y).  Real rows are transformed two at a time
// as one complex sequence (a + i b); the half spectrum of each is recovered from
// Z[k] and Z[N-k].  Only ncol = Nx/2 + 1 columns are kept.  Zero padding is never
// stored: the first stage of each transform skips the inputs beyond the data.
//
// Forward product, one launch a pass: rows (m -> Z) -> columns, multiplied by the layer
// spectra and summed over layers on chip (between layer groups through Y), and inverse
// columns of the sum (Z -> W) -> inverse rows cropped to the stations (W -> d).  Adjoint:
// rows (r -> W) -> columns kept on chip (V^), and per layer the inverse columns of
// conj(T^_r) V^ (W -> Z) -> inverse rows cropped to the prisms (Z -> g).
#pragma once
#include <utility>

#include "fft.cuh"

namespace gj {

template <typename R>
struct OpView {
    int sx, sy, nx, ny, nz, Nx, Ny, ncol;
    FftPlanDev px, py;
    const cpx<R> *twx;   // W_Nx^k, k < Nx
    const cpx<R> *twy;   // W_Ny^k, k < Ny
    const cpx<R> *spec;  // [nz][Ny][ncol] layer spectra / (Nx Ny)
    cpx<R> *Z;           // [nz*ny][ncol]  row-pass output / adjoint column output
    cpx<R> *Y;           // [slots][Ny][ncol]  layer groups' partial sums
    int *cnt;            // [ncol]         arrivals of a column tile's layer groups, zero between launches
    cpx<R> *W;           // [max(sy, ...)][ncol]  inverse-column output / residual rows
    cpx<R> *V;           // fast paths: data-row spectra [ncol][Ny/2] of the adjoint (unused otherwise)
    int real_spec;       // fast path: spec holds the real, even spectrum of an even table for
                         // ky <= Ny/2 only, R[nz][ncol][even_spec_len(Ny)]
    int split_half;      // 1: the row passes halve the split spectra; 0: the factor is in `spec`
    int tcol;            // 0: Z, W, V row-major ([line][ncol]); > 0: transposed, line iy of layer r and
                         // bin k at ((r * ncol + k) * tcol + iy) (the N_y = 1024 column kernels' layout)
};

// Stored entries per column of a real, even spectrum (fast path): ky = 0 .. Ny/2,
// padded to a multiple of four values so that every column starts on 16 bytes.
__host__ __device__ constexpr int even_spec_len(int Ny) { return Ny / 2 + 4; }

// How real lines are paired into complex transforms.
struct PairMap {
    int nlines;  // lines per side
    int joint;   // 1: pair q = (line q of op0, line q of op1); 0: lines (2q, 2q+1) of op0
    int lpl;     // lines per layer (0: one layer), for the transposed layout
    __device__ __forceinline__ int npairs() const { return joint ? nlines : (nlines + 1) >> 1; }
    __device__ __forceinline__ void lines(int q, int &la, int &lb, bool &hasb) const {
        if (joint) { la = q; lb = q; hasb = true; }
        else { la = 2 * q; lb = 2 * q + 1; hasb = lb < nlines; }
    }
    // element (line, bin k) of a row pass's output or input
    __device__ __forceinline__ size_t at(int line, int k, int ncol, int tcol) const {
        if (!tcol) return (size_t)line * ncol + k;
        const int L = lpl > 0 ? lpl : nlines;
        const int r = line / L;
        return ((size_t)r * ncol + k) * tcol + (line - r * L);
    }
};

__device__ __forceinline__ bool stopped(const int *done) {
    return done != nullptr && *(volatile const int *)done != 0;
}

// Block-strided loop over it < total in batches of U elements per thread: the U
// loads of a batch are issued before any of its stores, so that a thread keeps U
// global reads in flight instead of one.
template <int U, class Load, class Store>
__device__ __forceinline__ void staged_loop(int total, Load load, Store store) {
    for (int it0 = threadIdx.x; it0 < total; it0 += U * blockDim.x) {
        decltype(load(0)) v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int it = it0 + u * (int)blockDim.x;
            if (it < total) v[u] = load(it);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int it = it0 + u * (int)blockDim.x;
            if (it < total) store(it, v[u]);
        }
    }
}
// The same with the first batch taken apart: loads(...) issues it, stores(...) hands it over and
// runs the rest of the loop, so that other loads and waits can stand between the two.
template <int U, class Load>
struct FirstBatch {
    decltype(std::declval<Load>()(0)) v[U];
    __device__ __forceinline__ void loads(int total, const Load &load) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int it = threadIdx.x + u * (int)blockDim.x;
            if (it < total) v[u] = load(it);
        }
    }
    template <class Store>
    __device__ __forceinline__ void stores(int total, const Load &load, const Store &store) {
        for (int it0 = threadIdx.x; it0 < total;) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int it = it0 + u * (int)blockDim.x;
                if (it < total) store(it, v[u]);
            }
            it0 += U * blockDim.x;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int it = it0 + u * (int)blockDim.x;
                if (it < total) v[u] = load(it);
            }
        }
    }
};

// Static shared memory of the row passes: block_accumulate's scratch (four sums of the eight
// warps) and the functors' scalars.  gj_op_tune accepts tiles up to what is left beside
// kStaticSmem, so it must stay below that.
constexpr int kRowSums = 4 * 8, kRowScalars = 8;
constexpr size_t kStaticSmem = 1024;
static_assert((kRowSums + kRowScalars) * sizeof(double) <= kStaticSmem, "a tile that gj_op_tune accepts must launch");

// Elements of a row functor's loops in flight per thread.
template <typename R> constexpr int kRowU = sizeof(R) == 8 ? 2 : 4;

// ---------------------------------------------------------------------------
// Plain functors.

// row length of the staged functor rows of the 512 row passes (pre[a][i][kStageRow])
constexpr int kStageRow = 256;

template <typename R>
struct LoadPlain {  // a = x0[la*pitch + j], b = x1[lb*pitch + j]
    const R *x0;
    const R *x1;
    int pitch;
    static constexpr int NPRE = 1;  // rows la of x0 and lb of x1, staged by the 512 team passes
    __device__ const R *pre_src(int, int i) const { return i == 0 ? x0 : x1; }
    using Real = R;
    static constexpr int NS = 0;
    __device__ __forceinline__ R scalar(int) const { return R(0); }
    __device__ __forceinline__ void begin() {}
    __device__ __forceinline__ void set(const R *) {}
    __device__ void init() {}
    struct Raw { R a, b; };
    __device__ __forceinline__ Raw load(int la, int lb, bool hb, int j) const {
        const R a = x0[(size_t)la * pitch + j];
        const R b = *(hb ? x1 + (size_t)lb * pitch + j : x0 + (size_t)la * pitch + j);  // (no branch between loads)
        return Raw{a, hb ? b : R(0)};
    }
    __device__ __forceinline__ void apply(const Raw &q, int, int, bool, int, R &a, R &b) const {
        a = q.a;
        b = q.b;
    }
    __device__ __forceinline__ void fetch(int la, int lb, bool hb, int j, R &a, R &b) const {
        apply(load(la, lb, hb, j), la, lb, hb, j, a, b);
    }
    // elements j0 + k * stride (k < K) below n; zero beyond
    template <int K, bool PRE = false>
    __device__ __forceinline__ void fetch_batch(int la, int lb, bool hb, int j0, int stride, int n, R (&a)[K],
                                                R (&b)[K], const R *pre = nullptr) const {
        const R *pa = PRE ? pre : x0 + (size_t)la * pitch;
        const R *pb = PRE ? pre + kStageRow : x1 + (size_t)lb * pitch;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = j0 + k * stride;
            a[k] = j < n ? pa[j] : R(0);
            b[k] = (hb && j < n) ? pb[j] : R(0);
        }
    }
    __device__ __forceinline__ void flush(double *) const {}
};

template <typename R>
struct StorePlain {
    R *y0;
    R *y1;
    int pitch;
    static constexpr int NPRE = 0;  // reads nothing
    __device__ const R *pre_src(int, int) const { return nullptr; }
    __device__ __forceinline__ void prefetch(int, int, bool, int, int) const {}
    using Real = R;
    static constexpr int NS = 0;
    __device__ __forceinline__ R scalar(int) const { return R(0); }
    __device__ __forceinline__ void begin() {}
    __device__ __forceinline__ void set(const R *) {}
    __device__ void init() {}
    struct Raw {};
    __device__ __forceinline__ Raw load(int, int, bool, int) const { return Raw{}; }
    __device__ __forceinline__ void apply(const Raw &, int la, int lb, bool hb, int j, R a, R b) const {
        y0[(size_t)la * pitch + j] = a;
        if (hb) y1[(size_t)lb * pitch + j] = b;
    }
    __device__ __forceinline__ void store(int la, int lb, bool hb, int j, R a, R b) const {
        apply(Raw{}, la, lb, hb, j, a, b);
    }
    template <int K, bool PRE = false>
    __device__ __forceinline__ void store_batch(int la, int lb, bool hb, int j0, int stride, int n, const R (&a)[K],
                                                const R (&b)[K], const R * = nullptr) const {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = j0 + k * stride;
            if (j < n) {
                y0[(size_t)la * pitch + j] = a[k];
                if (hb) y1[(size_t)lb * pitch + j] = b[k];
            }
        }
    }
    __device__ __forceinline__ void flush(double *) const {}
};

// ---------------------------------------------------------------------------
// Two fields' single-field products in one launch (the pair calls): a functor per
// field, the one of field f taken with field_functor(pro, f).  The solver's data-line
// epilogues take the field there too; every other functor serves its launch's lines as it is.
template <typename R>
struct LoadPlain2 {  // field f: lines la and lb of x[f]
    const R *x[2];
    int pitch;
    static constexpr int NPRE = LoadPlain<R>::NPRE;
    using Real = R;
    static constexpr int NS = 0;
    __device__ __forceinline__ R scalar(int) const { return R(0); }
    __device__ __forceinline__ void begin() {}
    __device__ __forceinline__ void set(const R *) {}
    __device__ void init() {}
    __device__ void flush(double *) const {}
    __device__ LoadPlain<R> of(int f) const {  // a select, not an indexed load
        const R *p = f ? x[1] : x[0];
        return LoadPlain<R>{p, p, pitch};
    }
};
template <typename R>
struct StorePlain2 {  // field f: lines la and lb of y[f]
    R *y[2];
    int pitch;
    static constexpr int NPRE = StorePlain<R>::NPRE;
    using Real = R;
    static constexpr int NS = 0;
    __device__ __forceinline__ R scalar(int) const { return R(0); }
    __device__ __forceinline__ void begin() {}
    __device__ __forceinline__ void set(const R *) {}
    __device__ void init() {}
    __device__ void flush(double *) const {}
    __device__ StorePlain<R> of(int f) const {  // a select, not an indexed load
        R *p = f ? y[1] : y[0];
        return StorePlain<R>{p, p, pitch};
    }
};
template <class P>
__device__ __forceinline__ P &field_functor(P &p, int) { return p; }
template <typename R>
__device__ __forceinline__ LoadPlain<R> field_functor(const LoadPlain2<R> &p, int f) { return p.of(f); }
template <typename R>
__device__ __forceinline__ StorePlain<R> field_functor(const StorePlain2<R> &p, int f) { return p.of(f); }
template <typename R>
__device__ __forceinline__ LoadPlain<R> field_functor(LoadPlain2<R> &p, int f) { return p.of(f); }
template <typename R>
__device__ __forceinline__ StorePlain<R> field_functor(StorePlain2<R> &p, int f) { return p.of(f); }

// Launch shape of a row pass: P line pairs per CTA, element j of pair p at j * pitch + p
// (odd pitch: the global accesses run along j, the butterflies along p, and neither
// meets its own banks).
struct RowShape {
    int P, pitch;
    unsigned mP;
};

// Launch shape of a column pass: a CTA takes C columns and G layers of them at a time
// (B = C G interleaved lines, column fastest), L layers in all.
struct ColShape {
    int C, G, L;
    int pitch;       // of the C G lines
    int pitch1;      // of the C lines of the residual or summed spectrum
    unsigned mB, mC;
    int arrivals;    // layer groups of a column tile (1: the sum stays on chip)
};

template <typename C>
__device__ __forceinline__ void load_twiddles(C *tw, const C *src, int N) {
    for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = src[i];
}
// the same as asynchronous copies: the caller waits (cp_async_wait) before a barrier that
// precedes the first use
template <typename C>
__device__ __forceinline__ void copy_twiddles(C *tw, const C *src, int N) {
    for (int i = threadIdx.x; i < N; i += blockDim.x) cp_async(tw + i, src + i);
    cp_async_commit();
}
// The stop flag of a solve, read but not yet waited for (see stopped).
__device__ __forceinline__ int stop_flag(const int *done) { return done ? __ldcg(done) : 0; }

// In-place forward transform of P lines staged in buf0 (elements < valid): returns the
// buffer that holds the result (buf0 or buf1).  Ends with a barrier.
template <typename R, bool INV>
__device__ __forceinline__ cpx<R> *fft_staged(const FftPlanDev &plan, const RowShape &rs, cpx<R> *buf0, cpx<R> *buf1,
                                              const cpx<R> *tw, int valid, int need) {
    using C = cpx<R>;
    const int pitch = rs.pitch;
    C *X = (plan.nst & 1) ? buf1 : buf0;  // the buffer that the last stage does not read
    auto in = [&](int j, int p) { return j < valid ? buf0[j * pitch + p] : czero<C>(); };
    auto out = [&](int n, int p, C x) { X[n * pitch + p] = x; };
    fft_run<R, INV, !INV, INV>(plan, rs.P, rs.mP, pitch, buf1, buf0, tw, valid, need, in, out);
    __syncthreads();
    return X;
}

// The split of P transforms Z = FFT(a + i b) into the half spectra of their real lines:
// A[k] = (Z[k] + conj Z[N-k]) / 2, B[k] = (Z[k] - conj Z[N-k]) / 2i.
template <typename R>
__device__ __forceinline__ void split_lines(const OpView<R> &op, const PairMap &pm, const RowShape &rs, int q0,
                                            const cpx<R> *X, cpx<R> *out0, cpx<R> *out1) {
    using C = cpx<R>;
    const int N = op.Nx, ncol = op.ncol, np = pm.npairs();
    const unsigned mcol = div_magic(ncol);
    for (int it = threadIdx.x; it < ncol * rs.P; it += blockDim.x) {
        int p, k;
        if (op.tcol) { k = fast_div(it, rs.mP); p = it - k * rs.P; }  // consecutive lines are consecutive words
        else { p = fast_div(it, mcol); k = it - p * ncol; }
        const int q = q0 + p;
        if (q >= np) continue;
        const C zk = X[k * rs.pitch + p];
        const C zm = X[(k ? N - k : 0) * rs.pitch + p];
        int la, lb; bool hb;
        pm.lines(q, la, lb, hb);
        C A = mk<C>(zk.x + zm.x, zk.y - zm.y), B = mk<C>(zk.y + zm.y, zm.x - zk.x);
        if (op.split_half) {
            A = mk<C>(R(0.5) * A.x, R(0.5) * A.y);
            B = mk<C>(R(0.5) * B.x, R(0.5) * B.y);
        }
        out0[pm.at(la, k, ncol, op.tcol)] = A;
        if (hb) out1[pm.at(lb, k, ncol, op.tcol)] = B;
    }
}

// The Hermitian-extended A + i B of P pairs of half spectra into a buffer (each read once).
template <typename R>
struct SpectraStage {
    using C = cpx<R>;
    struct Two { C a, b; };
    const OpView<R> &op;
    PairMap pm;
    RowShape rs;
    int q0;
    const C *in0, *in1;
    unsigned mcol;
    __device__ __forceinline__ void at(int it, int &p, int &k) const {
        if (op.tcol) { k = fast_div(it, rs.mP); p = it - k * rs.P; }
        else { p = fast_div(it, mcol); k = it - p * op.ncol; }
    }
    __device__ __forceinline__ Two operator()(int it) const {
        int p, k;
        at(it, p, k);
        const int np = pm.npairs();
        int la, lb; bool hb;
        pm.lines(min(q0 + p, np - 1), la, lb, hb);
        Two t{in0[pm.at(la, k, op.ncol, op.tcol)], czero<C>()};
        if (hb) t.b = in1[pm.at(lb, k, op.ncol, op.tcol)];
        return t;
    }
    __device__ __forceinline__ void put(C *buf, int it, Two t) const {
        int p, k;
        at(it, p, k);
        const int N = op.Nx;
        const bool self = k == 0 || 2 * k == N;
        if (self) { t.a.y = 0; t.b.y = 0; }
        buf[k * rs.pitch + p] = mk<C>(t.a.x - t.b.y, t.a.y + t.b.x);
        if (!self) buf[(N - k) * rs.pitch + p] = mk<C>(t.a.x + t.b.y, t.b.x - t.a.y);
    }
};

// ---------------------------------------------------------------------------
// Row pass, real -> half spectrum.  Pro::fetch(la, lb, hasb, j, a, b) supplies the
// two real inputs of element j (< n_in); Pro::flush(scratch) runs once per block.
// grid y: the field of the pair calls (Pro2 functors).
template <typename R, class Pro>
__global__ void __launch_bounds__(256) k_row_fwd(OpView<R> op, PairMap pm, int n_in, RowShape rs,
                                                 cpx<R> *out0, cpx<R> *out1, Pro pro, const int *done) {
    using C = cpx<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = op.Nx, P = rs.P, ncol = op.ncol;
    C *buf0 = reinterpret_cast<C *>(smem_raw);
    C *buf1 = buf0 + N * rs.pitch;
    C *tw = buf1 + N * rs.pitch;
    __shared__ double red[kRowSums];
    __shared__ R sc[kRowScalars];
    pdl_go();
    copy_twiddles(tw, op.twx, N);
    pdl_wait();
    // the stop flag, the functor's scalars and the first elements: one memory latency for all
    const int stop = stop_flag(done);
    pro.begin();
    static_assert(Pro::NS <= kRowScalars, "scalars");
    R mine = R(0);
    if (threadIdx.x < Pro::NS) mine = pro.scalar((int)threadIdx.x);
    const int field = blockIdx.y;
    const int q0 = blockIdx.x * P;
    const int np = pm.npairs();
    const unsigned mn = div_magic(n_in);
    auto load = [&](int it) {
        const int p = fast_div(it, mn), j = it - p * n_in, q = q0 + p;
        int la, lb; bool hb;
        pm.lines(min(q, np - 1), la, lb, hb);
        return field_functor(pro, field).load(la, lb, hb, j);
    };
    FirstBatch<kRowU<R>, decltype(load)> first;
    first.loads(n_in * P, load);
    if (stop) {
        cp_async_wait<0>();
        return;
    }
    if constexpr (Pro::NS > 0) {
        if (threadIdx.x < Pro::NS) sc[threadIdx.x] = mine;
        __syncthreads();
    }
    pro.set(sc);
    first.stores(n_in * P, load, [&](int it, const auto &raw) {
        const int p = fast_div(it, mn), j = it - p * n_in, q = q0 + p;
        R a = 0, b = 0;
        if (q < np) {
            int la, lb; bool hb;
            pm.lines(q, la, lb, hb);
            field_functor(pro, field).apply(raw, la, lb, hb, j, a, b);
        }
        buf0[j * rs.pitch + p] = mk<C>(a, b);
    });
    cp_async_wait<0>();
    __syncthreads();
    const C *X = fft_staged<R, false>(op.px, rs, buf0, buf1, tw, n_in, N);
    split_lines<R>(op, pm, rs, q0, X, field ? out1 : out0, pm.joint ? out1 : (field ? out1 : out0));
    pro.flush(red);
}

// ---------------------------------------------------------------------------
// Row pass, half spectrum -> real, cropped to n_out.  Epi::store(la, lb, hasb, j, a, b).
template <typename R, class Epi>
__global__ void __launch_bounds__(256) k_row_inv(OpView<R> op, PairMap pm, int n_out, RowShape rs,
                                                 const cpx<R> *in0, const cpx<R> *in1, Epi epi,
                                                 const int *done) {
    using C = cpx<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = op.Nx, P = rs.P, ncol = op.ncol;
    C *buf0 = reinterpret_cast<C *>(smem_raw);
    C *buf1 = buf0 + N * rs.pitch;
    C *tw = buf1 + N * rs.pitch;
    __shared__ double red[kRowSums];
    __shared__ R sc[kRowScalars];
    pdl_go();
    copy_twiddles(tw, op.twx, N);
    pdl_wait();
    const int stop = stop_flag(done);
    epi.begin();
    static_assert(Epi::NS <= kRowScalars, "scalars");
    R mine = R(0);
    if (threadIdx.x < Epi::NS) mine = epi.scalar((int)threadIdx.x);
    const int field = blockIdx.y;
    const int q0 = blockIdx.x * P;
    const int np = pm.npairs();
    const SpectraStage<R> ss{op, pm, rs, q0, field ? in1 : in0, pm.joint ? in1 : (field ? in1 : in0), div_magic(ncol)};
    FirstBatch<4, SpectraStage<R>> first;
    first.loads(ncol * P, ss);
    if (stop) {
        cp_async_wait<0>();
        return;
    }
    if (threadIdx.x < Epi::NS) sc[threadIdx.x] = mine;
    first.stores(ncol * P, ss, [&](int it, const auto &t) { ss.put(buf0, it, t); });
    cp_async_wait<0>();
    __syncthreads();
    epi.set(sc);
    const C *X = fft_staged<R, true>(op.px, rs, buf0, buf1, tw, N, n_out);
    const unsigned mn = div_magic(n_out);
    auto &&fn = field_functor(epi, field);
    using Raw = decltype(fn.load(0, 0, false, 0));
    staged_loop<kRowU<R>>(
        n_out * P,
        [&](int it) {
            const int p = fast_div(it, mn), j = it - p * n_out;
            int la, lb; bool hb;
            pm.lines(min(q0 + p, np - 1), la, lb, hb);
            return fn.load(la, lb, hb, j);
        },
        [&](int it, const Raw &raw) {
            const int p = fast_div(it, mn), j = it - p * n_out, q = q0 + p;
            if (q >= np) return;
            int la, lb; bool hb;
            pm.lines(q, la, lb, hb);
            const C z = X[j * rs.pitch + p];
            fn.apply(raw, la, lb, hb, j, z.x, z.y);
        });
    fn.flush(red);
}

// Data-line pass of the solver: inverse rows of the cropped forward product, the residual
// epilogue (residual turns the predicted data into W_d r~), and the forward rows of the
// result for the adjoint's column pass.  Two lines of one field share a transform (grid y = field): magnetic data are
// some 200 times the gravity data and W_d r~ the other way round, and a transform that carried
// a line of each rounded each field by the larger one (50x30x10 FP32, 20 iterations, the worst
// of ten surveys: Phi and the models off by up to 7.7e-6, by 1.7e-7 and 2.5e-7 since, in the same
// time).
template <typename R, class Epi>
__global__ void __launch_bounds__(256) k_row_resid(OpView<R> op, PairMap pm, int n_out, RowShape rs,
                                                   const cpx<R> *in0, const cpx<R> *in1, cpx<R> *out0, cpx<R> *out1,
                                                   Epi epi, const int *done) {
    using C = cpx<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = op.Nx, P = rs.P, ncol = op.ncol;
    C *buf0 = reinterpret_cast<C *>(smem_raw);
    C *buf1 = buf0 + N * rs.pitch;
    C *tw = buf1 + N * rs.pitch;
    __shared__ double red[kRowSums];
    pdl_go();
    copy_twiddles(tw, op.twx, N);
    pdl_wait();
    const int stop = stop_flag(done);
    const int field = blockIdx.y;
    const int q0 = blockIdx.x * P;
    const int np = pm.npairs();
    const C *in = field ? in1 : in0;
    C *out = field ? out1 : out0;
    const SpectraStage<R> ss{op, pm, rs, q0, in, in, div_magic(ncol)};
    FirstBatch<4, SpectraStage<R>> first;
    first.loads(ncol * P, ss);
    if (stop) {
        cp_async_wait<0>();
        return;
    }
    epi.set(nullptr);
    first.stores(ncol * P, ss, [&](int it, const auto &t) { ss.put(buf0, it, t); });
    cp_async_wait<0>();
    __syncthreads();
    C *X = fft_staged<R, true>(op.px, rs, buf0, buf1, tw, N, n_out);
    const unsigned mn = div_magic(n_out);
    auto &&fn = field_functor(epi, field);
    staged_loop<kRowU<R>>(
        n_out * P,
        [&](int it) {
            const int p = fast_div(it, mn), j = it - p * n_out;
            int la, lb; bool hb;
            pm.lines(min(q0 + p, np - 1), la, lb, hb);
            return fn.load(la, lb, hb, j);
        },
        [&](int it, const typename Epi::Raw &raw) {
            const int p = fast_div(it, mn), j = it - p * n_out;
            C z = X[j * rs.pitch + p];
            if (q0 + p < np) {
                int la, lb; bool hb;
                pm.lines(q0 + p, la, lb, hb);
                fn.residual(raw, hb, z.x, z.y);
            }
            X[j * rs.pitch + p] = z;
        });
    __syncthreads();
    const C *Y = fft_staged<R, false>(op.px, rs, X, X == buf0 ? buf1 : buf0, tw, n_out, N);
    split_lines<R>(op, pm, rs, q0, Y, out, out);
    fn.flush(red);
}

// ---------------------------------------------------------------------------
// Column pass of the forward product: for a tile of C columns and a group of layers,
// sum_r T^_r . FFT_y(Z_r); the last group of a tile to arrive takes the sum of all
// groups (through Y) and writes W[jy] = IFFT_y(sum)[jy], jy < sy.  With one group the sum
// never leaves the CTA.

// Sources and sinks of the column passes.  Absent columns, layers and rows are clamped to
// present ones and masked afterwards, so that a butterfly's loads are unconditional and go
// out together: behind a branch each waited for the one before it (a layer of N = 256 took
// 16 memory latencies; 128x128x32 FP32, both fields: 66 us for the forward columns).
struct LineMap {  // line b of a group -> layer and column
    unsigned mC;
    int C, cols, rg, r1;
    __device__ __forceinline__ void at(int b, int &r, int &c) const {
        const int g = fast_div(b, mC);
        c = b - g * C;
        r = rg + g;
    }
    __device__ __forceinline__ bool clamp(int &r, int &c) const {
        const bool ok = c < cols && r < r1;
        c = min(c, cols - 1);
        r = min(r, r1 - 1);
        return ok;
    }
};
template <typename R>
struct FromZ {  // column elements of the row-pass output
    const OpView<R> &op;
    const cpx<R> *Z;  // column c0
    LineMap lm;
    __device__ __forceinline__ cpx<R> operator()(int j, int b) const {
        int r, c;
        lm.at(b, r, c);
        const bool ok = lm.clamp(r, c) && j < op.ny;
        const cpx<R> z = Z[((size_t)r * op.ny + min(j, op.ny - 1)) * op.ncol + c];
        return ok ? z : czero<cpx<R>>();
    }
};
template <typename R>
struct IntoSum {  // times the layer's spectrum, added to this thread's own entry of acc
    const OpView<R> &op;
    const cpx<R> *T;  // column c0
    LineMap lm;
    cpx<R> *acc;
    int pitch;
    bool first;
    __device__ __forceinline__ cpx<R> pre(int n, int b) const {
        int r, c;
        lm.at(b, r, c);
        lm.clamp(r, c);
        return __ldg(T + ((size_t)r * op.Ny + n) * op.ncol + c);
    }
    __device__ __forceinline__ void operator()(int n, int b, cpx<R> x, cpx<R> t) const {
        int r, c;
        lm.at(b, r, c);
        cpx<R> y = cmul(x, t);
        if (!lm.clamp(r, c)) y = czero<cpx<R>>();
        cpx<R> *a = acc + n * pitch + b;
        *a = first ? y : cadd(*a, y);
    }
};
template <typename R>
struct FromVhat {  // conj(spectrum) times the residual's column transform
    const OpView<R> &op;
    const cpx<R> *T;
    LineMap lm;
    const cpx<R> *vh;
    int pitch1;
    __device__ __forceinline__ cpx<R> operator()(int k, int b) const {
        int r, c;
        lm.at(b, r, c);
        const cpx<R> v = vh[k * pitch1 + c];
        lm.clamp(r, c);
        return cmulc(v, __ldg(T + ((size_t)r * op.Ny + k) * op.ncol + c));
    }
};

template <typename R>
__global__ void __launch_bounds__(256) k_col_fwd(OpView<R> op0, OpView<R> op1, ColShape cs, const int *done) {
    using Cx = cpx<R>;
    pdl_go();
    const OpView<R> &op = blockIdx.z ? op1 : op0;
    const int C = cs.C, G = cs.G, pitch = cs.pitch;
    const int c0 = blockIdx.x * C;
    const int r0 = blockIdx.y * cs.L;
    if (r0 >= op.nz || c0 >= op.ncol) return;
    const int r1 = min(r0 + cs.L, op.nz);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int last_in;
    const int N = op.Ny, ny = op.ny, ncol = op.ncol;
    const int cols = min(C, ncol - c0);
    Cx *bufA = reinterpret_cast<Cx *>(smem_raw);
    Cx *bufB = bufA + N * pitch;
    Cx *acc = bufB + N * pitch;
    Cx *tw = acc + N * pitch;
    load_twiddles(tw, op.twy, N);
    pdl_wait();
    if (stopped(done)) return;
    bool first = true;
    for (int rg = r0; rg < r1; rg += G) {
        const LineMap lm{cs.mC, C, cols, rg, r1};
        const FromZ<R> in{op, op.Z + c0, lm};
        const IntoSum<R> out{op, op.spec + c0, lm, acc, pitch, first};
        fft_run<R, false, true, false>(op.py, C * G, cs.mB, pitch, bufA, bufB, tw, ny, N, in, out);
        first = false;
        if (!(op.py.nst & 1)) { Cx *t = bufA; bufA = bufB; bufB = t; }  // the last stage may still be reading bufA
    }
    __syncthreads();
    auto tile_sum = [&](int k, int c) {
        Cx y = acc[k * pitch + c];
        for (int g = 1; g < G; ++g) y = cadd(y, acc[k * pitch + g * C + c]);
        return y;
    };
    // The groups of a tile meet in Y, a slot each, and the last to arrive adds them in the
    // order of the layers, so that a product repeats bit for bit.
    const size_t plane = (size_t)N * ncol;
    Cx *Yt = op.Y + c0;
    const int slots = cs.arrivals;
    if (slots > 1) {
        Cx *Ys = Yt + blockIdx.y * plane;
        for (int it = threadIdx.x; it < N * C; it += blockDim.x) {
            const int k = fast_div(it, cs.mC), c = it - k * C;
            if (c < cols) Ys[(size_t)k * ncol + c] = tile_sum(k, c);
        }
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last_in = atomicAdd(op.cnt + blockIdx.x, 1) == slots - 1;
        __syncthreads();
        if (!last_in) return;
        __threadfence();
        if (threadIdx.x == 0) op.cnt[blockIdx.x] = 0;
        // Two elements and four slots of loads in flight a thread.  (Summed inside the inverse
        // transform's first stage, every input waited for its slots one by one: the sums of
        // eight groups cost 16 us of a 128x128x32 product's 45 us column pass.)
        staged_loop<2>(
            N * C,
            [&](int it) {
                const int k = fast_div(it, cs.mC), c = it - k * C;
                const Cx *y = Yt + (size_t)k * ncol + min(c, cols - 1);  // (an absent column's result is dropped)
                Cx t = __ldcg(y);
                for (int s = 1; s < slots; s += 4) {
                    Cx v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) v[u] = s + u < slots ? __ldcg(y + (s + u) * plane) : czero<Cx>();
#pragma unroll
                    for (int u = 0; u < 4; ++u) t = cadd(t, v[u]);
                }
                return t;
            },
            [&](int it, Cx t) {
                const int k = fast_div(it, cs.mC), c = it - k * C;
                acc[k * pitch + c] = t;
            });
        __syncthreads();
    }
    if (slots == 1 && G > 1) {
        // (inside the inverse's first stage a thread added the layers of every input in turn)
        for (int it = threadIdx.x; it < N * C; it += blockDim.x) {
            const int k = fast_div(it, cs.mC), c = it - k * C;
            acc[k * pitch + c] = tile_sum(k, c);
        }
        __syncthreads();
    }
    auto in = [&](int k, int c) { return acc[k * pitch + c]; };  // the sum of all layers
    auto out = [&](int n, int c, Cx x) {
        if (n < op.sy && c < cols) op.W[(size_t)n * ncol + c0 + c] = x;
    };
    fft_run<R, true, false, true>(op.py, C, cs.mC, cs.pitch1, bufA, bufB, tw, N, op.sy, in, out);
}

// Column pass of the adjoint product: V^ = FFT_y(W) of a tile of C columns (W has sy
// nonzero rows), kept on chip; then for each layer of the group
// Z_r = IFFT_y(conj(T^_r) . V^), rows iy < ny.
template <typename R>
__global__ void __launch_bounds__(256) k_col_adj(OpView<R> op0, OpView<R> op1, ColShape cs, const int *done) {
    using Cx = cpx<R>;
    pdl_go();
    const OpView<R> &op = blockIdx.z ? op1 : op0;
    const int C = cs.C, G = cs.G, pitch1 = cs.pitch1;
    const int c0 = blockIdx.x * C;
    const int r0 = blockIdx.y * cs.L;
    if (c0 >= op.ncol || r0 >= op.nz) return;
    const int r1 = min(r0 + cs.L, op.nz);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = op.Ny, ncol = op.ncol, ny = op.ny;
    const int cols = min(C, ncol - c0);
    Cx *bufA = reinterpret_cast<Cx *>(smem_raw);
    Cx *bufB = bufA + N * cs.pitch;
    Cx *vh = bufB + N * cs.pitch;
    Cx *tw = vh + N * pitch1;
    load_twiddles(tw, op.twy, N);
    pdl_wait();
    if (stopped(done)) return;
    {
        auto in = [&](int j, int c) {
            const Cx w = op.W[(size_t)min(j, op.sy - 1) * ncol + c0 + min(c, cols - 1)];
            return (j < op.sy && c < cols) ? w : czero<Cx>();
        };
        auto out = [&](int n, int c, Cx x) { vh[n * pitch1 + c] = x; };
        fft_run<R, false, true, false>(op.py, C, cs.mC, pitch1, bufA, bufB, tw, op.sy, N, in, out);
    }
    __syncthreads();
    for (int rg = r0; rg < r1; rg += G) {
        const FromVhat<R> in{op, op.spec + c0, LineMap{cs.mC, C, cols, rg, r1}, vh, pitch1};
        auto out = [&](int n, int b, Cx x) {
            const int g = fast_div(b, cs.mC), c = b - g * C, r = rg + g;
            if (n < ny && c < cols && r < r1) op.Z[((size_t)r * ny + n) * ncol + c0 + c] = x;
        };
        fft_run<R, true, false, true>(op.py, C * G, cs.mB, cs.pitch, bufA, bufB, tw, N, ny, in, out);
        if (!(op.py.nst & 1)) { Cx *t = bufA; bufA = bufB; bufB = t; }  // the last stage may still be reading bufA
    }
}

// ---------------------------------------------------------------------------
// Column passes of the recompute mode, one layer a launch: the FP64 column transform of
// the layer's table rows (Zs) gives the layer's spectrum of a tile of C columns, which is
// rounded to R, used at once and never leaves the CTA.  The FP64 part keeps the SM's two
// FP64 lanes busy and the R part of other CTAs runs beside it.
// even: the table is even in both offsets, so its row spectra are real and even in y: Zs
// holds the rows 0 .. Ny/2, and two columns share one complex transform.

struct RecShape {
    int C, lines;  // columns per CTA; FP64 lines (C, or C / 2 when even)
    unsigned mC, mlines;
    int even;
    int buf;  // bytes of a transform buffer: N lines FP64 or N C values of R
};

template <typename R>
__device__ __forceinline__ void layer_spectrum(int N, int ncol, const RecShape &rs, const FftPlanDev &py, int c0, int cols,
                                               const double2 *Zs, double2 *bufA, double2 *bufB, const double2 *tw64,
                                               cpx<R> *S) {
    const int C = rs.C;
    const double2 *Z = Zs + c0;
    auto in = [&](int j, int l) {
        if (rs.even) {
            const double2 *row = Z + (size_t)(2 * j > N ? N - j : j) * ncol;
            return make_double2(__ldg(&row[min(2 * l, cols - 1)].x), __ldg(&row[min(2 * l + 1, cols - 1)].x));
        }
        return __ldg(Z + (size_t)j * ncol + min(l, cols - 1));
    };
    auto out = [&](int k, int l, double2 x) {
        if (rs.even) {
            S[k * C + 2 * l] = mk<cpx<R>>((R)x.x, R(0));
            S[k * C + 2 * l + 1] = mk<cpx<R>>((R)x.y, R(0));
        } else {
            S[k * C + l] = mk<cpx<R>>((R)x.x, (R)x.y);
        }
    };
    fft_run<double, false, false, false>(py, rs.lines, rs.mlines, rs.lines, bufA, bufB, tw64, N, N, in, out);
    __syncthreads();
}

// Y (+)= T^_r . FFT_y(Z_r); the first layer writes Y.
template <typename R>
struct IntoY {
    cpx<R> *Y;  // column c0
    const cpx<R> *S;
    int ncol, C, cols, first;
    __device__ __forceinline__ cpx<R> pre(int n, int c) const { return Y[(size_t)n * ncol + min(c, cols - 1)]; }
    __device__ __forceinline__ void operator()(int n, int c, cpx<R> x, cpx<R> y) const {
        const cpx<R> p = cmul(x, S[n * C + c]);
        if (c < cols) Y[(size_t)n * ncol + c] = first ? p : cadd(y, p);
    }
};

template <typename R>
__global__ void __launch_bounds__(256) k_col_rec_fwd(OpView<R> op, RecShape rs, const double2 *Zs,
                                                     const double2 *twy64, int r) {
    using Cx = cpx<R>;
    const int N = op.Ny, C = rs.C, c0 = blockIdx.x * C, cols = min(C, op.ncol - c0);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *bufA = smem_raw, *bufB = bufA + rs.buf;
    double2 *tw64 = reinterpret_cast<double2 *>(bufB + rs.buf);
    Cx *S = reinterpret_cast<Cx *>(tw64 + N), *tw = S + N * C;
    load_twiddles(tw64, twy64, N);
    load_twiddles(tw, op.twy, N);
    pdl_wait();
    pdl_go();  // only now: the next layer's table rows may rely on everything before this kernel
    layer_spectrum<R>(N, op.ncol, rs, op.py, c0, cols, Zs, reinterpret_cast<double2 *>(bufA), reinterpret_cast<double2 *>(bufB), tw64,
                      S);
    const FromZ<R> in{op, op.Z + c0, LineMap{rs.mC, C, cols, r, r + 1}};
    const IntoY<R> out{op.Y + c0, S, op.ncol, C, cols, r == 0};
    fft_run<R, false, true, false>(op.py, C, rs.mC, C, reinterpret_cast<Cx *>(bufA), reinterpret_cast<Cx *>(bufB), tw,
                                   op.ny, N, in, out);
}

// Z_r = IFFT_y(conj(T^_r) . Y), rows iy < ny (Y = FFT_y of the residual rows).
template <typename R>
__global__ void __launch_bounds__(256) k_col_rec_adj(OpView<R> op, RecShape rs, const double2 *Zs,
                                                     const double2 *twy64, int r) {
    using Cx = cpx<R>;
    const int N = op.Ny, C = rs.C, c0 = blockIdx.x * C, cols = min(C, op.ncol - c0), ncol = op.ncol, ny = op.ny;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *bufA = smem_raw, *bufB = bufA + rs.buf;
    double2 *tw64 = reinterpret_cast<double2 *>(bufB + rs.buf);
    Cx *S = reinterpret_cast<Cx *>(tw64 + N), *tw = S + N * C;
    load_twiddles(tw64, twy64, N);
    load_twiddles(tw, op.twy, N);
    pdl_wait();
    pdl_go();  // only now: the next layer's table rows may rely on everything before this kernel
    layer_spectrum<R>(N, op.ncol, rs, op.py, c0, cols, Zs, reinterpret_cast<double2 *>(bufA), reinterpret_cast<double2 *>(bufB), tw64,
                      S);
    const Cx *Y = op.Y + c0;
    Cx *Z = op.Z + (size_t)r * ny * ncol + c0;
    auto in = [&](int k, int c) { return cmulc(Y[(size_t)k * ncol + min(c, cols - 1)], S[k * C + c]); };
    auto out = [&](int n, int c, Cx x) {
        if (n < ny && c < cols) Z[(size_t)n * ncol + c] = x;
    };
    fft_run<R, true, false, true>(op.py, C, rs.mC, C, reinterpret_cast<Cx *>(bufA), reinterpret_cast<Cx *>(bufB), tw,
                                  N, ny, in, out);
}

// One column transform of the whole plane: Y = FFT_y(W) (W has sy rows) or, INV,
// W = IFFT_y(Y) cropped to sy rows.
template <typename R, bool INV>
__global__ void __launch_bounds__(256) k_col_plane(OpView<R> op, ColShape cs) {
    using Cx = cpx<R>;
    const int N = op.Ny, C = cs.C, c0 = blockIdx.x * C, cols = min(C, op.ncol - c0), ncol = op.ncol, sy = op.sy;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx *bufA = reinterpret_cast<Cx *>(smem_raw), *bufB = bufA + N * cs.pitch1, *tw = bufB + N * cs.pitch1;
    load_twiddles(tw, op.twy, N);
    pdl_wait();
    const Cx *src = (INV ? op.Y : op.W) + c0;
    Cx *dst = (INV ? op.W : op.Y) + c0;
    const int rows_in = INV ? N : sy, rows_out = INV ? sy : N;
    auto in = [&](int j, int c) {
        const Cx w = src[(size_t)min(j, rows_in - 1) * ncol + min(c, cols - 1)];
        return j < rows_in ? w : czero<Cx>();
    };
    auto out = [&](int n, int c, Cx x) {
        if (n < rows_out && c < cols) dst[(size_t)n * ncol + c] = x;
    };
    fft_run<R, INV, !INV, INV>(op.py, C, cs.mC, cs.pitch1, bufA, bufB, tw, rows_in, rows_out, in, out);
}

}  // namespace gj
