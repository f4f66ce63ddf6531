// Column passes for a 1024-row BCCB embedding (N_y = 1024, FP32, at most 512 prisms
// and 512 stations per column; the rows run on the general kernels for any N_x, which
// write and read the transposed intermediates these kernels stream).
//
// Warp FFT.  1024 = 32 x 32, one warp: lane l holds x[l + 32 j] (j < 16; the upper half of
// the inputs is zero), takes a 32-point DFT over j in registers (pruned: two 16-point DFTs,
// of x and of x W32^j, give the even and the odd outputs), multiplies by W1024^(l a),
// transposes through a swizzled 32 x 32 shared-memory tile and takes a full 32-point DFT
// over l (two 16-point DFTs and a radix-2 step).  Lane l then holds X[l + 32 b] in register
// b.  The inverse runs the steps backwards, its last DFT formed for the outputs n < 512 only.
// One table of W1024^(l a) (8 KB) serves both directions.  Two half-warps with a 512-point
// transform of one output parity each, the split of the 512 kernels, cost 17 more complex
// products, a second read of every input, and 64 shuffles and as many selects in the
// inverse, which joined the halves; its tables took 20 KB.
//
// Layouts (per field): spectra St[r][kx][ky < 1024] (the even real gravity spectrum
// as [r][kx][ky <= 512], 516 values per column), row-pass output Zt[r][kx][iy < 512],
// inverse-column output Wt[kx][jy < 512] and residual-row spectra Vt[kx][jy < 512].
#pragma once
#include "fast512.cuh"

namespace gj {
namespace f1024 {

using f512::ColItem;
using f512::View2;

constexpr int N = 1024, H = 512;
constexpr int CWF = 8;  // warps per CTA of the forward column kernel (24 KB of shared memory each)
constexpr int CWA = 8;  // warps per CTA of the adjoint column kernel (24 KB each)
constexpr int ST = f512::CSTAGES;  // TMA ring depth per warp
constexpr int kFwdWarpWords = 2 * H + N + N;  // forward column kernel, per warp: Z stages, spectrum, transpose tile
constexpr int KE = even_spec_len(N), KEB = KE * (int)sizeof(float);

// 32-point DFT in place, natural order in and out: the even- and odd-indexed halves
// by 16-point DFTs, then X[a] = E[a] + W32^a O[a], X[a + 16] = E[a] - W32^a O[a].
template <typename R, bool INV>
__device__ __forceinline__ void dft32(cpx<R> (&x)[32]) {
    using C = cpx<R>;
    C e[16], o[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) { e[i] = x[2 * i]; o[i] = x[2 * i + 1]; }
    f512::dft16<R, INV>(e);
    f512::dft16<R, INV>(o);
#pragma unroll
    for (int a = 0; a < 16; ++a) {
        const C w = f512::w32c<R>(a);
        const C t = a == 0 ? o[a] : (INV ? cmulc(o[a], w) : cmul(o[a], w));
        x[a] = cadd(e[a], t);
        x[a + 16] = mk<C>(e[a].x - t.x, e[a].y - t.y);
    }
}

// W1024^(l a), rows a of 32 lanes l, read from shared memory; the inverse conjugates.  The
// entries are the operator's W1024 table itself, so they carry no product rounding.
template <typename R>
struct Tab1024 {
    static constexpr int WORDS = 32 * 32;
    __device__ static void build(cpx<R> *t, const cpx<R> *__restrict__ tw1024) {
        for (int i = threadIdx.x; i < WORDS; i += blockDim.x) t[i] = __ldg(tw1024 + (i >> 5) * (i & 31));
    }
};

// swizzled 32 x 32 tile of one warp: entry (row, col) at row * 32 + (col ^ row)
__device__ __forceinline__ int swz32(int row, int col) { return row * 32 + (col ^ row); }

// Forward pruned 1024-point transform.  In: v[j] = x[lane + 32 j], j < 16 (the upper
// registers are not read).  Out: v[b] = X[lane + 32 b].
// buf: this warp's 1024-entry tile; tab: the CTA's Tab1024 (shared).
template <typename R>
__device__ __forceinline__ void fwd1024(cpx<R> (&v)[32], cpx<R> *buf, const cpx<R> *tab) {
    using C = cpx<R>;
    const int lane = threadIdx.x & 31;
    {
        C e[16], o[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            e[j] = v[j];
            o[j] = j == 0 ? v[0] : cmul(v[j], f512::w32c<R>(j));
        }
        f512::dft16<R, false>(e);  // over j -> index a = 2 i
        f512::dft16<R, false>(o);  // a = 2 i + 1
#pragma unroll
        for (int i = 0; i < 16; ++i) { v[2 * i] = e[i]; v[2 * i + 1] = o[i]; }
    }
#pragma unroll
    for (int a = 1; a < 32; ++a) v[a] = cmul(v[a], tab[a * 32 + lane]);
    __syncwarp();
#pragma unroll
    for (int a = 0; a < 32; ++a) buf[swz32(lane, a)] = v[a];
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 32; ++r) v[r] = buf[swz32(r, lane)];
    dft32<R, false>(v);  // over l -> index b, for a = this lane
}

// Inverse (unnormalised).  In: v[b] = Y[lane + 32 b].  Out: out[j] = y[lane + 32 j], j < 16.
template <typename R>
__device__ __forceinline__ void inv1024(cpx<R> (&v)[32], cpx<R> *buf, const cpx<R> *tab, cpx<R> (&out)[16]) {
    using C = cpx<R>;
    const int lane = threadIdx.x & 31;
    dft32<R, true>(v);  // over b -> index l, for a = this lane
#pragma unroll
    for (int l = 1; l < 32; ++l) v[l] = cmulc(v[l], tab[l * 32 + lane]);  // W1024^-(l a)
    __syncwarp();
#pragma unroll
    for (int l = 0; l < 32; ++l) buf[swz32(lane, l)] = v[l];
    __syncwarp();
    C e[16], o[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        e[i] = buf[swz32(2 * i, lane)];
        o[i] = buf[swz32(2 * i + 1, lane)];
    }
    f512::dft16<R, true>(e);  // over a -> index j < 16: y[j] = E[j] + W32^-j O[j]
    f512::dft16<R, true>(o);
#pragma unroll
    for (int j = 0; j < 16; ++j) out[j] = cadd(e[j], j == 0 ? o[0] : cmulc(o[j], f512::w32c<R>(j)));
}

// Position of spectrum index ky = lane + 32 b in an even real spectrum stored for
// ky <= 512: min(ky, 1024 - ky), which b, a compile-time index, decides.
__device__ __forceinline__ int even_pos1024(int lane, int b) { return b < 16 ? lane + 32 * b : N - 32 * b - lane; }

// Every CTA copies the operator's Tab1024 into shared memory with one bulk copy.
template <typename R>
__device__ __forceinline__ void load_tab(cpx<R> *tab, const cpx<R> *src, uint64_t *bar) {
    if (threadIdx.x == 0) {
        f512::mbar_expect(bar, Tab1024<R>::WORDS * sizeof(cpx<R>));
        f512::bulk_load(tab, src, Tab1024<R>::WORDS * sizeof(cpx<R>), bar);
    }
}

template <typename R>
__global__ void k_build_tab1024(cpx<R> *tab, const cpx<R> *tw1024) {
    Tab1024<R>::build(tab, tw1024);
}

// Forward column pass: for each (field, kx), Y = sum_r St_r[kx] . FFT1024(Zt_r[kx]),
// then Wt[kx][jy] = IFFT1024(Y)[jy] for jy < sy.  Persistent warps take balanced
// contiguous segments of the (kx, field, r) sequence; a column split across warps is
// summed in segment order by the last warp to finish it (as in the 512 kernels).
//
// Issue slots and instruction latency bound it, so it wants as many warps as the register file
// holds (8, two per scheduler).  Each has two stages for Z but one for the spectrum, which
// is fetched as soon as the last multiply has read it and is wanted one transform later;
// with two of both, a warp took 32 KB, six fitted, and two of the four schedulers had one.
// 512 x 512 x 48, one field: 66 / 69 us (even / complex spectra) with six warps and half-warp
// transforms, 51 / 62 now (153 / 305 MB from HBM).
template <typename R>
__global__ void __launch_bounds__(CWF * 32, 1) k_col_fwd1024(View2<R> V, const int *done) {
    using C = cpx<R>;
    if (stopped(done) || f512::op_failed(V.err)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int ZB = H * sizeof(C), TB = N * sizeof(C);
    constexpr size_t WB = kFwdWarpWords * sizeof(C);  // bytes per warp
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    C *zs = reinterpret_cast<C *>(smem_raw + (size_t)warp * WB);  // 2 x 512
    C *ts = zs + 2 * H;                                           // 1024
    C *xbuf = ts + N;                                             // 1024
    C *tab = reinterpret_cast<C *>(smem_raw + (size_t)CWF * WB);
    __shared__ __align__(8) uint64_t zbar[CWF][2], tbar[CWF];
    __shared__ __align__(8) uint64_t tabbar;
    if (lane == 0) {
        f512::mbar_init(&zbar[warp][0]);
        f512::mbar_init(&zbar[warp][1]);
        f512::mbar_init(&tbar[warp]);
    }
    if (threadIdx.x == 0) f512::mbar_init(&tabbar);
    f512::mbar_fence_init();
    __syncthreads();
    const int nz = V.op[0].nz, sy = V.op[0].sy, NC = V.op[0].ncol;
    const long long T = (long long)V.nfield * NC * nz;
    const long long Wt = f512::seg_warps((long long)gridDim.x * CWF, T);
    const long long w = (long long)blockIdx.x * CWF + warp;
    if ((long long)blockIdx.x * CWF < Wt) load_tab<R>(tab, V.twtab, &tabbar);
    if (w >= Wt) return;
    const int t0 = (int)f512::seg_begin(w, T, Wt), t1 = (int)f512::seg_begin(w + 1, T, Wt);
    ColItem cu, cz, ct;  // the item being consumed; (lane 0) the next ones whose columns are fetched
    cu.set(t0, nz, V.nfield);
    cz = ct = cu;
    int tz = t0, tt = t0;
    auto issue_z = [&]() {
        const int s = (tz - t0) & 1;
        f512::mbar_expect(&zbar[warp][s], ZB);
        f512::bulk_load(zs + s * H, V.op[cz.fld].Z + ((size_t)cz.r * NC + cz.kx) * H, ZB, &zbar[warp][s]);
        ++tz;
        cz.next(nz, V.nfield);
    };
    auto issue_t = [&]() {
        const OpView<R> &op = V.op[ct.fld];
        const size_t off = (size_t)ct.r * NC + ct.kx;
        f512::mbar_expect(&tbar[warp], op.real_spec ? KEB : TB);
        if (op.real_spec)
            f512::bulk_load(ts, reinterpret_cast<const R *>(op.spec) + off * KE, KEB, &tbar[warp]);
        else
            f512::bulk_load(ts, op.spec + off * N, TB, &tbar[warp]);
        ++tt;
        ct.next(nz, V.nfield);
    };
    if (lane == 0) {
        issue_z();
        issue_t();
        if (tz < t1) issue_z();
    }
    C acc[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) acc[k] = czero<C>();
    bool ok = __all_sync(0xffffffffu, f512::mbar_wait(&tabbar, 0, V.err));
    int seg_start = t0;
    for (int t = t0; t < t1 && ok; ++t, cu.next(nz, V.nfield)) {
        const int s = (t - t0) & 1;
        ok = __all_sync(0xffffffffu, f512::mbar_wait(&zbar[warp][s], (uint32_t)((t - t0) >> 1) & 1, V.err));
        if (!ok) break;
        C v[32];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = zs[s * H + lane + 32 * j];
        __syncwarp();
        if (lane == 0 && tz < t1) issue_z();  // item t + 2, into the stage just read
        fwd1024<R>(v, xbuf, tab);
        ok = __all_sync(0xffffffffu, f512::mbar_wait(&tbar[warp], (uint32_t)(t - t0) & 1, V.err));
        if (!ok) break;
        if (V.op[cu.fld].real_spec) {
            const R *tr = reinterpret_cast<const R *>(ts);
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const R q = tr[even_pos1024(lane, i)];
                acc[i] = mk<C>(acc[i].x + v[i].x * q, acc[i].y + v[i].y * q);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const C q = ts[lane + 32 * i];
                acc[i].x = fma(v[i].x, q.x, acc[i].x);
                acc[i].x = fma(-v[i].y, q.y, acc[i].x);
                acc[i].y = fma(v[i].x, q.y, acc[i].y);
                acc[i].y = fma(v[i].y, q.x, acc[i].y);
            }
        }
        __syncwarp();
        if (lane == 0 && tt < t1) issue_t();
        if (cu.r == nz - 1 || t == t1 - 1) {
            const int fld = cu.fld, kx = cu.kx;
            const long long col = cu.col;
            const OpView<R> &op = V.op[fld];
            const long long cb = col * nz, ce = cb + nz - 1;
            const bool whole = (seg_start <= cb) && (t == ce);
            if (!whole) {
                const long long wf = f512::seg_owner(cb, T, Wt), wl = f512::seg_owner(ce, T, Wt);
                const int slot = (int)(w - wf), nslots = (int)(wl - wf + 1);
                C *Pc = V.P[fld] + (size_t)kx * V.slots * N;
#pragma unroll
                for (int i = 0; i < 32; ++i) Pc[(size_t)slot * N + lane + 32 * i] = acc[i];
                __threadfence();
                __syncwarp();
                int old = 0;
                if (lane == 0) old = atomicAdd(V.cnt[fld] + kx, 1);
                old = __shfl_sync(0xffffffffu, old, 0);
                if (old == nslots - 1) {
                    __threadfence();
#pragma unroll
                    for (int i = 0; i < 32; ++i) acc[i] = czero<C>();
                    for (int sl = 0; sl < nslots; ++sl) {
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            acc[i] = cadd(acc[i], __ldcg(Pc + (size_t)sl * N + lane + 32 * i));
                    }
                    if (lane == 0) V.cnt[fld][kx] = 0;
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) acc[i] = czero<C>();
                    seg_start = t + 1;
                    continue;
                }
            }
            C out[16];
            inv1024<R>(acc, xbuf, tab, out);
            C *Wc = op.W + (size_t)kx * H;
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) {
                const int n = lane + 32 * jj;
                if (n < sy) Wc[n] = out[jj];
            }
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = czero<C>();
            seg_start = t + 1;
        }
    }
    if (!ok) {  // no copy may land after the CTA exits: wait (bounded) for the newest of each stage
        const int ez = __shfl_sync(0xffffffffu, tz, 0), et = __shfl_sync(0xffffffffu, tt, 0);
        for (int t = max(t0, ez - 2); t < ez; ++t)
            f512::mbar_wait(&zbar[warp][(t - t0) & 1], (uint32_t)((t - t0) >> 1) & 1, V.err);
        f512::mbar_wait(&tbar[warp], (uint32_t)(et - 1 - t0) & 1, V.err);
    }
}

// Adjoint column pass: for each (field, kx, r),
// Zt_r[kx][iy] = IFFT1024(conj(St_r[kx]) . FFT1024(Vt[kx]))[iy], iy < ny.  Bound like the
// forward pass; 50 / 57 us (even / complex spectra) at 512 x 512 x 48 with half-warp
// transforms, 41 / 48 with the 32 x 32 ones.
template <typename R>
__global__ void __launch_bounds__(CWA * 32, 1) k_col_adj1024(View2<R> V, const int *done) {
    using C = cpx<R>;
    if (stopped(done) || f512::op_failed(V.err)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int TB = N * sizeof(C);
    constexpr size_t WB = (size_t)ST * TB + N * sizeof(C);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *wbase = smem_raw + (size_t)warp * WB;
    C *ts = reinterpret_cast<C *>(wbase);
    C *xbuf = reinterpret_cast<C *>(wbase + ST * TB);
    C *tab = reinterpret_cast<C *>(smem_raw + (size_t)CWA * WB);
    __shared__ __align__(8) uint64_t bars[CWA][ST];
    __shared__ __align__(8) uint64_t tabbar;
    if (lane == 0)
        for (int s = 0; s < ST; ++s) f512::mbar_init(&bars[warp][s]);
    if (threadIdx.x == 0) f512::mbar_init(&tabbar);
    f512::mbar_fence_init();
    __syncthreads();
    const int nz = V.op[0].nz, ny = V.op[0].ny, NC = V.op[0].ncol;
    const long long T = (long long)V.nfield * NC * nz;
    const long long Wt = f512::seg_warps((long long)gridDim.x * CWA, T);
    const long long w = (long long)blockIdx.x * CWA + warp;
    if ((long long)blockIdx.x * CWA < Wt) load_tab<R>(tab, V.twtab, &tabbar);
    if (w >= Wt) return;
    const int t0 = (int)f512::seg_begin(w, T, Wt), t1 = (int)f512::seg_begin(w + 1, T, Wt);
    ColItem cu, ci;
    cu.set(t0, nz, V.nfield);
    ci = cu;
    int ti = t0;
    auto issue = [&]() {
        const int s = (ti - t0) % ST;
        const OpView<R> &op = V.op[ci.fld];
        const size_t off = (size_t)ci.r * NC + ci.kx;
        if (op.real_spec) {
            f512::mbar_expect(&bars[warp][s], KEB);
            f512::bulk_load(ts + s * N, reinterpret_cast<const R *>(op.spec) + off * KE, KEB, &bars[warp][s]);
        } else {
            f512::mbar_expect(&bars[warp][s], TB);
            f512::bulk_load(ts + s * N, op.spec + off * N, TB, &bars[warp][s]);
        }
        ++ti;
        ci.next(nz, V.nfield);
    };
    if (lane == 0)
        while (ti < t1 && ti < t0 + ST) issue();
    C vh[32];
    bool ok = __all_sync(0xffffffffu, f512::mbar_wait(&tabbar, 0, V.err));
    int t_fail = ok ? t1 : t0;
    for (int t = t0; t < t1 && ok; ++t, cu.next(nz, V.nfield)) {
        const int r = cu.r, fld = cu.fld, kx = cu.kx;
        const OpView<R> &op = V.op[fld];
        if (t == t0 || r == 0) {  // a new column: V^ = FFT1024 of the residual column (rows >= sy are zero)
            const C *Vc = op.V + (size_t)kx * H;
#pragma unroll
            for (int j = 0; j < 16; ++j) vh[j] = Vc[lane + 32 * j];
            fwd1024<R>(vh, xbuf, tab);
        }
        const int s = (t - t0) % ST;
        const uint32_t par = (uint32_t)(((t - t0) / ST) & 1);
        ok = __all_sync(0xffffffffu, f512::mbar_wait(&bars[warp][s], par, V.err));
        if (!ok) { t_fail = t; break; }
        C v[32];
        if (op.real_spec) {
            const R *tr = reinterpret_cast<const R *>(ts + s * N);
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const R tt = tr[even_pos1024(lane, i)];
                v[i] = mk<C>(vh[i].x * tt, vh[i].y * tt);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = cmulc(vh[i], ts[s * N + lane + 32 * i]);
        }
        __syncwarp();
        if (lane == 0 && ti < t1) issue();
        C out[16];
        inv1024<R>(v, xbuf, tab, out);
        C *Zc = op.Z + ((size_t)r * NC + kx) * H;
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) {
            const int n = lane + 32 * jj;
            if (n < ny) Zc[n] = out[jj];
        }
    }
    if (!ok) f512::drain(bars[warp], t_fail, t0, t1, V.err);
}

// ---------------------------------------------------------------------------
// Row passes for N_x = 1024 and lines of at most 512 values (with the N_y = 1024 column
// kernels): real lines <-> half spectra in the transposed layout, through the general
// kernels' per-element functors.  A CTA of RW warps runs one complex transform per warp: two lines of one
// field (pair map, joint = 0) or one line of each field (joint = 1).  The half
// spectra of the CTA's lines meet in a shared tile [k < 513][slot], a transform's two
// lines side by side (one 16-byte word), and move to or from the transposed layout with
// consecutive lines in consecutive words: two lines per 16-byte access where the pairs of
// one field lie side by side there too (an even number of lines per layer), else one.
// Each thread keeps its slots, so its lines' address is formed once.  The warps' transform
// buffers share the tile's memory (barriers separate the two uses).
//
// Waiting bounds both passes: for the lines, for the barriers around the tile.  So CTAs are
// small, four warps (eight lines, 64-byte runs in the transposed layout) and four CTAs per SM
// (128 registers), each at its own point of the read-transform-write sequence: 42.6 us
// forward and 34.2 inverse for the 24 576 cell lines of 512 x 512 x 48 (3.5 and 3.6 TB/s),
// 47.9 and 39.1 with two CTAs of eight warps, 44.4 and 38.5 with three of six (96
// registers); 53.7 and 53.9 with one line per 8-byte access, a [slot][k] tile and the
// half-warp transforms.

constexpr int RW = 4;                 // warps (transforms) per CTA
constexpr int RCTA = 4;               // CTAs per SM
constexpr int RSLOT = 2 * RW;         // tile slots: two lines per transform
constexpr int NCR = N / 2 + 1;        // 513 bins
constexpr int TP = RSLOT + 2;         // words per tile row: rows stay 16-byte aligned, and the 16-byte
                                      // accesses of eight consecutive rows fall in distinct banks
static_assert((RW * 32) % RSLOT == 0, "a thread keeps one tile slot");

// tile slot s of the CTA -> its line and field, and whether it exists
__device__ __forceinline__ bool slot_line(const PairMap &pm, int base, int s, int &line, int &field) {
    const int np = pm.npairs();
    const int q = base + (s >> 1);
    if (pm.joint) {
        field = s & 1;
        line = q;
        return q < np;
    }
    field = 0;
    line = 2 * q + (s & 1);
    return q < np && line < pm.nlines;
}

// While its own copies are in flight, a CTA of the inverse asks for the half spectra of the
// CTA that follows it on the SM, one wave of CTAs ahead, so that those find them in L2 (36.0 ->
// 34.2 us at 512 x 512 x 48; the forward's lines, a long run each, gained nothing from it).
constexpr int RAHEAD = RCTA * 152;
__device__ __forceinline__ void l2_prefetch(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// two adjacent words, one 16-byte access (p on 16 bytes) in FP32
template <typename C>
__device__ __forceinline__ void put2(C *p, C a, C b) {
    if constexpr (sizeof(C) == 8) *reinterpret_cast<float4 *>(p) = make_float4(a.x, a.y, b.x, b.y);
    else { p[0] = a; p[1] = b; }
}
template <typename C>
__device__ __forceinline__ void get2(const C *p, C &a, C &b) {
    if constexpr (sizeof(C) == 8) {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        a = mk<C>(q.x, q.y);
        b = mk<C>(q.z, q.w);
    } else { a = p[0]; b = p[1]; }
}

// The operator's twiddle table into shared memory with 16-byte asynchronous copies,
// all in flight at once (committed as one group; the caller waits and synchronises).
template <typename R>
__device__ __forceinline__ void load_tab_async(cpx<R> *tab, const cpx<R> *src) {
    constexpr int CH = Tab1024<R>::WORDS * (int)sizeof(cpx<R>) / 16;
    const char *s = reinterpret_cast<const char *>(src);
    char *d = reinterpret_cast<char *>(tab);
    for (int i = threadIdx.x; i < CH; i += blockDim.x) f512::cp_async16(d + 16 * i, s + 16 * i);
    f512::cp_async_commit();
}

// words of the tile / transform-buffer overlay
constexpr int row_overlay_words() { return NCR * TP > RW * N ? NCR * TP : RW * N; }

// Whether slots 2 i and 2 i + 1 hold lines side by side in 16-byte words of the transposed
// layout: pairs of one field that do not straddle layers, and an even column stride.
__device__ __forceinline__ bool pairs_aligned(const PairMap &pm, int tcol) {
    return !pm.joint && tcol && (tcol & 1) == 0 && (pm.lpl & 1) == 0 && (pm.nlines & 1) == 0;
}

template <typename R, class Pro>
__global__ void __launch_bounds__(RW * 32, RCTA) k_row_fwd1024(OpView<R> op, PairMap pm, int n_in, cpx<R> *out0,
                                                            cpx<R> *out1, const cpx<R> *tab_src, Pro pro,
                                                            const int *done) {
    using C = cpx<R>;
    if (stopped(done)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *tab = reinterpret_cast<C *>(smem_raw);
    C *tile = tab + Tab1024<R>::WORDS;  // [RSLOT][TP], or the warps' buffers before it is filled
    __shared__ double red[128];
    pro.init();
    load_tab_async<R>(tab, tab_src);  // in flight while the lines are read
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int base = blockIdx.x * RW, q = base + warp;
    const bool act = q < pm.npairs();
    C v[32];
    if (act) {
        int la, lb;
        bool hb;
        pm.lines(q, la, lb, hb);
        // every element through the functor once, in the lane layout of the transform
        R a[16], b[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int e = lane + 32 * i;
            a[i] = b[i] = R(0);
            if (e < n_in) field_functor(pro, blockIdx.y).fetch(la, lb, hb, e, a[i], b[i]);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = mk<C>(a[i], b[i]);
    }
    f512::cp_async_wait<0>();
    __syncthreads();  // the table is in
    if (act) fwd1024<R>(v, tile + warp * N, tab);
    __syncthreads();  // the buffers become the tile
    if (act) {
        // Z = FFT(a + i b) -> A = (Z[k] + conj Z[N - k]) / 2, B = (Z[k] - conj Z[N - k]) / 2i,
        // k = lane + 32 m <= 512.  For lane != 0, Z[N - k] sits in lane 32 - lane at register
        // 31 - m; lane 0 holds it at 32 - m.
        const int partner = (32 - lane) & 31;
        C *row = tile + 2 * warp;
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            C zm;
            zm.x = __shfl_sync(0xffffffffu, v[31 - m].x, partner);
            zm.y = __shfl_sync(0xffffffffu, v[31 - m].y, partner);
            if (lane == 0) zm = v[(32 - m) & 31];
            const C zk = v[m];
            put2(row + (lane + 32 * m) * TP, mk<C>(R(0.5) * (zk.x + zm.x), R(0.5) * (zk.y - zm.y)),
                 mk<C>(R(0.5) * (zk.y + zm.y), R(-0.5) * (zk.x - zm.x)));
        }
        if (lane == 0)  // k = 512 is its own partner
            put2(row + H * TP, mk<C>(v[16].x, R(0)), mk<C>(v[16].y, R(0)));
    }
    __syncthreads();
    if (pairs_aligned(pm, op.tcol)) {
        const int i = threadIdx.x % RW, line = 2 * (base + i);
        if (line < pm.nlines) {
            C *o = (blockIdx.y ? out1 : out0) + pm.at(line, 0, op.ncol, op.tcol);
#pragma unroll 4
            for (int k = threadIdx.x / RW; k < NCR; k += 32) {
                C a, b;
                get2(tile + k * TP + 2 * i, a, b);
                put2(o + (size_t)k * op.tcol, a, b);
            }
        }
    } else {
        const int s = threadIdx.x % RSLOT;
        int line, field;
        if (slot_line(pm, base, s, line, field)) {
            if (!pm.joint) field = blockIdx.y;  // pairs of one field: the launch's grid y
            C *o = (field ? out1 : out0) + pm.at(line, 0, op.ncol, op.tcol);
            const size_t step = op.tcol ? (size_t)op.tcol : 1;
            for (int k = threadIdx.x / RSLOT; k < NCR; k += blockDim.x / RSLOT) o[k * step] = tile[k * TP + s];
        }
    }
    pro.flush(red);
}

template <typename R, class Epi>
__global__ void __launch_bounds__(RW * 32, RCTA) k_row_inv1024(OpView<R> op, PairMap pm, int n_out, const cpx<R> *in0,
                                                            const cpx<R> *in1, const cpx<R> *tab_src, Epi epi,
                                                            const int *done) {
    using C = cpx<R>;
    if (stopped(done)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *tab = reinterpret_cast<C *>(smem_raw);
    C *tile = tab + Tab1024<R>::WORDS;  // [RSLOT][TP], then the warps' buffers
    __shared__ double red[128];
    epi.init();
    load_tab_async<R>(tab, tab_src);
    const int base = blockIdx.x * RW;
    // every copy of the CTA's half spectra in flight at once (asynchronous copies)
    if (sizeof(C) == 8 && pairs_aligned(pm, op.tcol)) {
        const int i = threadIdx.x % RW, line = 2 * (base + i);
        if (line < pm.nlines) {
            const C *src = (blockIdx.y ? in1 : in0) + pm.at(line, 0, op.ncol, op.tcol);
            for (int k = threadIdx.x / RW; k < NCR; k += 32) f512::cp_async16(tile + k * TP + 2 * i, src + (size_t)k * op.tcol);
        }
    } else {
        const int s = threadIdx.x % RSLOT;
        int line, field;
        const bool ok = slot_line(pm, base, s, line, field);
        if (!pm.joint) field = blockIdx.y;  // pairs of one field: the launch's grid y
        const C *src = ok ? (field ? in1 : in0) + pm.at(line, 0, op.ncol, op.tcol) : nullptr;
        const size_t step = op.tcol ? (size_t)op.tcol : 1;
        for (int k = threadIdx.x / RSLOT; k < NCR; k += blockDim.x / RSLOT) {
            C *dst = tile + k * TP + s;
            if (!ok) *dst = czero<C>();
            else if constexpr (sizeof(C) == 8) f512::cp_async8(dst, src + k * step);
            else f512::cp_async16(dst, src + k * step);
        }
    }
    f512::cp_async_commit();
    if (const int line = 2 * (base + RAHEAD * RW); pairs_aligned(pm, op.tcol) && line < pm.nlines) {
        const C *src = (blockIdx.y ? in1 : in0) + pm.at(line, 0, op.ncol, op.tcol);
        for (int k = threadIdx.x; k < NCR; k += RW * 32) l2_prefetch(src + (size_t)k * op.tcol);
    }
    f512::cp_async_wait<0>();
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = base + warp;
    const bool act = q < pm.npairs();
    int la = 0, lb = 0;
    bool hb = false;
    C v[32];
    if (act) {
        pm.lines(q, la, lb, hb);
        // Hermitian-extended A + i B in the lane layout, k = lane + 32 m (an absent second
        // line reads as zero)
        const C *row = tile + 2 * warp;
#pragma unroll
        for (int m = 0; m < 32; ++m) {
            C A, B;
            get2(row + (m < 16 ? lane + 32 * m : N - 32 * m - lane) * TP, A, B);
            if ((m == 0 || m == 16) && lane == 0) { A.y = 0; B.y = 0; }  // k = 0, 512
            v[m] = m < 16 ? mk<C>(A.x - B.y, A.y + B.x) : mk<C>(A.x + B.y, B.x - A.y);
        }
    }
    __syncthreads();  // the tile becomes the warps' buffers
    if (act) {
        C out[16];
        inv1024<R>(v, tile + warp * N, tab, out);
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) {
            const int n = lane + 32 * jj;
            if (n < n_out) field_functor(epi, blockIdx.y).store(la, lb, hb, n, out[jj].x, out[jj].y);
        }
    }
    field_functor(epi, blockIdx.y).flush(red);
}

template <typename R> inline size_t smem_row() {
    return ((size_t)Tab1024<R>::WORDS + (size_t)row_overlay_words()) * sizeof(cpx<R>);
}

template <typename R> inline size_t smem_col_fwd() {
    return ((size_t)CWF * kFwdWarpWords + Tab1024<R>::WORDS) * sizeof(cpx<R>);
}
template <typename R> inline size_t smem_col_adj() {
    return (size_t)CWA * ((size_t)ST * N + N) * sizeof(cpx<R>) + Tab1024<R>::WORDS * sizeof(cpx<R>);
}

}  // namespace f1024
}  // namespace gj
