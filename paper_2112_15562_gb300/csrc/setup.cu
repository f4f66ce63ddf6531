// Operator setup (Sec. 2.7.1): prism kernel tables of every depth layer, their
// BCCB embedding and 2-D spectra.  All geometry arithmetic runs in FP64.
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

#include "fast1024.cuh"
#include "fast512.cuh"
#include "general_launch.cuh"

namespace gj {

// ---------------------------------------------------------------------------
// Closed-form prism fields as corner sums of antiderivatives (Sec. 2.1 cites
// Haaz for the vertical gravity and Rao & Babu for the total-field anomaly).
// u = x' - x0, v = y' - y0, w = z' - z0 (z down) with w >= 0 at every corner;
// u and v are never zero because corners sit half a cell from the stations.

// ln(a + R) for R = sqrt(a^2 + b^2 + c^2); for a < 0 use (b^2 + c^2) / (R - a).
__device__ __forceinline__ double log_a_plus_r(double a, double R, double b, double c) {
    return a >= 0.0 ? log(a + R) : log((b * b + c * c) / (R - a));
}

// Antiderivative whose mixed third derivative is w / R^3.
__device__ __forceinline__ double gravity_corner(double u, double v, double w) {
    const double R = sqrt(u * u + v * v + w * w);
    return -(u * log_a_plus_r(v, R, u, w) + v * log_a_plus_r(u, R, v, w) - w * atan2(u * v, w * R));
}

// t^T H t with H the antiderivatives of the second derivatives of 1/R, weights
// c = (txx, tyy, tzz, 2txy, 2txz, 2tyz).
struct MagCoef { double c[6]; };

__device__ __forceinline__ double magnetic_corner(double u, double v, double w, const MagCoef &k) {
    const double R = sqrt(u * u + v * v + w * w);
    const double hxx = -atan(v * w / (u * R));
    const double hyy = -atan(u * w / (v * R));
    const double hzz = -atan2(u * v, w * R);
    const double hxy = log_a_plus_r(w, R, u, v);
    const double hxz = log_a_plus_r(v, R, u, w);
    const double hyz = log_a_plus_r(u, R, v, w);
    return k.c[0] * hxx + k.c[1] * hyy + k.c[2] * hzz + k.c[3] * hxy + k.c[4] * hxz + k.c[5] * hyz;
}

struct Lattice {
    int nbx1, nby1, nz1;     // lattice points in u, v, w
    int a_max, b_max;
    double dx, dy;
    const double *zw;        // nz + 1 values of w
};

__global__ void k_corner_lattice(Lattice L, int magnetic, MagCoef mc, double *out) {
    pdl_wait();  // (the launch before may still read the lattice)
    const size_t total = (size_t)L.nbx1 * L.nby1 * L.nz1;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int e = (int)(i % L.nbx1);
        const int f = (int)((i / L.nbx1) % L.nby1);
        const int k = (int)(i / ((size_t)L.nbx1 * L.nby1));
        const double u = (-(double)L.b_max - 0.5 + e) * L.dx;
        const double v = (-(double)L.a_max - 0.5 + f) * L.dy;
        const double w = L.zw[k];
        out[i] = magnetic ? magnetic_corner(u, v, w, mc) : gravity_corner(u, v, w);
    }
}

// Far from the station the 8-corner sums cancel (their terms grow like R log R
// while the field falls like 1/R^2): a prism whose centre is at least kFar times its
// largest side away is integrated by tensor Gauss-Legendre cubature of the smooth
// integrand instead, 5 points per axis up to 3 kFar sides, 4 up to 8 kFar and 3
// beyond (relative error at most about 5e-13 there, against 1e-7 for the corner
// sums at 100 sides).
constexpr double kFar = 8.0;
// Gauss-Legendre nodes and weights on [-1, 1], as constants of the unrolled rules
__host__ __device__ constexpr double gl_node(int np, int i) {
    return np == 5 ? (i == 0 ? -0.90617984593866399280 : i == 1 ? -0.53846931010568309104 : i == 2 ? 0.0
                      : i == 3 ? 0.53846931010568309104 : 0.90617984593866399280)
         : np == 4 ? (i == 0 ? -0.86113631159405257522 : i == 1 ? -0.33998104358485626480
                      : i == 2 ? 0.33998104358485626480 : 0.86113631159405257522)
                   : (i == 0 ? -0.77459666924148337704 : i == 1 ? 0.0 : 0.77459666924148337704);
}
__host__ __device__ constexpr double gl_weight(int np, int i) {
    return np == 5 ? (i == 0 || i == 4 ? 0.23692688505618908751 : i == 2 ? 0.56888888888888888889 : 0.47862867049936646804)
         : np == 4 ? (i == 0 || i == 3 ? 0.34785484513745385737 : 0.65214515486254614263)
                   : (i == 1 ? 0.88888888888888888889 : 0.55555555555555555556);
}

// The integral over [u1, u2] x [v1, v2] x [w1, w2] of w / R^3 (gravity) or of
// t^T (d2(1/R)/dr dr) t = (c0 (3u^2 - R^2) + c1 (3v^2 - R^2) + c2 (3w^2 - R^2)
// + 3 (c3 uv + c4 uw + c5 vw)) / R^5 (magnetic), by an n-point tensor rule in
// precision F.  The integrand is smooth there and the sum has no cancellation to
// speak of, so for an FP32 operator (whose spectra are rounded to FP32) the rule runs
// in FP32, some 60 times the FP64 rate; FP64 operators keep FP64.
// The parts that keep their sign, or change it, when u or v does come out apart, so
// that one evaluation serves the offsets (+-u, +-v): part[0] + su sv part[1] + su part[2]
// + sv part[3] (gravity: part[0] alone).
template <typename F> __device__ __forceinline__ F rsqrt_t(F x);
template <> __device__ __forceinline__ double rsqrt_t<double>(double x) { return rsqrt(x); }
template <> __device__ __forceinline__ float rsqrt_t<float>(float x) { return rsqrtf(x); }

// magnetic coefficients of the cubature, t = (c0, c1, c2) on the diagonal, c3 c4 c5 off it:
// 3 (t . r)^2 - R^2 = au u^2 + av v^2 + aw w^2 + 3 c3 uv + 3 c4 uw + 3 c5 vw
template <typename F> struct FarCoef { F au, av, aw, uv, uw, vw; };

template <int NP, typename F, bool MAG>
__device__ __forceinline__ void far_cubature(F uc, F hu, F vc, F hv, F wc, F hw, const FarCoef<F> &k, F (&part)[4]) {
    F s0 = 0, suv = 0, su = 0, sv = 0;
#pragma unroll
    for (int a = 0; a < NP; ++a) {
        const F u = uc + hu * (F)gl_node(NP, a), u2 = u * u;
#pragma unroll
        for (int b = 0; b < NP; ++b) {
            const F v = vc + hv * (F)gl_node(NP, b);
            const F uv2 = u2 + v * v, e = MAG ? k.au * u2 + k.av * (v * v) : F(0);
            const F wab = (F)(gl_weight(NP, a) * gl_weight(NP, b));
            F i0 = 0, i5 = 0, i5w = 0;  // sums over w: the even part, 1/R^5, w/R^5 (gravity: w/R^3)
#pragma unroll
            for (int c = 0; c < NP; ++c) {
                const F w = wc + hw * (F)gl_node(NP, c), w2 = w * w;
                const F ir = rsqrt_t<F>(uv2 + w2);
                const F ir2 = ir * ir, g3 = (F)gl_weight(NP, c) * ir * ir2;
                if (MAG) {
                    const F g5 = g3 * ir2;
                    i0 += g5 * (e + k.aw * w2);
                    i5 += g5;
                    i5w += g5 * w;
                } else {
                    i0 += g3 * w;
                }
            }
            s0 += wab * i0;
            if (MAG) {
                suv += wab * (u * v) * i5;
                su += wab * u * i5w;
                sv += wab * v * i5w;
            }
        }
    }
    part[0] = s0;
    part[1] = MAG ? k.uv * suv : F(0);
    part[2] = MAG ? k.uw * su : F(0);
    part[3] = MAG ? k.vw * sv : F(0);
}

// Depth range of a layer (centre and half height below the stations), its squared
// near-field radius, all in length_unit, and the cubature's volume element times the scale of
// the spectra.
template <typename F> struct LayerGeom {
    F wc, hw, near2;
    double vol;
};

// The circulant tables of a build's layers, T[c_y mod Ny][c_x mod Nx] =
// K(c_y + off_y, c_x + off_x) for c in [-(n-1), s-1], zero elsewhere.  K is the 8-corner
// sum of the lattice, or the far-field cubature.
template <typename F> struct TableGeom {
    const double *lat;
    int nbx1, nby1, k0;  // lattice points, and the lattice plane of the launch's first layer
    int Nx, Ny, sx, sy, nx, ny, off_x, off_y, a_max, b_max;
    int a0, na, b0, nb;  // |c + off| runs over [a0, a0 + na) along y and [b0, b0 + nb) along x
    double scale;
    const F *axis;              // prism centres -|c + off| cell: [nb] along x, then [na] along y
    const LayerGeom<F> *layer;  // of the launch's first layer
    F hu, hv;                   // half cells (lengths in length_unit)
    FarCoef<F> k;
};

// 8-corner sum at offsets (cy + off_y, cx + off_x) = (a, b), inside the lattice window
template <typename F>
__device__ __forceinline__ double corner_sum(const TableGeom<F> &G, int r, int a, int b) {
    const int e = G.b_max - b, f = G.a_max - a;
    double s = 0.0;
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int df = 0; df < 2; ++df)
#pragma unroll
            for (int de = 0; de < 2; ++de) {
                const double t = G.lat[((size_t)(G.k0 + r + dk) * G.nby1 + (f + df)) * G.nbx1 + (e + de)];
                s += ((de + df + dk) & 1) ? t : -t;
            }
    return s;
}

// Two table rows and their FP64 row transform: a CTA takes the rows of offsets a and -a
// (even: those of |a| = 2q and 2q + 1, all an even table needs), one thread per |b|
// evaluates the prism once for every row and sign it serves.  The FP64 units of this GPU
// do two operations a cycle and SM, so what decides an entry's address, distance and rule
// must not use them (done entry by entry in FP64 inside the transform, a 1023 x 1023 layer
// of an FP32 operator took 205 us; a table kernel of its own and the transform 75 us),
// and evaluation in FP32 runs beside the FP64 butterflies of other CTAs.
template <typename F, bool MAG>
__global__ void __launch_bounds__(256) k_table_rows(TableGeom<F> G, OpView<double> op, RowShape rs, int even,
                                                    int after_lattice, double2 *Zs) {
    using C = double2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = op.Nx, ncol = op.ncol, q = blockIdx.x, r = blockIdx.y;
    int ia[2], iy[2];
    bool ok[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        ia[l] = even ? 2 * q + l : q;
        const int a = G.a0 + ia[l], cy = (even || l == 0 ? a : -a) - G.off_y;
        ok[l] = ia[l] < G.na && cy >= -(G.ny - 1) && cy <= G.sy - 1 && !(!even && l == 1 && a == 0);
        iy[l] = cy < 0 ? cy + G.Ny : cy;
    }
    if (!ok[0] && !ok[1]) return;
    // Where one lattice serves the whole build, launches after the first follow a column launch
    // that started its own work when everything before it was complete: the lattice is there,
    // and only Zs is waited for.
    if (after_lattice) pdl_wait();
    C *buf0 = reinterpret_cast<C *>(smem_raw), *buf1 = buf0 + N, *tw = buf1 + N;
    load_twiddles(tw, op.twx, N);
    for (int i = threadIdx.x; i < N; i += blockDim.x) buf0[i] = czero<C>();
    __syncthreads();
    const LayerGeom<F> lg = G.layer[r];
    for (int ib = threadIdx.x; ib < G.nb; ib += blockDim.x) {
        const F uc = G.axis[ib];  // offset (a, b) sees the prism centred at u = -b dx, v = -a dy
        const int b = G.b0 + ib;
        for (int l = 0; l < (even ? 2 : 1); ++l) {
            const int il = l == 0 ? ia[0] : ia[1];
            if (il >= G.na) break;
            const F vc = G.axis[G.nb + il];
            const F d2 = uc * uc + vc * vc + lg.wc * lg.wc;
            const bool far = d2 >= lg.near2;
            F part[4] = {0, 0, 0, 0};
            if (far) {
                if (d2 < F(9) * lg.near2) far_cubature<5, F, MAG>(uc, G.hu, vc, G.hv, lg.wc, lg.hw, G.k, part);
                else if (d2 < F(64) * lg.near2) far_cubature<4, F, MAG>(uc, G.hu, vc, G.hv, lg.wc, lg.hw, G.k, part);
                else far_cubature<3, F, MAG>(uc, G.hu, vc, G.hv, lg.wc, lg.hw, G.k, part);
            }
#pragma unroll
            for (int sg = 0; sg < 4; ++sg) {  // signs of a and b
                const int sa = (sg & 1) ? -1 : 1, sb = (sg & 2) ? -1 : 1;
                if ((even && sa < 0) || (sb < 0 && b == 0)) continue;
                const int comp = even ? l : (sg & 1), cx = sb * b - G.off_x;
                if (!(comp ? ok[1] : ok[0]) || cx < -(G.nx - 1) || cx > G.sx - 1) continue;
                double v;
                if (far) v = (double)(part[0] + (F)(sa * sb) * part[1] + (F)sb * part[2] + (F)sa * part[3]) * lg.vol;
                else v = corner_sum(G, r, sa * (G.a0 + il), sb * b) * G.scale;
                reinterpret_cast<double *>(buf0 + (cx < 0 ? cx + N : cx))[comp] = v;
            }
        }
    }
    __syncthreads();
    const C *X = fft_staged<double, false>(op.px, rs, buf0, buf1, tw, N, N);
    if (!after_lattice) pdl_wait();  // the column launch before this one may still read Zs
    pdl_go();
    C *out0 = Zs + ((size_t)r * G.Ny + iy[0]) * ncol, *out1 = Zs + ((size_t)r * G.Ny + iy[1]) * ncol;
    for (int k = threadIdx.x; k < ncol; k += blockDim.x) {
        const C zk = X[k], zm = X[k ? N - k : 0];
        if (ok[0]) out0[k] = mk<C>(zk.x + zm.x, zk.y - zm.y);
        if (ok[1]) out1[k] = mk<C>(zk.y + zm.y, zm.x - zk.x);
    }
}

// Column pass of the setup: spec[r] = FFT_y of layer r's row transforms, rounded, in the
// layout of the operator's kernels.
template <typename Rout>
__global__ void __launch_bounds__(256) k_col_spec(OpView<double> op, RecShape rs, const double2 *Zs, cpx<Rout> *spec,
                                                  int transposed, int real_only) {
    using Cx = cpx<Rout>;
    const int N = op.Ny, ncol = op.ncol, C = rs.C, c0 = blockIdx.x * C, cols = min(C, ncol - c0), r = blockIdx.y;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *bufA = smem_raw, *bufB = bufA + rs.buf;
    double2 *tw64 = reinterpret_cast<double2 *>(bufB + rs.buf);
    Cx *S = reinterpret_cast<Cx *>(tw64 + N);
    load_twiddles(tw64, op.twy, N);
    pdl_wait();
    pdl_go();
    layer_spectrum<Rout>(N, ncol, rs, op.py, c0, cols, Zs + (size_t)r * N * ncol, reinterpret_cast<double2 *>(bufA),
                         reinterpret_cast<double2 *>(bufB), tw64, S);
    Cx *Sr = spec + (size_t)r * N * ncol;
    if (real_only) {
        // the table is even in both offsets: the spectrum is real and even in ky, so only
        // ky <= Ny/2 is kept, as R[r][kx][ke] (fast paths)
        const int ke = even_spec_len(N), h = N / 2 + 1;
        Rout *out = reinterpret_cast<Rout *>(spec) + ((size_t)r * ncol + c0) * ke;
        for (int c = 0; c < cols; ++c)
            for (int k = threadIdx.x; k < h; k += blockDim.x) out[(size_t)c * ke + k] = S[k * C + c].x;
    } else if (transposed) {
        for (int c = 0; c < cols; ++c)
            for (int k = threadIdx.x; k < N; k += blockDim.x) Sr[(size_t)(c0 + c) * N + k] = S[k * C + c];
    } else {
        for (int it = threadIdx.x; it < N * C; it += blockDim.x) {
            const int k = fast_div(it, rs.mC), c = it - k * C;
            if (c < cols) Sr[(size_t)k * ncol + c0 + c] = S[it];
        }
    }
}

// ---------------------------------------------------------------------------
// Host helpers

// Radix plan of an N-point transform.  order 0: the cheapest product of codelet radices
// (by the codelets' operation counts, twiddles and a shared-memory round trip a stage),
// with even radices first and last where there are any (the pruned stages halve those);
// order 1: the same stages in reverse; order 2: the power-of-two part in radix 4 (and one
// radix 2), then the odd primes.
static void cheapest_radices(int n, int N, int most, double cost, std::vector<int> &cur, double &best,
                             std::vector<int> &out) {
    // real operations of the codelets, radix 0 to 17
    static const double ops[kMaxRadix + 1] = {0,   0,   4,   14,  16,  40,  40,  84,  56,
                                              104, 100, 220, 104, 312, 196, 250, 168, 544};
    if (n == 1) {
        if (cost < best) { best = cost; out = cur; }
        return;
    }
    for (int r = std::min(n, most); r >= 2; --r) {
        if (n % r) continue;
        // butterflies, the round trip and the twiddles of one stage
        const double c = (double)N / r * ops[r] + 14.0 * N + 300.0;
        if (cost + c >= best) continue;
        cur.push_back(r);
        cheapest_radices(n / r, N, r, cost + c, cur, best, out);
        cur.pop_back();
    }
}

bool plan_size(int N, FftPlanDev &plan, int order) {
    if (N < 1 || N > 2048 || order < 0 || order > 2) return false;
    int n = N, e = 0;
    while (n % 2 == 0) { n /= 2; ++e; }
    std::vector<int> rs, odd;
    for (int p : {3, 5, 7, 11, 13, 17})
        while (n % p == 0) { n /= p; odd.push_back(p); }
    if (n != 1) return false;
    if (order == 2) {
        rs.assign(e / 2, 4);
        if (e % 2) rs.push_back(2);
        rs.insert(rs.end(), odd.begin(), odd.end());
    } else {
        std::vector<int> cur;
        double best = 1e300;
        cheapest_radices(N, N, kMaxRadix, 0.0, cur, best, rs);  // descending
        std::stable_sort(rs.begin(), rs.end(), [](int a, int b) { return a % 2 < b % 2; });
        if (rs.size() > 2 && rs[1] % 2 == 0) std::swap(rs[1], rs.back());  // an even one last as well
        if (order == 1) std::reverse(rs.begin(), rs.end());
    }
    while (rs.size() < 2) rs.push_back(1);  // the transforms run at least two stages
    if ((int)rs.size() > kMaxStages) return false;
    plan.N = N;
    plan.nst = (int)rs.size();
    plan.mmax = 1;
    int Ns = 1;
    for (int i = 0; i < kMaxStages; ++i) {
        const int r = i < plan.nst ? rs[i] : 1;
        FftStage &st = plan.st[i];
        st.rad = r;
        st.M = N / r;
        st.Ns = Ns;
        st.tws = std::max(1, N / (Ns * r));
        st.mNs = div_magic(Ns);
        if (i < plan.nst && r > 1) plan.mmax = std::max(plan.mmax, st.M);
        Ns *= r;
    }
    return true;
}

int autotune_size(int minN) {
    for (int N = std::max(1, minN);; ++N) {
        int n = N;
        for (int p : {2, 3, 5, 7})
            while (n % p == 0) n /= p;
        if (n == 1) return N;
    }
}

void make_twiddles(int N, std::vector<double> &re, std::vector<double> &im) {
    re.resize(N);
    im.resize(N);
    const double two_pi = 6.283185307179586476925286766559;
    for (int k = 0; k < N; ++k) {
        // exact values at the quarter points keep the small radices exact
        if (4 * k % N == 0) {
            const int q = 4 * k / N;
            const double c[4] = {1, 0, -1, 0}, s[4] = {0, -1, 0, 1};
            re[k] = c[q];
            im[k] = s[q];
        } else {
            const double a = two_pi * (double)k / (double)N;
            re[k] = std::cos(a);
            im[k] = -std::sin(a);
        }
    }
}

size_t elem_bytes(gj_precision p) { return p == GJ_FP64 ? sizeof(double) : sizeof(float); }

// FP32, N_x = 512 with at most 256 prisms and stations along x, and N_y = 512 (or
// 256) with at most 256 (128) along y.
bool fast_eligible(const gj_op *op) {
    const int hy = op->Ny / 2;
    return op->prec == GJ_FP32_MIXED && op->Nx == 512 && (op->Ny == 512 || op->Ny == 256) && op->nx <= 256 &&
           op->sx <= 256 && op->ny <= hy && op->sy <= hy;
}

// Items per (field, kx) column of the fast column kernels: one per layer at N_y = 512,
// one per layer pair at N_y = 256.
int fast_col_items(int Ny, int nz) { return Ny == 256 ? (nz + 1) / 2 : nz; }

// Largest number of warps that share one (field, kx) column when persistent column
// kernels of `warps` warps split the (kx, field, item) sequence into balanced segments.
int fast_slots(int nfield, int ncol, int nz, long long warps) {
    const long long T = (long long)nfield * ncol * nz;
    const long long Wt = std::min(warps, T);
    auto owner = [&](long long t) { return ((t + 1) * Wt + T - 1) / T - 1; };
    long long mx = 1;
    for (long long c = 0; c < (long long)nfield * ncol; ++c)
        mx = std::max(mx, owner(c * nz + nz - 1) - owner(c * nz) + 1);
    return (int)mx;
}

bool fast1024_eligible(const gj_op *op) {
    return op->prec == GJ_FP32_MIXED && !op->fast && op->Ny == 1024 && op->ny <= 512 && op->sy <= 512;
}
// its row kernels hold 512 values of a line (16 a lane); longer lines take the general ones
bool rows1024_eligible(const gj_op *op) { return op->fast1024 && op->Nx == 1024 && op->nx <= 512 && op->sx <= 512; }

static gj_status upload_twiddles(int N, gj_precision prec, void **out) {
    std::vector<double> re, im;
    make_twiddles(N, re, im);
    if (prec == GJ_FP64) {
        std::vector<double2> h(N);
        for (int k = 0; k < N; ++k) h[k] = make_double2(re[k], im[k]);
        GJ_CUDA(cudaMalloc(out, N * sizeof(double2)));
        GJ_CUDA(cudaMemcpy(*out, h.data(), N * sizeof(double2), cudaMemcpyHostToDevice));
    } else {
        std::vector<float2> h(N);
        for (int k = 0; k < N; ++k) h[k] = make_float2((float)re[k], (float)im[k]);
        GJ_CUDA(cudaMalloc(out, N * sizeof(float2)));
        GJ_CUDA(cudaMemcpy(*out, h.data(), N * sizeof(float2), cudaMemcpyHostToDevice));
    }
    return GJ_OK;
}

struct gj_setup_scratch_impl;
static void scratch_free(gj_setup_scratch_impl *sc);

static void free_op_memory(gj_op *op) {
    if (!op) return;
    scratch_free(op->scratch);
    op->scratch = nullptr;
    cudaFree(op->twx); cudaFree(op->twy); cudaFree(op->spec);
    cudaFree(op->Z); cudaFree(op->Y); cudaFree(op->W); cudaFree(op->V); cudaFree(op->twtab);
    op->twx = op->twy = op->spec = op->Z = op->Y = op->W = op->V = op->twtab = nullptr;
}

// Work buffers of the spectrum build for `layers` consecutive layers at a time: the FP64
// corner lattice (the depth planes of lat_layers consecutive layers: about 20 x 20 points each
// for cubic cells), the FP64 row transforms of the tables (rows outside the offsets in use stay
// zero), the geometry and FP64 twiddles.  Kept by operators that rebuild their spectra per
// layer.
struct gj_setup_scratch_impl {
    double *lat = nullptr;
    void *axis = nullptr, *layer = nullptr;  // TableGeom's, in the far field's precision
    double2 *Zs = nullptr;
    double *zw = nullptr;
    void *twx64 = nullptr, *twy64 = nullptr;
    bool own_tw = false;
    int layers = 0, lat_layers = 0;
};

static void scratch_free(gj_setup_scratch_impl *sc) {
    if (!sc) return;
    cudaFree(sc->lat); cudaFree(sc->axis); cudaFree(sc->layer); cudaFree(sc->Zs); cudaFree(sc->zw);
    if (sc->own_tw) { cudaFree(sc->twx64); cudaFree(sc->twy64); }
    delete sc;
}

// The corner lattice serves only the prisms nearer than kFar sizes (the rest take
// the cubature), so it spans the offsets c + off in [-W, W] of each direction that the
// table uses, W = ceil(kFar * largest side / cell) + 1: 2W + 2 points per direction
// at most, whatever the grid.  b_max is the largest offset in the window, nb1 the
// lattice points (offsets b_max down to the smallest, plus one).
struct LatticeWindow { int b_max, nbx1, a_max, nby1; };
static LatticeWindow lattice_window(const gj_op *op) {
    double size = std::max(op->dx, op->dy);
    for (int k = 0; k < op->nz; ++k) size = std::max(size, op->z_edges[k + 1] - op->z_edges[k]);
    auto one = [&](int off, int s, int n, double cell, int &hi, int &nb) {
        const int W = (int)std::ceil(kFar * size / cell) + 1;
        hi = std::min(off + s - 1, W);
        const int lo = std::max(off - n + 1, -W);
        nb = std::max(2, hi - lo + 2);
    };
    LatticeWindow w;
    one(op->off_x, op->sx, op->nx, op->dx, w.b_max, w.nbx1);
    one(op->off_y, op->sy, op->ny, op->dy, w.a_max, w.nby1);
    return w;
}

static MagCoef mag_coef(const gj_op *op) {
    MagCoef mc{};
    const double d2r = 3.14159265358979323846 / 180.0;
    const double I = op->mag.incl_deg * d2r, D = op->mag.decl_deg * d2r;
    const double t[3] = {std::cos(I) * std::sin(D), std::cos(I) * std::cos(D), std::sin(I)};
    mc.c[0] = t[0] * t[0]; mc.c[1] = t[1] * t[1]; mc.c[2] = t[2] * t[2];
    mc.c[3] = 2 * t[0] * t[1]; mc.c[4] = 2 * t[0] * t[2]; mc.c[5] = 2 * t[1] * t[2];
    return mc;
}

static double table_scale(const gj_op *op) {
    // the row passes of the build, and those of the general kernels, leave out the half of
    // the real-line split: it is part of the spectra (a power of two: nothing rounds)
    const double scale = (op->fast || op->fast1024 ? 0.5 : 0.25) / ((double)op->Nx * (double)op->Ny);
    if (op->field == GJ_MAGNETIC) return scale * op->mag.F_nT / (4.0 * 3.14159265358979323846);
    // G = 6.6743e-11 m^3 kg^-1 s^-2; g/cc -> kg/m^3 (1e3); m/s^2 -> mGal (1e5)
    return scale * 6.6743e-11 * 1.0e3 * 1.0e5;
}

// range of |c + off| over c in [-(n-1), s-1]
static void offset_span(int off, int s, int n, int &lo, int &count) {
    const int first = off - (n - 1), last = off + s - 1;
    lo = first > 0 ? first : (last < 0 ? -last : 0);
    count = std::max(std::abs(first), std::abs(last)) - lo + 1;
}

// The cubature's lengths are in units of about a cell, a power of two, so that nothing rounds:
// in metres, a distance's fifth power left FP32 beyond 3e7 m (or below 3e-8).
static double length_unit(const gj_op *op) { return std::ldexp(1.0, std::ilogb(std::max(op->dx, op->dy))); }

// TableGeom's axis and layer arrays in precision F (as bytes)
template <typename F>
static void table_geometry(const gj_op *op, const std::vector<double> &zw, std::vector<char> &axis,
                           std::vector<char> &geom) {
    int a0, na, b0, nb;
    offset_span(op->off_y, op->sy, op->ny, a0, na);
    offset_span(op->off_x, op->sx, op->nx, b0, nb);
    axis.resize((nb + na) * sizeof(F));
    geom.resize(op->nz * sizeof(LayerGeom<F>));
    F *ax = reinterpret_cast<F *>(axis.data());
    const double to = 1.0 / length_unit(op);
    for (int i = 0; i < nb; ++i) ax[i] = (F)(-(double)(b0 + i) * op->dx * to);
    for (int i = 0; i < na; ++i) ax[nb + i] = (F)(-(double)(a0 + i) * op->dy * to);
    // of w / R^3 (gravity) and 1 / R^3 (magnetic) per unit of volume
    const double per = op->field == GJ_MAGNETIC ? to * to * to : to * to;
    LayerGeom<F> *lg = reinterpret_cast<LayerGeom<F> *>(geom.data());
    for (int k = 0; k < op->nz; ++k) {
        const double size = std::max(std::max(op->dx, op->dy), zw[k + 1] - zw[k]);
        lg[k].wc = (F)(0.5 * (zw[k] + zw[k + 1]) * to);
        lg[k].hw = (F)(0.5 * (zw[k + 1] - zw[k]) * to);
        lg[k].near2 = (F)(kFar * kFar * (size * to) * (size * to));
        lg[k].vol = 0.125 * op->dx * op->dy * (zw[k + 1] - zw[k]) * per * table_scale(op);
    }
}

// Layers that the corner lattice of a rebuilding operator covers at a time: all (one launch a
// product) while their planes take no more than one layer's row transforms, or a megabyte;
// layers much thicker than the cells are wide spread the near field over the whole grid, where
// all planes would outweigh the spectra that the operator does not keep: then one.
constexpr size_t kLatticeKeep = 1 << 20;
static int kept_lattice_layers(const gj_op *op) {
    const LatticeWindow lw = lattice_window(op);
    const size_t all = (size_t)lw.nbx1 * lw.nby1 * (op->nz + 1) * sizeof(double);
    return all <= std::max(kLatticeKeep, (size_t)op->Ny * op->ncol * sizeof(double2)) ? op->nz : 1;
}

static gj_status scratch_alloc(const gj_op *op, int layers, int lat_layers, gj_setup_scratch_impl **out) {
    gj_setup_scratch_impl *sc = new (std::nothrow) gj_setup_scratch_impl();
    if (!sc) { set_error("setup scratch: host allocation failed"); return GJ_ERR_OOM; }
    sc->layers = layers;
    sc->lat_layers = lat_layers;
    gj_status rc = GJ_OK;
    cudaError_t e;
    if (op->prec == GJ_FP64) {
        sc->twx64 = op->twx;
        sc->twy64 = op->twy;
    } else {
        sc->own_tw = true;
        if ((rc = upload_twiddles(op->Nx, GJ_FP64, &sc->twx64)) != GJ_OK) { scratch_free(sc); return rc; }
        if ((rc = upload_twiddles(op->Ny, GJ_FP64, &sc->twy64)) != GJ_OK) { scratch_free(sc); return rc; }
    }
    const LatticeWindow lw = lattice_window(op);
    const size_t plane = (size_t)lw.nbx1 * lw.nby1;
    std::vector<double> zw(op->nz + 1);
    for (int k = 0; k <= op->nz; ++k) zw[k] = op->z_edges[k] - op->station_z;
    std::vector<char> axis, geom;
    if (op->prec == GJ_FP32_MIXED) table_geometry<float>(op, zw, axis, geom);
    else table_geometry<double>(op, zw, axis, geom);
    const size_t zsb = (size_t)layers * op->Ny * op->ncol * sizeof(double2);
    if ((e = cudaMalloc(&sc->lat, plane * (lat_layers + 1) * sizeof(double))) != cudaSuccess ||
        (e = cudaMalloc(&sc->Zs, zsb)) != cudaSuccess || (e = cudaMemset(sc->Zs, 0, zsb)) != cudaSuccess ||
        (e = cudaMalloc(&sc->zw, zw.size() * sizeof(double))) != cudaSuccess ||
        (e = cudaMalloc(&sc->axis, axis.size())) != cudaSuccess ||
        (e = cudaMalloc(&sc->layer, geom.size())) != cudaSuccess ||
        (e = cudaMemcpy(sc->axis, axis.data(), axis.size(), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(sc->layer, geom.data(), geom.size(), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(sc->zw, zw.data(), zw.size() * sizeof(double), cudaMemcpyHostToDevice)) != cudaSuccess) {
        scratch_free(sc);
        return cuda_fail(e, "setup scratch");
    }
    *out = sc;
    return GJ_OK;
}

// The corner lattice of the depth planes of layers r0 .. r0 + lat_layers - 1 (enqueues one
// launch).  A point is a chain of FP64 logarithms and arctangents, so the points are spread
// one warp a block.
static void build_lattice(const gj_op *op, const gj_setup_scratch_impl &sc, int r0, cudaStream_t st) {
    const LatticeWindow lw = lattice_window(op);
    Lattice L;
    L.b_max = lw.b_max;
    L.a_max = lw.a_max;
    L.nbx1 = lw.nbx1;
    L.nby1 = lw.nby1;
    L.nz1 = sc.lat_layers + 1;
    L.dx = op->dx;
    L.dy = op->dy;
    L.zw = sc.zw + r0;
    const size_t pts = (size_t)L.nbx1 * L.nby1 * L.nz1;
    launch_after(k_corner_lattice, dim3((unsigned)std::min<size_t>(4864, (pts + 31) / 32)), dim3(32), 0, st, L,
                 op->field == GJ_MAGNETIC, mag_coef(op), sc.lat);
}

// Tables of layers r0 .. r0 + count - 1 (count <= the scratch's layers), after
// build_lattice, and their FP64 row transforms into the scratch's Zs (even_rows: the rows
// 0 .. Ny/2 alone).  Enqueues only (no synchronisation).
// The builds go through the layers in order, from layer 0.
template <typename F>
static void launch_table_rows(const gj_op *op, const gj_setup_scratch_impl &sc, int r0, int count,
                              const OpView<double> &v, cudaStream_t st) {
    const bool all = sc.lat_layers == op->nz;     // one lattice for the whole build
    const bool after_lattice = r0 == 0 || !all;  // else it is older than the launch before this one
    const LatticeWindow lw = lattice_window(op);
    TableGeom<F> G;
    G.lat = sc.lat; G.nbx1 = lw.nbx1; G.nby1 = lw.nby1; G.k0 = all ? r0 : 0;
    G.Nx = op->Nx; G.Ny = op->Ny; G.sx = op->sx; G.sy = op->sy; G.nx = op->nx; G.ny = op->ny;
    G.off_x = op->off_x; G.off_y = op->off_y; G.a_max = lw.a_max; G.b_max = lw.b_max;
    offset_span(op->off_y, op->sy, op->ny, G.a0, G.na);
    offset_span(op->off_x, op->sx, op->nx, G.b0, G.nb);
    G.scale = table_scale(op);
    G.axis = static_cast<const F *>(sc.axis);
    G.layer = static_cast<const LayerGeom<F> *>(sc.layer) + r0;
    G.hu = (F)(0.5 * op->dx / length_unit(op));
    G.hv = (F)(0.5 * op->dy / length_unit(op));
    const MagCoef mc = mag_coef(op);
    const double tr = mc.c[0] + mc.c[1] + mc.c[2];
    G.k = FarCoef<F>{(F)(3 * mc.c[0] - tr), (F)(3 * mc.c[1] - tr), (F)(3 * mc.c[2] - tr),
                     (F)(3 * mc.c[3]),      (F)(3 * mc.c[4]),      (F)(3 * mc.c[5])};
    const RowShape rs = row_shape_of(op->px, 1, sizeof(double2));
    const dim3 grid(op->even_rows ? (G.na + 1) / 2 : G.na, count);
    const int T = gen_threads(op->px.mmax, 1), even = op->even_rows ? 1 : 0;
    const size_t sm = row_smem(op->Nx, rs.pitch, sizeof(double2));
    launch_after(op->field == GJ_MAGNETIC ? k_table_rows<F, true> : k_table_rows<F, false>, grid, dim3(T), sm, st, G, v,
                 rs, even, after_lattice ? 1 : 0, sc.Zs);
}

static OpView<double> build_rows(const gj_op *op, const gj_setup_scratch_impl &sc, int r0, int count, cudaStream_t st) {
    OpView<double> v{};
    v.sx = op->sx; v.sy = op->sy; v.nx = op->nx; v.ny = op->ny; v.nz = count;
    v.Nx = op->Nx; v.Ny = op->Ny; v.ncol = op->ncol; v.px = op->px; v.py = op->py;
    v.twx = static_cast<const double2 *>(sc.twx64);
    v.twy = static_cast<const double2 *>(sc.twy64);
    if (op->prec == GJ_FP32_MIXED) launch_table_rows<float>(op, sc, r0, count, v, st);
    else launch_table_rows<double>(op, sc, r0, count, v, st);
    return v;
}

// Spectra of layers r0 .. r0 + count - 1 into spec[0 .. count): the row transforms above,
// column transforms, rounding to the operator's precision.
template <typename Rout>
static void build_layers(const gj_op *op, const gj_setup_scratch_impl &sc, int r0, int count, cpx<Rout> *spec,
                         cudaStream_t st) {
    const OpView<double> v = build_rows(op, sc, r0, count, st);
    const RecShape cs = rec_shape(op->py, op->even_rows, sizeof(cpx<Rout>));
    launch_after(k_col_spec<Rout>, dim3((op->ncol + cs.C - 1) / cs.C, count), dim3(gen_threads(op->py.mmax, cs.lines)),
                 rec_smem(cs, op->Ny, sizeof(cpx<Rout>)), st, v, cs, sc.Zs, spec, (op->fast || op->fast1024) ? 1 : 0,
                 op->real_spec ? 1 : 0);
}

static void set_build_attributes() {
    allow_max_smem(k_table_rows<float, false>);
    allow_max_smem(k_table_rows<float, true>);
    allow_max_smem(k_table_rows<double, false>);
    allow_max_smem(k_table_rows<double, true>);
    allow_max_smem(k_col_spec<float>);
    allow_max_smem(k_col_spec<double>);
}

// The library's choice of the launch shapes, as reported: those of both fields' launches (others
// pick their own until tuned).
static void auto_shapes(gj_op *op, bool rows, bool cols, bool layers) {
    const size_t cs = 2 * elem_bytes(op->prec);
    if (rows) {
        op->rows_tuned = false;
        op->P_row = pick_row_pairs(op->px, (long long)op->nz * op->ny, cs);
        if (op->fast1024) {  // transposed intermediates: runs of P lines
            op->P_row = 16;
            while (op->P_row > 1 && row_smem(op->Nx, odd_pitch(op->P_row), cs) > kGenSmem) op->P_row >>= 1;
        }
    }
    const ColPick both = pick_cols(op->py, op->ncol, op->recompute ? 1 : op->nz, 2, cs, false);
    if (cols) { op->cols_tuned = false; op->C_col = both.C; }
    if (layers) { op->layers_tuned = false; op->L_grp = both.L; }
}

// where layer r's spectrum starts, in complex values (the even real spectra: two values each)
static size_t spec_offset(const gj_op *op, int r) {
    return op->real_spec ? (size_t)r * op->ncol * even_spec_len(op->Ny) / 2 : (size_t)r * op->Ny * op->ncol;
}

template <typename Rout>
static gj_status build_spectra(gj_op *op, cudaStream_t st) {
    gj_setup_scratch_impl *sc = nullptr;
    // as many layers at a time as fit a quarter of a gigabyte of row transforms
    const size_t per = (size_t)op->Ny * op->ncol * sizeof(double2);
    const int most = (int)std::max<size_t>(1, std::min<size_t>(op->nz, ((size_t)256 << 20) / per));
    gj_status rc = scratch_alloc(op, most, op->nz, &sc);
    if (rc != GJ_OK) return rc;
    set_build_attributes();
    build_lattice(op, *sc, 0, st);
    for (int r = 0; r < op->nz; r += most)
        build_layers<Rout>(op, *sc, r, std::min(most, op->nz - r),
                           static_cast<cpx<Rout> *>(op->spec) + spec_offset(op, r), st);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    scratch_free(sc);
    if (e != cudaSuccess) return cuda_fail(e, "spectra setup");
    return GJ_OK;
}

void recompute_begin(const gj_op *op, cudaStream_t st) {
    if (op->scratch->lat_layers == op->nz) build_lattice(op, *op->scratch, 0, st);
}

void recompute_rows(const gj_op *op, int r, cudaStream_t st) {
    if (op->scratch->lat_layers != op->nz) build_lattice(op, *op->scratch, r, st);
    build_rows(op, *op->scratch, r, 1, st);
}
const double2 *recompute_rows_out(const gj_op *op) { return op->scratch->Zs; }
const double2 *recompute_twy64(const gj_op *op) { return static_cast<const double2 *>(op->scratch->twy64); }

}  // namespace gj

using namespace gj;

extern "C" gj_status gj_bttb_setup_ex(const gj_grid *grid, gj_field field, const gj_mag *mag, gj_precision prec,
                                      int Npad_y, int Npad_x, int flags, gj_stream_t stream, gj_op **out) {
    if (!out) { set_error("gj_bttb_setup: out is NULL"); return GJ_ERR_ARG; }
    if (flags & ~GJ_SETUP_RECOMPUTE_SPECTRA) { set_error("gj_bttb_setup_ex: unknown flags"); return GJ_ERR_ARG; }
    *out = nullptr;
    if (!grid) { set_error("gj_bttb_setup: grid is NULL"); return GJ_ERR_ARG; }
    const gj_grid &G = *grid;
    if (G.sx < 1 || G.sy < 1 || G.nx < 1 || G.ny < 1 || G.nz < 1) {
        set_error("gj_bttb_setup: sizes must be >= 1"); return GJ_ERR_ARG;
    }
    if (!(G.dx > 0) || !(G.dy > 0) || !G.z_edges) {
        set_error("gj_bttb_setup: dx, dy must be > 0 and z_edges set"); return GJ_ERR_ARG;
    }
    for (int k = 0; k < G.nz; ++k)
        if (!(G.z_edges[k + 1] > G.z_edges[k])) { set_error("gj_bttb_setup: z_edges must increase"); return GJ_ERR_ARG; }
    if (!(G.station_z <= G.z_edges[0])) {
        set_error("gj_bttb_setup: stations must lie at or above the top of the mesh"); return GJ_ERR_ARG;
    }
    if (field != GJ_GRAVITY && field != GJ_MAGNETIC) { set_error("gj_bttb_setup: bad field"); return GJ_ERR_ARG; }
    if (field == GJ_MAGNETIC && !mag) { set_error("gj_bttb_setup: magnetic field needs gj_mag"); return GJ_ERR_ARG; }
    if (prec != GJ_FP64 && prec != GJ_FP32_MIXED) { set_error("gj_bttb_setup: bad precision"); return GJ_ERR_ARG; }
    const int minx = G.sx + G.nx - 1, miny = G.sy + G.ny - 1;
    int Nx = Npad_x > 0 ? Npad_x : autotune_size(minx);
    int Ny = Npad_y > 0 ? Npad_y : autotune_size(miny);
    if (Nx < minx || Ny < miny) {
        set_error("gj_bttb_setup: padded size must be >= stations + prisms - 1 in each direction");
        return GJ_ERR_ARG;
    }
    gj_op *op = new (std::nothrow) gj_op();
    if (!op) { set_error("gj_bttb_setup: host allocation failed"); return GJ_ERR_OOM; }
    if (!plan_size(Nx, op->px) || !plan_size(Ny, op->py)) {
        delete op;
        set_error("gj_bttb_setup: padded size unsupported (must be <= 2048 with prime factors <= 17)");
        return GJ_ERR_UNSUPPORTED;
    }
    op->sx = G.sx; op->sy = G.sy; op->nx = G.nx; op->ny = G.ny; op->nz = G.nz;
    op->off_x = G.off_x; op->off_y = G.off_y; op->dx = G.dx; op->dy = G.dy; op->station_z = G.station_z;
    op->z_edges.assign(G.z_edges, G.z_edges + G.nz + 1);
    op->field = field;
    op->mag = mag ? *mag : gj_mag{0, 0, 0};
    op->prec = prec;
    op->Nx = Nx; op->Ny = Ny; op->ncol = Nx / 2 + 1;
    const size_t cs = 2 * elem_bytes(prec);
    op->recompute = (flags & GJ_SETUP_RECOMPUTE_SPECTRA) != 0;
    // gravity over a station grid that covers the prisms with no offset: the table is even
    // in both offsets, so its spectrum is real
    op->even_table = field == GJ_GRAVITY && G.sx == G.nx && G.sy == G.ny && G.off_x == 0 && G.off_y == 0;
    op->even_rows = op->even_table && rec_smem(rec_shape(op->py, true, cs), Ny, cs) <= kGenSmemMax;
    op->fast = !op->recompute && fast_eligible(op);
    if (op->fast) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        op->col_grid = std::max(1, sms);
        const int ci = fast_col_items(Ny, G.nz);
        const long long warps = (long long)op->col_grid * f512::CWARPS;
        op->slots = std::max(fast_slots(1, 257, ci, warps), fast_slots(2, 257, ci, warps));
        op->real_spec = op->even_table;
    }
    op->fast1024 = !op->recompute && fast1024_eligible(op);
    op->rows1024 = rows1024_eligible(op);
    if (op->fast1024) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        op->col_grid = std::max(1, sms);
        const long long warps = (long long)op->col_grid * f1024::CWF;
        op->slots = std::max(fast_slots(1, op->ncol, G.nz, warps), fast_slots(2, op->ncol, G.nz, warps));
        op->real_spec = op->even_table;
    }
    const int layers = op->recompute ? 1 : G.nz;
    auto_shapes(op, true, true, true);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    gj_status rc;
    cudaError_t e;
    if ((rc = upload_twiddles(Nx, prec, &op->twx)) != GJ_OK) goto fail;
    if ((rc = upload_twiddles(Ny, prec, &op->twy)) != GJ_OK) goto fail;
    op->spec_bytes = op->real_spec ? (size_t)G.nz * op->ncol * even_spec_len(Ny) * (cs / 2)
                                   : (size_t)(op->recompute ? 1 : G.nz) * Ny * op->ncol * cs;
    if ((e = cudaMalloc(&op->spec, op->spec_bytes)) != cudaSuccess) { rc = cuda_fail(e, "spectra"); goto fail; }
    // the even spectra's padding entries stay zero
    if (op->real_spec && (e = cudaMemset(op->spec, 0, op->spec_bytes)) != cudaSuccess) {
        rc = cuda_fail(e, "spectra");
        goto fail;
    }
    if (op->recompute) {
        // one layer's spectrum plus the build's work buffers for one layer, kept
        if ((rc = scratch_alloc(op, 1, kept_lattice_layers(op), &op->scratch)) != GJ_OK) goto fail;
        set_build_attributes();
    } else {
        rc = (prec == GJ_FP64) ? build_spectra<double>(op, st) : build_spectra<float>(op, st);
        if (rc != GJ_OK) goto fail;
    }
    if (!op->fast && !op->fast1024) {
        const size_t zb = (size_t)G.nz * G.ny * op->ncol * cs;
        // partial layer sums (as many groups as a launch of one field or of both makes; a
        // tuned L_grp makes no more) and arrival counters, which are zero between launches
        for (int nf = 1; nf <= 2 && !op->recompute; ++nf) {
            const int L = pick_cols(op->py, op->ncol, layers, nf, cs, false).L;
            op->gen_slots = std::max(op->gen_slots, (layers + L - 1) / L);
        }
        // (the recompute mode sums in the plane of `spec`)
        const size_t sb = op->recompute ? 0 : (size_t)op->gen_slots * Ny * op->ncol * cs, yb = sb + op->ncol * sizeof(int);
        const size_t wb = (size_t)std::max(G.sy, 1) * op->ncol * cs;
        op->ws_bytes = zb + yb + wb;
        if ((e = cudaMalloc(&op->Z, zb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        if ((e = cudaMalloc(&op->Y, yb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        if ((e = cudaMalloc(&op->W, wb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        if ((e = cudaMemsetAsync(op->Y, 0, yb, st)) != cudaSuccess || (e = cudaStreamSynchronize(st)) != cudaSuccess) {
            rc = cuda_fail(e, "workspace");
            goto fail;
        }
        op->cnt = reinterpret_cast<int *>(static_cast<char *>(op->Y) + sb);
    } else {
        // transposed intermediates [r][kx][Ny/2], partials [kx][slots][Ny], counters
        const size_t zb = (size_t)G.nz * op->ncol * (Ny / 2) * cs;
        const size_t wb = (size_t)op->ncol * (Ny / 2) * cs;
        const size_t pb = (size_t)op->ncol * op->slots * Ny * cs;
        const size_t yb = pb + op->ncol * sizeof(int) + 64;
        op->ws_bytes = zb + wb + yb;
        if ((e = cudaMalloc(&op->Z, zb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        if ((e = cudaMalloc(&op->W, wb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        if ((e = cudaMalloc(&op->V, wb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        if ((e = cudaMalloc(&op->Y, yb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        op->ws_bytes += wb;
        // rows beyond the prisms / stations must read as zero; counters start at zero
        if ((e = cudaMemset(op->Z, 0, zb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        if ((e = cudaMemset(op->W, 0, wb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        if ((e = cudaMemset(op->V, 0, wb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        if ((e = cudaMemset(op->Y, 0, yb)) != cudaSuccess) { rc = cuda_fail(e, "workspace"); goto fail; }
        op->P = op->Y;
        op->cnt = reinterpret_cast<int *>(static_cast<char *>(op->Y) + pb);
        op->err = op->cnt + op->ncol + 8;
        const size_t tb = (size_t)(op->fast ? f512::TabTw<float>::WORDS : f1024::Tab1024<float>::WORDS) * sizeof(float2);
        if ((e = cudaMalloc(&op->twtab, tb)) != cudaSuccess) { rc = cuda_fail(e, "twiddle table"); goto fail; }
        if (op->fast)  // from the W512 table of the rows (N_x = 512 on this path, whatever N_y)
            f512::k_build_twtab<float><<<1, 256, 0, st>>>(static_cast<float2 *>(op->twtab),
                                                        static_cast<const float2 *>(op->twx));
        else  // from the W1024 table of the columns
            f1024::k_build_tab1024<float><<<1, 256, 0, st>>>(static_cast<float2 *>(op->twtab),
                                                           static_cast<const float2 *>(op->twy));
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) { rc = cuda_fail(e, "twiddle table"); goto fail; }
    }
    *out = op;
    return GJ_OK;
fail:
    free_op_memory(op);
    delete op;
    return rc;
}

extern "C" gj_status gj_bttb_setup(const gj_grid *grid, gj_field field, const gj_mag *mag, gj_precision prec,
                                   int Npad_y, int Npad_x, gj_stream_t stream, gj_op **out) {
    return gj_bttb_setup_ex(grid, field, mag, prec, Npad_y, Npad_x, 0, stream, out);
}

extern "C" gj_status gj_op_tune(gj_op *op, int P_row, int C_col, int L_grp, int radix_order) {
    if (!op) { set_error("gj_op_tune: NULL operator"); return GJ_ERR_ARG; }
    int dev = 0, optin = 48 * 1024;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const size_t cs = 2 * elem_bytes(op->prec);
    const size_t room = (size_t)optin - kStaticSmem;
    if (P_row > 0 && (P_row > 64 || row_smem(op->Nx, P_row, cs) > room)) {
        set_error("gj_op_tune: P_row too large for shared memory"); return GJ_ERR_ARG;
    }
    if (C_col > 0 && (C_col > 64 || col_smem(op->Ny, C_col, C_col, cs) > room)) {
        set_error("gj_op_tune: C_col too large for shared memory"); return GJ_ERR_ARG;
    }
    if (L_grp > 0 && L_grp > op->nz) { set_error("gj_op_tune: L_grp above nz"); return GJ_ERR_ARG; }
    FftPlanDev px = op->px, py = op->py;
    if (radix_order >= 0 && (!plan_size(op->Nx, px, radix_order) || !plan_size(op->Ny, py, radix_order))) {
        set_error("gj_op_tune: radix_order must be 0, 1 or 2"); return GJ_ERR_ARG;
    }
    if (radix_order >= 0) op->radix_order = radix_order;
    op->px = px;
    op->py = py;
    auto_shapes(op, !op->rows_tuned || P_row == GJ_TUNE_AUTO, !op->cols_tuned || C_col == GJ_TUNE_AUTO,
                !op->layers_tuned || L_grp == GJ_TUNE_AUTO);
    if (P_row > 0) { op->P_row = P_row; op->rows_tuned = true; }
    if (C_col > 0) { op->C_col = C_col; op->cols_tuned = true; }
    if (L_grp > 0) { op->L_grp = L_grp; op->layers_tuned = true; }
    return GJ_OK;
}

extern "C" gj_status gj_op_info(const gj_op *op, gj_op_info_t *info) {
    if (!op || !info) { set_error("gj_op_info: NULL argument"); return GJ_ERR_ARG; }
    info->sx = op->sx; info->sy = op->sy; info->nx = op->nx; info->ny = op->ny; info->nz = op->nz;
    info->Nx = op->Nx; info->Ny = op->Ny; info->ncol = op->ncol;
    info->field = op->field; info->precision = op->prec;
    info->spectrum_bytes = (int64_t)op->spec_bytes;
    info->workspace_bytes = (int64_t)op->ws_bytes;
    info->fast_path = op->fast ? 1 : (op->fast1024 ? 2 : 0);
    info->P_row = op->P_row; info->C_col = op->C_col; info->L_grp = op->L_grp;
    info->radix_order = op->radix_order;
    info->recompute = op->recompute ? 1 : 0;
    return GJ_OK;
}

extern "C" void gj_op_destroy(gj_op *op) {
    if (!op) return;
    sync_device();
    free_op_memory(op);
    delete op;
}
