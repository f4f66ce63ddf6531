// Batched mixed-radix FFTs in shared memory (self-sorting Stockham form), for any
// length up to 2048 whose prime factors are at most 17.
//
// A CTA transforms B interleaved lines of length N: element j of line b lives at
// buf[j * pitch + b].  Each stage of radix RAD reads the inputs j + r N/RAD (r < RAD)
// of butterfly j, applies the twiddles W_N^(r k N/(Ns RAD)) with k = j mod Ns,
// transforms them with a length-RAD DFT in registers and writes them to
// (j div Ns) Ns RAD + k + r Ns.  Radices 2 to 17 are codelets (the composite ones
// built from two smaller DFTs), so that two stages reach N = 289 and three any
// supported length: a stage costs a shared-memory round trip and a barrier, which is
// what bounded the transforms when every prime factor was a stage of its own.
// The first stage reads its inputs through a functor and the last one hands its outputs
// to one, so that global loads and stores, spectrum multiplies and layer sums need no
// passes of their own.  When at most half of the inputs (outputs) exist, the first
// (last) stage uses pruned codelets.
// Forward transforms use exp(-2 pi i jk/N); inverse ones are unnormalised.
#pragma once
#include <type_traits>
#include <utility>

#include "common.cuh"

namespace gj {

constexpr int kMaxStages = 8;
constexpr int kMaxRadix = 17;

struct FftStage {
    int rad, M, Ns, tws;  // radix, N / radix, product of the earlier radices, N / (Ns rad)
    unsigned mNs;         // fast_div multiplier of Ns
};

struct FftPlanDev {
    int N;
    int nst;
    int mmax;  // largest M: butterflies per line of the widest stage
    FftStage st[kMaxStages];
};

// n / d for 0 <= n, n d < 2^32, with m = div_magic(d) (0 stands for d = 1): with
// m = ceil(2^32 / d) the error of n m / 2^32 is below n d / 2^32 / d < 1 / d.
__host__ __device__ constexpr unsigned div_magic(int d) {
    return d <= 1 ? 0u : (unsigned)(((1ull << 32) + (unsigned)d - 1) / (unsigned)d);
}
__device__ __forceinline__ int fast_div(int n, unsigned m) { return m ? (int)__umulhi((unsigned)n, m) : n; }

// ---------------------------------------------------------------------------
// Roots of unity as compile-time constants: sine and cosine of 2 pi K / N by their
// Taylor series on the first octant (|x| <= pi/4: 13 terms leave less than 1e-26).

// sqrt(2)/2
template <typename R> __host__ __device__ constexpr R rsqrt2() { return R(0.70710678118654752440084436210485); }

constexpr double root_sin_series(double x) {
    const double q = x * x;
    double s = 1.0;
    for (int i = 12; i >= 1; --i) s = 1.0 - s * q / (double)((2 * i) * (2 * i + 1));
    return x * s;
}
constexpr double root_cos_series(double x) {
    const double q = x * x;
    double s = 1.0;
    for (int i = 12; i >= 1; --i) s = 1.0 - s * q / (double)((2 * i - 1) * (2 * i));
    return s;
}
constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr double root_cos(int k, int n) {
    k %= n;
    if (k < 0) k += n;
    if (2 * k > n) k = n - k;
    double sg = 1.0;
    if (4 * k > n) { sg = -1.0; k = n - 2 * k; n = 2 * n; }  // cos(pi - x)
    if (4 * k == n) return 0.0;
    if (8 * k > n) return sg * root_sin_series(kTwoPi * (double)(n - 4 * k) / (4.0 * (double)n));
    return sg * root_cos_series(kTwoPi * (double)k / (double)n);
}
constexpr double root_sin(int k, int n) { return root_cos(4 * k - n, 4 * n); }  // cos(x - pi/2)
template <int K, int N> struct Root {
    static constexpr double c = root_cos(K, N);
    static constexpr double s = root_sin(K, N);
};

template <int I0, int I1, class F>
__device__ __forceinline__ void static_for(F f) {
    if constexpr (I0 < I1) {
        f(std::integral_constant<int, I0>{});
        static_for<I0 + 1, I1>(f);
    }
}

// a * W_N^K (forward) or a * W_N^-K (inverse), K and N known at compile time
template <typename R, bool INV, int K, int N>
__device__ __forceinline__ cpx<R> rot(cpx<R> a) {
    using C = cpx<R>;
    constexpr int k = ((K % N) + N) % N;
    if constexpr (k == 0) return a;
    else if constexpr (2 * k == N) return mk<C>(-a.x, -a.y);
    else if constexpr (4 * k == N) return mul_mi<C, INV>(a);
    else if constexpr (4 * k == 3 * N) return mul_mi<C, !INV>(a);
    else if constexpr (8 * k % N == 0) {
        // (+-1 -+ i) / sqrt 2: two additions, and the factor joins the additions that follow
        constexpr R h = rsqrt2<R>();
        constexpr int o = 8 * k / N;  // 1, 3, 5, 7
        constexpr bool re = o == 1 || o == 7, im = (o == 1 || o == 3) == INV;  // signs of the root's parts
        const R x = re == im ? a.x - a.y : a.x + a.y, y = re == im ? a.x + a.y : a.x - a.y;
        // a (c + i d) with |c| = |d| = h: (c a.x - d a.y, d a.x + c a.y)
        return mk<C>(re ? h * x : -h * x, im ? h * y : -h * y);
    } else {
        constexpr R wr = root_part<R>(Root<k, N>::c), wi = root_part<R>(INV ? Root<k, N>::s : -Root<k, N>::s);
        return mk<C>(a.x * wr - a.y * wi, a.x * wi + a.y * wr);
    }
}

// ---------------------------------------------------------------------------
// Codelets: length-RAD DFTs in registers, natural order in and out.  Only the first NZ
// inputs may be nonzero (the others are not read where that saves work).

template <typename R, bool INV>
__device__ __forceinline__ void dft4(cpx<R> &a0, cpx<R> &a1, cpx<R> &a2, cpx<R> &a3) {
    using C = cpx<R>;
    C s02 = cadd(a0, a2), d02 = csub(a0, a2);
    C s13 = cadd(a1, a3), d13 = mul_mi<C, INV>(csub(a1, a3));
    a0 = cadd(s02, s13);
    a2 = csub(s02, s13);
    a1 = cadd(d02, d13);
    a3 = csub(d02, d13);
}
// the same with a2 = a3 = 0 on entry
template <typename R, bool INV>
__device__ __forceinline__ void dft4_half(cpx<R> &a0, cpx<R> &a1, cpx<R> &a2, cpx<R> &a3) {
    using C = cpx<R>;
    const C s = a0, t = a1, ti = mul_mi<C, INV>(a1);
    a0 = cadd(s, t);
    a2 = csub(s, t);
    a1 = cadd(s, ti);
    a3 = csub(s, ti);
}

template <typename R, int RAD, bool INV, int NZ = RAD>
__device__ __forceinline__ void dft(cpx<R> (&v)[RAD]);

// Odd prime: with a_j = x_j + x_(p-j) and b_j = x_j - x_(p-j), X_q and X_(p-q) are
// (x_0 + sum_j cos(2 pi jq/p) a_j) -+ i sum_j sin(2 pi jq/p) b_j: 2 (p-1)^2 / 2 real
// multiply-adds by constants in place of (p-1)^2 complex ones by table entries.
template <typename R, int P, bool INV, int NZ>
__device__ __forceinline__ void dft_prime(cpx<R> (&v)[P]) {
    using C = cpx<R>;
    constexpr int Hh = (P - 1) / 2;
    C a[Hh + 1], b[Hh + 1];
    static_for<1, Hh + 1>([&](auto J) {
        constexpr int j = J;
        if constexpr (P - j >= NZ) { a[j] = v[j]; b[j] = v[j]; }
        else { a[j] = cadd(v[j], v[P - j]); b[j] = csub(v[j], v[P - j]); }
    });
    const C x0 = v[0];
    C mid = x0, dif = x0;  // radix 5
    if constexpr (P == 5) {
        // (c1 + c2) / 2 = -1/4, (c1 - c2) / 2 = sqrt(5) / 4: equal inputs cancel exactly, where
        // rounded c1 and c2 leave 1e-8 of them in every output
        const C t = cadd(a[1], a[2]);
        v[0] = cadd(x0, t);
        mid = mk<C>(x0.x - R(0.25) * t.x, x0.y - R(0.25) * t.y);
        dif = csub(a[1], a[2]);
    } else {
        C sum = x0;
        static_for<1, Hh + 1>([&](auto J) { sum = cadd(sum, a[J]); });
        v[0] = sum;
    }
    static_for<1, Hh + 1>([&](auto Q) {
        constexpr int q = Q;
        C A = x0, Bs = czero<C>();
        if constexpr (P == 5) {
            constexpr R k = (R)(q == 1 ? 0.55901699437494742410 : -0.55901699437494742410);
            A = mk<C>(mid.x + k * dif.x, mid.y + k * dif.y);
        }
        static_for<1, Hh + 1>([&](auto J) {
            constexpr int j = J;
            constexpr R c = (R)Root<(j * q) % P, P>::c, s = (R)Root<(j * q) % P, P>::s;
            if constexpr (P != 5) {
                A.x += c * a[j].x;
                A.y += c * a[j].y;
            }
            if constexpr (j == 1) { Bs.x = s * b[j].x; Bs.y = s * b[j].y; }
            else { Bs.x += s * b[j].x; Bs.y += s * b[j].y; }
        });
        const C t = mul_mi<C, INV>(Bs);  // forward: -i B
        v[q] = cadd(A, t);
        v[P - q] = csub(A, t);
    });
}

// RAD = R1 R2: DFTs of length R1 over n1 (n = R2 n1 + n2), twiddles W_RAD^(n2 k1), DFTs of
// length R2 over n2; X[k1 + R1 k2].
template <typename R, int R1, int R2, bool INV, int NZ>
__device__ __forceinline__ void dft_comp(cpx<R> (&v)[R1 * R2]) {
    using C = cpx<R>;
    constexpr int RAD = R1 * R2;
    constexpr int NZ1 = NZ >= RAD ? R1 : (R1 + 1) / 2;
    static_assert(NZ >= RAD || NZ <= R2 * NZ1, "half of the inputs at most");
    static_for<0, R2>([&](auto N2) {
        constexpr int n2 = N2;
        C t[R1];
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) t[n1] = v[R2 * n1 + n2];
        dft<R, R1, INV, NZ1>(t);
        static_for<0, R1>([&](auto K1) {
            constexpr int k1 = K1;
            v[R2 * k1 + n2] = rot<R, INV, (n2 * k1) % RAD, RAD>(t[k1]);
        });
    });
    C o[RAD];
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
        C t[R2];
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) t[n2] = v[R2 * k1 + n2];
        dft<R, R2, INV>(t);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) o[k1 + R1 * k2] = t[k2];
    }
#pragma unroll
    for (int i = 0; i < RAD; ++i) v[i] = o[i];
}

template <typename R, int RAD, bool INV, int NZ>
__device__ __forceinline__ void dft(cpx<R> (&v)[RAD]) {
    using C = cpx<R>;
    if constexpr (RAD == 1) {
    } else if constexpr (RAD == 2) {
        if constexpr (NZ == 1) {
            v[1] = v[0];
        } else {
            const C a = v[0], b = v[1];
            v[0] = cadd(a, b);
            v[1] = csub(a, b);
        }
    } else if constexpr (RAD == 4) {
        if constexpr (NZ <= 2) dft4_half<R, INV>(v[0], v[1], v[2], v[3]);
        else dft4<R, INV>(v[0], v[1], v[2], v[3]);
    } else if constexpr (RAD == 3 || RAD == 5 || RAD == 7 || RAD == 11 || RAD == 13 || RAD == 17) {
        dft_prime<R, RAD, INV, NZ>(v);
    } else if constexpr (RAD == 6) {
        dft_comp<R, 2, 3, INV, NZ>(v);
    } else if constexpr (RAD == 8) {
        dft_comp<R, 4, 2, INV, NZ>(v);
    } else if constexpr (RAD == 9) {
        dft_comp<R, 3, 3, INV, NZ>(v);
    } else if constexpr (RAD == 10) {
        dft_comp<R, 2, 5, INV, NZ>(v);
    } else if constexpr (RAD == 12) {
        dft_comp<R, 4, 3, INV, NZ>(v);
    } else if constexpr (RAD == 14) {
        dft_comp<R, 2, 7, INV, NZ>(v);
    } else if constexpr (RAD == 15) {
        dft_comp<R, 3, 5, INV, NZ>(v);
    } else {
        static_assert(RAD == 16, "codelet radix");
        dft_comp<R, 4, 4, INV, NZ>(v);
    }
}

// ---------------------------------------------------------------------------
// Stages.  MID: shared memory to shared memory with twiddles; the first stage has none.

// the inputs (outputs) of butterfly j are j + r M: with at most `valid` of them in use, the
// ones from r = (RAD + 1) / 2 on are absent when valid <= M (RAD + 1) / 2
__device__ __forceinline__ bool half_enough(const FftStage &s, int valid) { return valid <= s.M * ((s.rad + 1) / 2); }

// A sink with a member pre(n, b) has it called for every output before the inputs are
// read: its loads are in flight during the butterfly.  The result is handed back to it.
struct NoPre {};
template <class Out, class = void> struct PreOf {
    using T = NoPre;
    static __device__ __forceinline__ T load(const Out &, int, int) { return T{}; }
    template <class C> static __device__ __forceinline__ void store(const Out &out, int n, int b, C x, T) { out(n, b, x); }
};
template <class Out> struct PreOf<Out, decltype((void)&Out::pre)> {
    using T = decltype(std::declval<const Out &>().pre(0, 0));
    static __device__ __forceinline__ T load(const Out &out, int n, int b) { return out.pre(n, b); }
    template <class C> static __device__ __forceinline__ void store(const Out &out, int n, int b, C x, T t) { out(n, b, x, t); }
};

template <typename R, int RAD, bool INV, bool TW, bool HIN, bool HOUT, class In, class Out>
__device__ __forceinline__ void fft_stage(const FftStage &s, int B, unsigned mB, const cpx<R> *tw, const In &in,
                                          const Out &out) {
    using C = cpx<R>;
    constexpr int NZ = HIN ? (RAD + 1) / 2 : RAD;
    constexpr int NO = HOUT ? (RAD + 1) / 2 : RAD;
    const int total = s.M * B;
    for (int it = threadIdx.x; it < total; it += blockDim.x) {
        const int j = fast_div(it, mB), b = it - j * B;
        const int k = TW ? j - fast_div(j, s.mNs) * s.Ns : 0;
        const int d0 = (j - k) * RAD + k;
        typename PreOf<Out>::T t[RAD];
#pragma unroll
        for (int r = 0; r < NO; ++r) t[r] = PreOf<Out>::load(out, d0 + r * s.Ns, b);
        C v[RAD];
#pragma unroll
        for (int r = 0; r < RAD; ++r) v[r] = r < NZ ? in(j + r * s.M, b) : czero<C>();
        if constexpr (TW) {
            const int e = k * s.tws;
#pragma unroll
            for (int r = 1; r < RAD; ++r) v[r] = INV ? cmulc(v[r], tw[r * e]) : cmul(v[r], tw[r * e]);
        }
        dft<R, RAD, INV, NZ>(v);
#pragma unroll
        for (int r = 0; r < NO; ++r) PreOf<Out>::store(out, d0 + r * s.Ns, b, v[r], t[r]);
    }
}

template <typename R, bool INV, bool TW, bool HIN, bool HOUT, class In, class Out>
__device__ __forceinline__ void fft_stage_any(const FftStage &s, int B, unsigned mB, const cpx<R> *tw, const In &in,
                                              const Out &out) {
    switch (s.rad) {
#define GJ_RADIX(RAD) \
    case RAD: fft_stage<R, RAD, INV, TW, HIN, HOUT>(s, B, mB, tw, in, out); break;
        GJ_RADIX(1) GJ_RADIX(2) GJ_RADIX(3) GJ_RADIX(4) GJ_RADIX(5) GJ_RADIX(6) GJ_RADIX(7) GJ_RADIX(8) GJ_RADIX(9)
        GJ_RADIX(10) GJ_RADIX(11) GJ_RADIX(12) GJ_RADIX(13) GJ_RADIX(14) GJ_RADIX(15) GJ_RADIX(16) GJ_RADIX(17)
#undef GJ_RADIX
        default: break;
    }
}

// The whole transform: in(j, b) supplies input j < valid of line b (others are zero; in is
// called for every j of a stage, so it returns zero beyond valid), out(n, b, x) receives
// output n (at least those below `need`; it drops the rest).  bufA and bufB hold N pitch
// values each; every thread of the CTA calls.  tw (shared) may still be loading on
// entry: the first stage does not read it, and the barrier behind that stage covers it.
// The caller separates this call's use of bufA and bufB from others' with barriers:
// on return bufB may still be read by other threads when the plan has three stages
// (bufA when it has two).  Plans have at least two stages.
template <typename R, bool INV, bool HIN_OK, bool HOUT_OK, class In, class Out>
__device__ __forceinline__ void fft_run(const FftPlanDev &plan, int B, unsigned mB, int pitch, cpx<R> *bufA,
                                        cpx<R> *bufB, const cpx<R> *tw, int valid, int need, const In &in,
                                        const Out &out) {
    using C = cpx<R>;
    const int last = plan.nst - 1;
    C *src = bufA, *dst = bufB;
    {
        auto put = [&](int n, int b, C x) { bufA[n * pitch + b] = x; };
        if (HIN_OK && half_enough(plan.st[0], valid)) fft_stage_any<R, INV, false, HIN_OK, false>(plan.st[0], B, mB, tw, in, put);
        else fft_stage_any<R, INV, false, false, false>(plan.st[0], B, mB, tw, in, put);
    }
    __syncthreads();
    for (int s = 1; s < last; ++s) {
        auto get = [&](int j, int b) { return src[j * pitch + b]; };
        auto put = [&](int n, int b, C x) { dst[n * pitch + b] = x; };
        fft_stage_any<R, INV, true, false, false>(plan.st[s], B, mB, tw, get, put);
        __syncthreads();
        C *t = src; src = dst; dst = t;
    }
    auto get = [&](int j, int b) { return src[j * pitch + b]; };
    if (HOUT_OK && half_enough(plan.st[last], need)) fft_stage_any<R, INV, true, false, HOUT_OK>(plan.st[last], B, mB, tw, get, out);
    else fft_stage_any<R, INV, true, false, false>(plan.st[last], B, mB, tw, get, out);
}

}  // namespace gj
