// Shared device helpers: complex arithmetic, block reductions.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <set>
#include <utility>

namespace gj {

template <typename R> struct CplxOf;
template <> struct CplxOf<float> { using T = float2; };
template <> struct CplxOf<double> { using T = double2; };
template <typename R> using cpx = typename CplxOf<R>::T;

template <typename C> __host__ __device__ __forceinline__ C mk(decltype(C::x) a, decltype(C::x) b) {
    C c; c.x = a; c.y = b; return c;
}
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return mk<C>(a.x + b.x, a.y + b.y); }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return mk<C>(a.x - b.x, a.y - b.y); }
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
// Blackwell paired FP32 arithmetic: one instruction per complex add or subtract
template <> __device__ __forceinline__ float2 cadd<float2>(float2 a, float2 b) { return __fadd2_rn(a, b); }
template <> __device__ __forceinline__ float2 csub<float2>(float2 a, float2 b) {
    return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);  // a - b, exact product by -1
}
#endif
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
    return mk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
template <typename C> __device__ __forceinline__ C cmulc(C a, C b) {
    return mk<C>(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
template <typename C> __device__ __forceinline__ C cconj(C a) { return mk<C>(a.x, -a.y); }
// multiply by -i (forward) or +i (inverse)
template <typename C, bool INV> __device__ __forceinline__ C mul_mi(C a) {
    return INV ? mk<C>(-a.y, a.x) : mk<C>(a.y, -a.x);
}
template <typename C> __device__ __forceinline__ C czero() { return mk<C>(0, 0); }

// A root of unity's real or imaginary part as a constant of a transform.  In FP32 cos(pi/8) is
// rounded up, to 0.53 units in the last place instead of 0.47 down: sqrt(1/2) and cos(pi/8) both
// round down, so that every 16-point DFT shrank its values by 1.1e-8 and a product by 1.1e-7
// (N = 256), 1.3e-7 (512) or 1.7e-7 (1024), most of its error; now by less than 1e-8.
template <typename R> __host__ __device__ constexpr R root_part(double x) { return (R)x; }
template <> __host__ __device__ constexpr float root_part<float>(double x) {
    constexpr double c8 = 0.92387953251128675613;
    const double d = (x < 0 ? -x : x) - c8;
    if (d < 1e-12 && d > -1e-12) return x < 0 ? -0.92387956380844f : 0.92387956380844f;
    return (float)x;
}

// Sum of `v` over the block; every thread gets the result.  `scratch` holds
// at least 32 doubles.  All threads of the block must call it.
__device__ __forceinline__ double block_sum(double v, double *scratch) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    double t = (threadIdx.x < nw) ? scratch[threadIdx.x] : 0.0;
    if (warp == 0) {
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) scratch[0] = t;
    }
    __syncthreads();
    double r = scratch[0];
    __syncthreads();
    return r;
}

// Sums K values over the 32 lanes of a warp together: at the first steps half of the lanes
// hand over half of the values, so that four sums take six FP64 additions a lane and not
// twenty (the FP64 units do two a cycle and SM: the solver's row passes spent up to 40 % of
// their time there).  On return lane l holds the sum of value (l >> 4) of two, or of
// 2 (l >> 4) + ((l >> 3) & 1) of four.
__device__ __forceinline__ double warp_sums2(double v0, double v1) {
    const bool up = threadIdx.x & 16;
    double t = (up ? v1 : v0) + __shfl_xor_sync(0xffffffffu, up ? v0 : v1, 16);
    for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}
__device__ __forceinline__ double warp_sums4(double v0, double v1, double v2, double v3) {
    const bool up = threadIdx.x & 16, up8 = threadIdx.x & 8;
    const double a = (up ? v2 : v0) + __shfl_xor_sync(0xffffffffu, up ? v0 : v2, 16);
    const double b = (up ? v3 : v1) + __shfl_xor_sync(0xffffffffu, up ? v1 : v3, 16);
    double t = (up8 ? b : a) + __shfl_xor_sync(0xffffffffu, up8 ? a : b, 8);
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// Adds per-thread partials acc[0..K) into out[0..K) (one double atomic per
// block per entry).  All K sums share one pass: warp sums, one barrier, and
// the first warp finishes (whose `out` counts).  `scratch` holds at least 4 * warps doubles.
// All threads must call it.
template <int K, typename A>
__device__ __forceinline__ void block_accumulate(const A *acc, double *out, double *scratch) {
    static_assert(K >= 1 && K <= 4, "one to four sums");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    double t;
    if constexpr (K == 1) {
        t = (double)acc[0];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        __syncthreads();  // scratch may still be in use by an earlier call
        if (lane == 0) scratch[warp] = t;
        __syncthreads();
        if (warp == 0) {
            t = lane < nw ? scratch[lane] : 0.0;
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0 && out) atomicAdd(out, t);
        }
        return;
    }
    if constexpr (K == 2) t = warp_sums2((double)acc[0], (double)acc[1]);
    else t = warp_sums4((double)acc[0], (double)acc[1], (double)acc[2], K > 3 ? (double)acc[K - 1] : 0.0);
    __syncthreads();  // scratch may still be in use by an earlier call
    if constexpr (K == 2) {
        if ((lane & 15) == 0) scratch[(lane >> 4) * nw + warp] = t;
    } else {
        if ((lane & 7) == 0) scratch[(lane >> 3) * nw + warp] = t;
    }
    __syncthreads();
    if (warp == 0) {
        if (nw <= 8) {  // few warps: one lane a value (an FP64 addition holds its scheduler for 64 cycles)
            if (lane < K) {
                double s = scratch[lane * nw];
                for (int w = 1; w < nw; ++w) s += scratch[lane * nw + w];
                if (out) atomicAdd(out + lane, s);
            }
            return;
        }
        // sixteen lanes per value
#pragma unroll
        for (int k = 0; k < K; k += 2) {
            const int mine = k + (lane >> 4);
            double s = 0.0;
            if (mine < K)
                for (int w = lane & 15; w < nw; w += 16) s += scratch[mine * nw + w];
            for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if ((lane & 15) == 0 && mine < K && out) atomicAdd(out + mine, s);
        }
    }
}

// ---------------------------------------------------------------------------
// asynchronous global -> shared copies (cp.async), completed per thread by groups

__device__ __forceinline__ uint32_t s_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async(float2 *dst, const float2 *src) { cp_async8(dst, src); }
__device__ __forceinline__ void cp_async(double2 *dst, const double2 *src) { cp_async16(dst, src); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int NPEND>
__device__ __forceinline__ void cp_async_wait() {  // at most NPEND of the newest groups still in flight
    asm volatile("cp.async.wait_group %0;\n" ::"n"(NPEND) : "memory");
}

// ---------------------------------------------------------------------------
// Programmatic dependent launch: a kernel launched with launch_after may start, up to its
// pdl_wait, while the kernel before it in the stream drains (that one allows it with
// pdl_go).  pdl_wait returns when every earlier kernel has completed and its memory is
// visible, because each of them waits for the ones before it; before it a kernel touches
// nothing but data that no launch writes (twiddles).  Both are no-ops otherwise.
__device__ __forceinline__ void pdl_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                const A &...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    // Not in a graph: replayed, such edges cost more than they hide (256x256x40 FP32 iteration
    // 199 -> 207 us, 16x16x8 FP64 102 -> 106 us; in a stream the 251x243x37 adjoint pair went
    // from 52.1 to 47.2 us).
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cfg.numAttrs = cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Allows launches of `f` with any dynamic shared memory up to the device's opt-in
// maximum less the kernel's static shared memory.  The attribute belongs to the
// function, not to a launch, so setting it to the maximum keeps callers with
// different sizes from overriding each other.
// Done once per kernel and device: later calls return at once, so that a product's
// launches cost no attribute queries on the host.
template <typename F>
inline cudaError_t allow_max_smem(F *f) {
    static std::mutex mu;
    static std::set<std::pair<int, const void *>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const std::pair<int, const void *> key{dev, reinterpret_cast<const void *>(f)};
    {
        std::lock_guard<std::mutex> lk(mu);
        if (done.count(key)) return cudaSuccess;
    }
    int optin = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) optin = 48 * 1024;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
    const int dyn = optin - (int)fa.sharedSizeBytes;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn > 0 ? dyn : 0);
    if (e == cudaSuccess) {
        std::lock_guard<std::mutex> lk(mu);
        done.insert(key);
    }
    return e;
}

}  // namespace gj
