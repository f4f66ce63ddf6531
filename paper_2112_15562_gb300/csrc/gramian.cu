// The Gramian coupling term (Eq. Gramian) and its ascent directions (RRCG:2-3).
#include <algorithm>
#include <mutex>
#include <string>

#include "view.cuh"

namespace gj {

// Both passes stream the vectors: 2 n R in, then 2 n R in (from L2 where they fit) and 2 n R
// out.  A thread keeps eight 16-byte loads in flight, the products of sixteen elements at most
// go into an FP32 partial sum before FP64 takes it, and the sums over blocks happen inside
// the two launches (every block of the second sums the first's partials, the last block to
// finish sums the second's), where two one-block launches of 4 to 6 us each stood before.
// 2.6 M values FP32, us: partial sums 13.7 + 6.4 and directions 16.4 + 4.5 before.
constexpr int kGramBlocks = 304;    // two blocks an SM
constexpr int kGramThreads = 256;
constexpr int kGramChunk = 16;      // elements of a thread between FP64 additions
// scratch: 3 partial sums a block, 1 residual sum a block, the ticket
constexpr int kGramDoubles = 4 * kGramBlocks + 1;

template <typename R> struct Vec16;
template <> struct Vec16<float> { using T = float4; static constexpr int N = 4; };
template <> struct Vec16<double> { using T = double2; static constexpr int N = 2; };

// Calls each(i, x, y) for this thread's elements i, a vector of them (VEC: 16-byte loads, for
// aligned vectors) or one at a time, and done() after each chunk of at most kGramChunk.  The
// directions may be written over the vectors (a thread reads an element before it writes it, and
// no other thread does either), so nothing here promises that they do not overlap.
template <typename R, bool VEC, class Each, class Done>
__device__ __forceinline__ void gram_chunks(int64_t n, const R *m1, const R *m2, Each each, Done done) {
    const int64_t thread = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, threads = (int64_t)gridDim.x * blockDim.x;
    if constexpr (VEC) {
        using V = typename Vec16<R>::T;
        constexpr int N = Vec16<R>::N, U = 4;  // vectors of each input in flight (N U <= kGramChunk elements)
        const int64_t nv = n / N;
        const V *a = reinterpret_cast<const V *>(m1), *b = reinterpret_cast<const V *>(m2);
        for (int64_t v0 = thread; v0 < nv; v0 += U * threads) {
            V x[U], y[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t v = v0 + u * threads;
                if (v < nv) { x[u] = a[v]; y[u] = b[v]; }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t v = v0 + u * threads;
                if (v < nv) each(v * N, reinterpret_cast<const R(&)[N]>(x[u]), reinterpret_cast<const R(&)[N]>(y[u]));
            }
            done();
        }
        for (int64_t i = nv * N + thread; i < n; i += threads) {  // the last n % N elements
            const R x[1] = {m1[i]}, y[1] = {m2[i]};
            each(i, x, y);
            done();
        }
    } else {
        for (int64_t i0 = thread; i0 < n; i0 += kGramChunk * threads) {
            R x[kGramChunk], y[kGramChunk];
#pragma unroll
            for (int u = 0; u < kGramChunk; ++u) {
                const int64_t i = i0 + u * threads;
                if (i < n) { x[u] = m1[i]; y[u] = m2[i]; }
            }
#pragma unroll
            for (int u = 0; u < kGramChunk; ++u) {
                const int64_t i = i0 + u * threads;
                const R xu[1] = {x[u]}, yu[1] = {y[u]};
                if (i < n) each(i, xu, yu);
            }
            done();
        }
    }
}

// (m1,m1), (m2,m2), (m1,m2): part[c nb + block].  Also zeroes the second pass's ticket.
template <typename R, bool VEC>
__global__ void __launch_bounds__(kGramThreads) k_gram_dots(int64_t n, const R *m1, const R *m2, double *part,
                                                            unsigned *ticket) {
    __shared__ double red[32];
    pdl_go();
    pdl_wait();
    double s11 = 0, s22 = 0, s12 = 0;
    R a11 = 0, a22 = 0, a12 = 0;
    gram_chunks<R, VEC>(
        n, m1, m2,
        [&](int64_t, const auto &x, const auto &y) {
            constexpr int N = (int)(sizeof(x) / sizeof(R));
#pragma unroll
            for (int k = 0; k < N; ++k) { a11 += x[k] * x[k]; a22 += y[k] * y[k]; a12 += x[k] * y[k]; }
        },
        [&]() {
            s11 += (double)a11; s22 += (double)a22; s12 += (double)a12;
            a11 = a22 = a12 = 0;
        });
    s11 = block_sum(s11, red);
    s22 = block_sum(s22, red);
    s12 = block_sum(s12, red);
    if (threadIdx.x == 0) {
        const int nb = gridDim.x;
        part[blockIdx.x] = s11;
        part[nb + blockIdx.x] = s22;
        part[2 * nb + blockIdx.x] = s12;
        if (blockIdx.x == 0) *ticket = 0;
    }
}

// Ascent directions, and ||m2 - (a12/a11) m1||^2, which gives
// S = a11 ||m2 - (a12/a11) m1||^2 without the cancellation of a11 a22 - a12^2.
template <typename R, bool VEC>
__global__ void __launch_bounds__(kGramThreads) k_gram_dirs(int64_t n, const R *m1, const R *m2, const double *part,
                                                            R *l1, R *l2, double *part2, unsigned *ticket, double *S) {
    __shared__ double red[32], sums[3];
    __shared__ R coef[4];
    __shared__ bool last;
    const int nb = gridDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_wait();
    if (warp < 3) {  // one warp a sum, in a fixed order
        double t = 0.0;
        for (int b = lane; b < nb; b += 32) t += part[warp * nb + b];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) sums[warp] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        coef[0] = (R)sums[0];
        coef[1] = (R)sums[1];
        coef[2] = (R)sums[2];
        coef[3] = sums[0] > 0 ? (R)(sums[2] / sums[0]) : R(0);
    }
    __syncthreads();
    const R c11 = coef[0], c22 = coef[1], c12 = coef[2], ratio = coef[3];
    double s = 0;
    R res = 0;
    gram_chunks<R, VEC>(
        n, m1, m2,
        [&](int64_t i, const auto &x, const auto &y) {
            constexpr int N = (int)(sizeof(x) / sizeof(R));
            R u[N], v[N];
#pragma unroll
            for (int k = 0; k < N; ++k) {
                u[k] = c22 * x[k] - c12 * y[k];
                v[k] = c11 * y[k] - c12 * x[k];
                const R d = y[k] - ratio * x[k];
                res += d * d;
            }
            if constexpr (N > 1) {
                using V = typename Vec16<R>::T;
                if (l1) *reinterpret_cast<V *>(l1 + i) = reinterpret_cast<const V &>(u);
                if (l2) *reinterpret_cast<V *>(l2 + i) = reinterpret_cast<const V &>(v);
            } else {
                if (l1) l1[i] = u[0];
                if (l2) l2[i] = v[0];
            }
        },
        [&]() {
            s += (double)res;
            res = 0;
        });
    s = block_sum(s, red);
    if (threadIdx.x == 0) {
        part2[blockIdx.x] = s;
        __threadfence();
        last = atomicAdd(ticket, 1u) == (unsigned)nb - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double t = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) t += __ldcg(part2 + b);
    t = block_sum(t, red);
    if (threadIdx.x == 0) *S = sums[0] > 0 ? sums[0] * t : 0.0;
}

// The two launches on a scratch of kGramDoubles doubles.
template <typename R, bool VEC>
static cudaError_t gramian_kernels(int64_t n, const R *m1, const R *m2, double *S, R *l1, R *l2, double *scratch,
                                   cudaStream_t st) {
    const int64_t per = (int64_t)kGramThreads * kGramChunk;
    const int nb = (int)std::min<int64_t>(kGramBlocks, (n + per - 1) / per);
    double *part = scratch, *part2 = scratch + 3 * kGramBlocks;
    unsigned *ticket = reinterpret_cast<unsigned *>(scratch + 4 * kGramBlocks);
    launch_after(k_gram_dots<R, VEC>, dim3(nb), dim3(kGramThreads), 0, st, n, m1, m2, part, ticket);
    launch_after(k_gram_dirs<R, VEC>, dim3(nb), dim3(kGramThreads), 0, st, n, m1, m2, part, l1, l2, part2, ticket, S);
    return cudaGetLastError();
}
template <typename R>
static cudaError_t gramian_on(int64_t n, const void *m1, const void *m2, double *S, void *l1, void *l2,
                              double *scratch, cudaStream_t st) {
    // 16-byte loads and stores where every vector starts on 16 bytes
    const uintptr_t at = (uintptr_t)m1 | (uintptr_t)m2 | (uintptr_t)l1 | (uintptr_t)l2;
    return (at & 15) == 0 ? gramian_kernels<R, true>(n, (const R *)m1, (const R *)m2, S, (R *)l1, (R *)l2, scratch, st)
                          : gramian_kernels<R, false>(n, (const R *)m1, (const R *)m2, S, (R *)l1, (R *)l2, scratch, st);
}

// Under stream capture the default pool serves: the block becomes a node of the graph.
static cudaError_t scratch_take(double **p, size_t doubles, cudaStream_t st) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess) return e;
    if (cap == cudaStreamCaptureStatusNone) return pool_alloc(reinterpret_cast<void **>(p), doubles * sizeof(double), st);
    return cudaMallocAsync(reinterpret_cast<void **>(p), doubles * sizeof(double), st);
}

template <typename R>
static gj_status gramian_launch(int64_t n, const void *m1, const void *m2, double *S, void *l1, void *l2,
                                cudaStream_t st) {
    double *scratch = nullptr;
    GJ_CUDA(scratch_take(&scratch, kGramDoubles, st));
    cudaError_t e = gramian_on<R>(n, m1, m2, S, l1, l2, scratch, st);
    cudaFreeAsync(scratch, st);
    if (e != cudaSuccess) return cuda_fail(e, "gramian launch");
    return GJ_OK;
}

}  // namespace gj

// Pearson coefficient of two vectors: means in a first pass, centred sums in a
// second (FP64 accumulation), the ratio in one thread.
namespace gj {
template <typename R>
__global__ void __launch_bounds__(256) k_sums2(int64_t n, const R *a, const R *b, double *part) {
    __shared__ double red[32];
    double sa = 0, sb = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        sa += (double)a[i];
        sb += (double)b[i];
    }
    sa = block_sum(sa, red);
    sb = block_sum(sb, red);
    if (threadIdx.x == 0) { part[2 * blockIdx.x] = sa; part[2 * blockIdx.x + 1] = sb; }
}
template <typename R>
__global__ void __launch_bounds__(256) k_centred3(int64_t n, const R *a, const R *b, const double *part, int nb,
                                                  double *part2) {
    __shared__ double red[32];
    __shared__ double mean[2];
    if (threadIdx.x < 2) {
        double t = 0;
        for (int k = 0; k < nb; ++k) t += part[2 * k + threadIdx.x];
        mean[threadIdx.x] = t / (double)n;
    }
    __syncthreads();
    const double ma = mean[0], mb = mean[1];
    double saa = 0, sbb = 0, sab = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double x = (double)a[i] - ma, y = (double)b[i] - mb;
        saa += x * x; sbb += y * y; sab += x * y;
    }
    saa = block_sum(saa, red);
    sbb = block_sum(sbb, red);
    sab = block_sum(sab, red);
    if (threadIdx.x == 0) { part2[3 * blockIdx.x] = saa; part2[3 * blockIdx.x + 1] = sbb; part2[3 * blockIdx.x + 2] = sab; }
}
__global__ void k_pearson_finish(int nb, const double *part2, double *r) {
    double saa = 0, sbb = 0, sab = 0;
    for (int k = 0; k < nb; ++k) { saa += part2[3 * k]; sbb += part2[3 * k + 1]; sab += part2[3 * k + 2]; }
    const double den = sqrt(saa * sbb);
    *r = den > 0 ? sab / den : 0.0;
}
template <typename R>
static gj_status pearson_launch(int64_t n, const void *a, const void *b, double *r, cudaStream_t st) {
    const int nb = (int)std::min<int64_t>(2 * 152, std::max<int64_t>(1, (n + 255) / 256));
    double *scratch = nullptr;
    GJ_CUDA(scratch_take(&scratch, 5 * (size_t)nb, st));
    k_sums2<R><<<nb, 256, 0, st>>>(n, (const R *)a, (const R *)b, scratch);
    k_centred3<R><<<nb, 256, 0, st>>>(n, (const R *)a, (const R *)b, scratch, nb, scratch + 2 * nb);
    k_pearson_finish<<<1, 1, 0, st>>>(nb, scratch + 2 * nb, r);
    cudaError_t e = cudaGetLastError();
    cudaFreeAsync(scratch, st);
    return e == cudaSuccess ? GJ_OK : cuda_fail(e, "pearson launch");
}
}  // namespace gj

extern "C" gj_status gj_pearson(int64_t n, gj_precision prec, const void *a, const void *b, double *r,
                                gj_stream_t stream) {
    if (n < 1 || !a || !b || !r) { gj::set_error("gj_pearson: bad argument"); return GJ_ERR_ARG; }
    if (prec != GJ_FP64 && prec != GJ_FP32_MIXED) { gj::set_error("gj_pearson: bad precision"); return GJ_ERR_ARG; }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return prec == GJ_FP64 ? gj::pearson_launch<double>(n, a, b, r, st) : gj::pearson_launch<float>(n, a, b, r, st);
}

extern "C" gj_status gj_gramian_value_grad(int64_t n, gj_precision prec, const void *m1, const void *m2,
                                           double *S, void *l1, void *l2, gj_stream_t stream) {
    if (n < 1 || !m1 || !m2 || !S) { gj::set_error("gj_gramian_value_grad: bad argument"); return GJ_ERR_ARG; }
    if (prec != GJ_FP64 && prec != GJ_FP32_MIXED) { gj::set_error("gj_gramian_value_grad: bad precision"); return GJ_ERR_ARG; }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return prec == GJ_FP64 ? gj::gramian_launch<double>(n, m1, m2, S, l1, l2, st)
                           : gj::gramian_launch<float>(n, m1, m2, S, l1, l2, st);
}

// ---------------------------------------------------------------------------
// Allocation-free variant.  The reduction scratch lives in a file-scope device
// array (every GPU that loads the library keeps it until exit) instead of a
// per-call cudaMallocAsync.  Host code never passes the array's name to a kernel
// (on the host it is only a stand-in symbol): its device address is looked up once
// per device with cudaGetSymbolAddress while that device is current.

namespace gj {
namespace {

constexpr int64_t kNoAllocMaxN = 16777216;

constexpr int kMaxDevices = 64;

static __device__ __align__(256) double g_noalloc_scratch[kGramDoubles];

std::mutex g_noalloc_mu;
double *g_noalloc_addr[kMaxDevices] = {};

gj_status noalloc_scratch(double **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "gj_gramian_value_grad_noalloc: cudaGetDevice");
    if (dev < 0 || dev >= kMaxDevices) {
        set_error("gj_gramian_value_grad_noalloc: device index above 63");
        return GJ_ERR_UNSUPPORTED;
    }
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "gj_gramian_value_grad_noalloc: cudaGetSymbolAddress");
        g_noalloc_addr[dev] = static_cast<double *>(p);
    }
    *out = g_noalloc_addr[dev];
    return GJ_OK;
}

template <typename R>
gj_status gramian_launch_noalloc(int64_t n, const void *m1, const void *m2, double *S, void *l1, void *l2,
                                 cudaStream_t st) {
    double *scratch = nullptr;
    gj_status rc = noalloc_scratch(&scratch);
    if (rc != GJ_OK) return rc;
    // every slot that is read is written earlier in the same call: nothing needs clearing
    cudaError_t e = gramian_on<R>(n, m1, m2, S, l1, l2, scratch, st);
    return e == cudaSuccess ? GJ_OK : cuda_fail(e, "gramian (no allocation) launch");
}

}  // namespace
}  // namespace gj

extern "C" gj_status gj_gramian_value_grad_noalloc(int64_t n, gj_precision prec, const void *m1, const void *m2,
                                                   double *S, void *l1, void *l2, gj_stream_t stream) {
    if (n > gj::kNoAllocMaxN) {
        gj::set_error("gj_gramian_value_grad_noalloc: n = " + std::to_string(n) +
                      " exceeds the allocation-free limit of 16777216 elements (use gj_gramian_value_grad)");
        return GJ_ERR_ARG;
    }
    if (n < 1 || !m1 || !m2 || !S) { gj::set_error("gj_gramian_value_grad_noalloc: bad argument"); return GJ_ERR_ARG; }
    if (prec != GJ_FP64 && prec != GJ_FP32_MIXED) {
        gj::set_error("gj_gramian_value_grad_noalloc: bad precision");
        return GJ_ERR_ARG;
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return prec == GJ_FP64 ? gj::gramian_launch_noalloc<double>(n, m1, m2, S, l1, l2, st)
                           : gj::gramian_launch_noalloc<float>(n, m1, m2, S, l1, l2, st);
}
