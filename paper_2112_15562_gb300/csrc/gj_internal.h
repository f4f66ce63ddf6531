// Host-side internals shared by the translation units of the library.
#pragma once
#include <cuda_runtime.h>

#include <mutex>
#include <string>
#include <vector>

#include "../../include/gj.h"
#include "fft.cuh"

namespace gj { struct gj_setup_scratch_impl; }

struct gj_op {
    // geometry
    int sx, sy, nx, ny, nz, off_x, off_y;
    double dx, dy, station_z;
    std::vector<double> z_edges;
    gj_field field;
    gj_mag mag;
    gj_precision prec;
    // padded sizes and plans
    int Nx, Ny, ncol;
    gj::FftPlanDev px, py;
    // device memory (op precision unless noted)
    void *twx = nullptr, *twy = nullptr;  // twiddles W_N^k
    void *spec = nullptr;                 // [nz][Ny][ncol] complex
    void *Z = nullptr, *Y = nullptr, *W = nullptr, *V = nullptr;
    size_t spec_bytes = 0, ws_bytes = 0;
    // launch shapes
    int P_row = 8, C_col = 8, L_grp = 4;
    bool rows_tuned = false, cols_tuned = false, layers_tuned = false;  // set by gj_op_tune: use them as they are
    int radix_order = 0;
    int gen_slots = 1;  // general kernels: layer groups that Y has room for
    // fast path (FP32, N_x = 512 and N_y = 512 or 256, at most N/2 prisms and stations
    // per direction): transposed spectra and intermediates, layer-sum partials and counters
    bool fast = false;
    bool real_spec = false;  // fast path: the table is even in both offsets, its spectrum is real
    void *P = nullptr;     // [ncol][slots][Ny] complex
    int *cnt = nullptr;    // [ncol] arrival counters (every path)
    int *err = nullptr;    // device error word (bounded waits)
    void *twtab = nullptr; // the column kernels' twiddle table (FP32, TabTw or Tab1024 layout)
    // N_y = 1024 (FP32, at most 512 prisms and stations per column): warp-FFT column
    // kernels with the general row kernels writing and reading transposed Z, W, V;
    // spectra, partials, counters and the error word as on the fast path
    bool fast1024 = false;
    bool rows1024 = false;  // with the warp-FFT row kernels: N_x = 1024 and at most 512 values a line
    // per-layer spectrum recomputation (GJ_SETUP_RECOMPUTE_SPECTRA): `spec` holds one
    // layer, rebuilt from the closed forms before each use
    bool recompute = false;
    bool even_table = false;  // the table is even in both offsets: its spectrum is real and even
    bool even_rows = false;   // the build of an even table transforms half the rows, and columns in pairs
    gj::gj_setup_scratch_impl *scratch = nullptr;
    int slots = 0;
    int col_grid = 0;      // CTAs of the persistent column kernels
};

namespace gj {

void set_error(const std::string &msg);
gj_status cuda_fail(cudaError_t e, const char *what);
bool plan_size(int N, FftPlanDev &plan, int order = 0);  // false if N has an unsupported factor
int  autotune_size(int minN);               // smallest 7-smooth N >= minN
size_t elem_bytes(gj_precision p);           // bytes of one real value
void make_twiddles(int N, std::vector<double> &re, std::vector<double> &im);

// Stream-ordered device memory from a pool of the library's own, one per device, which keeps
// up to 128 MB between uses and gives the rest back at the next synchronisation (the default
// pool gives everything back, and an allocation then costs some 100 us; so does cudaMalloc).
// Any stream or thread may call; free with cudaFreeAsync in the stream, or with cudaFree once
// the kernels on it are done: unlike cudaMalloc's memory, it is given back without waiting.
cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t st);

// Held while the library captures a graph, and by sync_device: synchronising a device fails, and
// breaks the capture, while a stream of it is being captured, from whichever thread.
std::mutex &capture_mutex();
// Waits for the current device (an error, for instance of a capture by somebody else, is
// returned and not left behind for the next check).
cudaError_t sync_device();

// Makes `dev` the current device until the end of the scope.
class DeviceScope {
    int before = 0;
    bool other = false;
public:
    explicit DeviceScope(int dev) {
        other = cudaGetDevice(&before) == cudaSuccess && before != dev && cudaSetDevice(dev) == cudaSuccess;
    }
    ~DeviceScope() {
        if (other) cudaSetDevice(before);
    }
    DeviceScope(const DeviceScope &) = delete;
    DeviceScope &operator=(const DeviceScope &) = delete;
};

template <typename R> struct OpView;
template <typename R> OpView<R> view_of(const gj_op *op);

// fast-path helpers (setup.cu)
bool fast_eligible(const gj_op *op);
int fast_col_items(int Ny, int nz);  // items per column of the fast column kernels
// partial slots per column for persistent column kernels of `warps` warps in total
int fast_slots(int nfield, int ncol, int items_per_col, long long warps);
bool fast1024_eligible(const gj_op *op);

// recompute mode (setup.cu): the corner lattice of every depth plane, once per product (or, where
// that is large, each layer's two planes with the layer); then layer r's table and its FP64 row
// transforms, and where those are
void recompute_begin(const gj_op *op, cudaStream_t st);
void recompute_rows(const gj_op *op, int r, cudaStream_t st);
const double2 *recompute_rows_out(const gj_op *op);
const double2 *recompute_twy64(const gj_op *op);

// enqueue products (matvec.cu)
gj_status forward_enqueue(const gj_op *op, const void *m, void *d, cudaStream_t s);
gj_status adjoint_enqueue(const gj_op *op, const void *r, void *g, cudaStream_t s);

}  // namespace gj

#define GJ_CUDA(call)                                                  \
    do {                                                               \
        cudaError_t _e = (call);                                       \
        if (_e != cudaSuccess) return gj::cuda_fail(_e, #call);        \
    } while (0)
