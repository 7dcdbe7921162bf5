// fsl_noalloc.cu -- bubble labelling for callers that cannot allocate device
// memory.
//
// Some callers cannot call cudaMalloc: latency-critical loops in which an
// allocation may synchronise the device, deployments that hand all device
// memory to their own pool up front, and host frameworks that own the device
// memory budget and forbid libraries to allocate behind their back.
// fsl_label_bubbles_static gives them the library's
// bubble labelling (connected components of gas + interface cells under the
// 18-neighbourhood, label = minimum linear index, the same labels that
// fsl_fields(FSL_F_ID) reports after fsl_init_geometry) using only the
// caller's input and output buffers plus a fixed scratch array compiled into
// the library.
//
// The scratch is a file-scope static __device__ array of FSL_STATIC_MAX_CELLS
// int32 labels (8 MiB); every GPU that loads the library holds it until the
// process exits.  In host code the array's name is only a host-side stand-in,
// not a device address, so its device address is looked up once per device
// with cudaGetSymbolAddress (with that device current) and cached.
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "../../include/fsl.h"

#define FSL_STATIC_MAX_CELLS (1 << 21)
#define FSL_STATIC_MAX_DEVICES 64

namespace {

static __device__ __align__(256) int g_label_scratch[FSL_STATIC_MAX_CELLS];

// device address of the scratch per device ordinal, looked up once per device
// (under the mutex; later calls read the atomic slot without locking)
std::atomic<void*> g_scratch_ptr[FSL_STATIC_MAX_DEVICES];
std::mutex g_scratch_mutex;

__host__ __device__ inline bool is_bubble_cell(uint8_t f) {
    const uint8_t t = (uint8_t)(f & 7);
    return t == FSL_GAS || t == FSL_INTERFACE;
}

__device__ inline int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// Three kernels: runs, unions, labels.  All are bound by the latency of
// dependent L2 accesses, not by their 9 B a cell, so the work is in shortening
// the chains:
//   - a cell starts on the first cell of its run along x inside its warp (one
//     ballot) instead of on itself, which leaves about one root per warp and
//     run and makes all unions along x inside a run unnecessary;
//   - a cell unites with a neighbour row only where its left neighbour does not
//     already do so (both left neighbours present means the same two runs);
//   - the walk to a root halves the path behind it, and roots are hooked by
//     compare-and-swap, so every cell points at an ancestor at all times.
// 128^3 foam: 214 us with one union per cell and direction over unshortened
// paths, 69 us in this form (host call included).

__global__ void __launch_bounds__(256) k_static_init(const uint8_t* __restrict__ flags, int n, int nx,
                                                     int* __restrict__ lab) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool fg = i < n && is_bubble_cell(flags[i]);
    const unsigned m = __ballot_sync(0xffffffffu, fg);
    if (i >= n) return;
    if (!fg) { lab[i] = -1; return; }
    // first cell of the run: after the last gap below this lane, not before the
    // warp's first cell nor the row's
    const int lane = threadIdx.x & 31;
    const unsigned gaps = ~m & ((1u << lane) - 1u);
    const int back = gaps ? lane - (32 - __clz((int)gaps)) : lane;
    lab[i] = i - min(back, i % nx);
}

// Root of a, halving the path: a cell's parent only ever changes to an ancestor
// (from itself to a smaller root, or to its grandparent), so a store, however
// late, keeps the cell in its tree, and a load, however old (a line of the L1
// cache may be), names an ancestor.  (Loads past L1: 80 us against 66 us on the
// 128^3 foam.)
__device__ inline int static_root_halving(int* L, int a) {
    for (int it = 0; it < FSL_STATIC_MAX_CELLS; ++it) {
        const int p = L[a];
        if (p == a) return a;
        const int gp = L[p];
        if (gp == p) return p;
        L[a] = gp;
        a = gp;
    }
    return a;
}

__device__ inline int static_root(const int* L, int a) {
    // labels only decrease along a chain, so this walk ends within a steps
    for (int it = 0; it < FSL_STATIC_MAX_CELLS; ++it) {
        const int p = L[a];
        if (p == a) return a;
        a = p;
    }
    return a;
}

// Union: hook the larger root under the smaller while it is still a root.  A swap
// that fails goes on from the parent it met, which is smaller than a: every turn
// lowers a + b, whatever the loads of the walks have seen, so the union is made
// within the 2 n turns of the cap.
__device__ inline void static_unite(int* L, int a, int b) {
    for (int it = 0; it < 2 * FSL_STATIC_MAX_CELLS; ++it) {
        a = static_root_halving(L, a);
        b = static_root_halving(L, b);
        if (a == b) return;
        if (a < b) { const int t = a; a = b; b = t; }
        const int met = atomicCAS(&L[a], a, b);
        if (met == a) return;
        a = met;
    }
}

__global__ void __launch_bounds__(256) k_static_hook(const uint8_t* __restrict__ flags, int nx, int ny, int nz,
                                                     int* __restrict__ lab) {
    const int n = nx * ny * nz;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || !is_bubble_cell(flags[i])) return;
    const int x = i % nx, y = (i / nx) % ny, z = i / (nx * ny);
    const int row = i - x, xl = wrap1(x - 1, nx), xr = wrap1(x + 1, nx);
    const int yp = nx * wrap1(y + 1, ny), ym = nx * wrap1(y - 1, ny), y0 = nx * y;
    const int zp = nx * ny * wrap1(z + 1, nz), z0 = nx * ny * z;
    // the rows of the nine neighbour pairs' second cells: +y, +z (with their x
    // neighbours), +y+z and -y+z (straight only); every type loaded up front
    const int ry = z0 + yp, rz = zp + y0, rd = zp + yp, ru = zp + ym;
    const bool left_w = is_bubble_cell(flags[row + xl]), right = is_bubble_cell(flags[row + xr]);
    const bool yl = is_bubble_cell(flags[ry + xl]), yc = is_bubble_cell(flags[ry + x]), yr = is_bubble_cell(flags[ry + xr]);
    const bool zl = is_bubble_cell(flags[rz + xl]), zc = is_bubble_cell(flags[rz + x]), zr = is_bubble_cell(flags[rz + xr]);
    const bool dl = is_bubble_cell(flags[rd + xl]), dc = is_bubble_cell(flags[rd + x]);
    const bool ul = is_bubble_cell(flags[ru + xl]), uc = is_bubble_cell(flags[ru + x]);
    // along x: only where a run goes on past its warp or the row's end
    if (right && lab[row + xr] != lab[i] && (((threadIdx.x & 31) == 31) || xr != x + 1))
        static_unite(lab, i, row + xr);
    // straight neighbour: the left cells make the same union when both are there
    // (never past the row's start, or a full row would leave it to itself)
    const bool left = left_w && x > 0;
    if (yc && !(left && yl)) static_unite(lab, i, ry + x);
    if (zc && !(left && zl)) static_unite(lab, i, rz + x);
    if (dc && !(left && dl)) static_unite(lab, i, rd + x);
    if (uc && !(left && ul)) static_unite(lab, i, ru + x);
    // diagonal neighbour: only where no straight union leads there (the cell
    // below it, or this cell's neighbour on that side, would)
    if (yr && !yc && !right) static_unite(lab, i, ry + xr);
    if (yl && !yc && !left_w) static_unite(lab, i, ry + xl);
    if (zr && !zc && !right) static_unite(lab, i, rz + xr);
    if (zl && !zc && !left_w) static_unite(lab, i, rz + xl);
}

__global__ void __launch_bounds__(256) k_static_out(const uint8_t* __restrict__ flags, int n,
                                                    const int* __restrict__ lab, int64_t* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = is_bubble_cell(flags[i]) ? (int64_t)static_root(lab, i) : -1;
}

}  // namespace

extern "C" fsl_status fsl_label_bubbles_static(const uint8_t* flags, int32_t nx, int32_t ny, int32_t nz,
                                               int64_t* labels, void* cuda_stream) {
    if (!flags || !labels || nx <= 0 || ny <= 0 || nz <= 0) return FSL_ERR_ARG;
    const long long n = (long long)nx * ny * nz;
    if (n > FSL_STATIC_MAX_CELLS) return FSL_ERR_ARG;   // larger lattices need fsl_create
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= FSL_STATIC_MAX_DEVICES) return FSL_ERR_CUDA;
    void* lab_ptr = g_scratch_ptr[dev].load(std::memory_order_acquire);
    if (!lab_ptr) {
        // first call on this device: look up the device address of the scratch
        std::lock_guard<std::mutex> lock(g_scratch_mutex);
        lab_ptr = g_scratch_ptr[dev].load(std::memory_order_relaxed);
        if (!lab_ptr) {
            if (cudaGetSymbolAddress(&lab_ptr, g_label_scratch) != cudaSuccess || !lab_ptr) return FSL_ERR_CUDA;
            g_scratch_ptr[dev].store(lab_ptr, std::memory_order_release);
        }
    }
    int* lab = (int*)lab_ptr;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int nb = (int)((n + 255) / 256);
    k_static_init<<<nb, 256, 0, s>>>(flags, (int)n, nx, lab);
    k_static_hook<<<nb, 256, 0, s>>>(flags, nx, ny, nz, lab);
    k_static_out<<<nb, 256, 0, s>>>(flags, (int)n, lab, labels);
    return cudaGetLastError() == cudaSuccess ? FSL_OK : FSL_ERR_CUDA;
}
