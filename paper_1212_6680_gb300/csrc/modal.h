// modal.h -- the SMG V-cycle in the sine eigenvectors of the x-lines (modal.cuh has the kernels).
#pragma once

#include <cuda_runtime.h>

#include "smg_internal.h"

namespace smg {

constexpr int kMaxZLevels = 13;   // nz <= 4096

// The V-cycle of one system on its mode grids, as the kernels read it (T: float or double).
// "Tail" levels are the z-levels lt .. L-1, which one CTA per mode runs in shared memory.
template <class T>
struct ModalArgs {
    int nmode, ny, pitch;      // x-modes, lines, and lines per plane in global memory (ny rounded up to 4)
    int L, lt;                 // z-levels; first tail level
    int P, sum_ny;             // 2D levels and their lines in all
    int npre, npost, coarse_iters;
    int ny_m[kMaxPlaneLevels], line_base[kMaxPlaneLevels];
    int nz[kMaxZLevels];       // planes of each z-level
    int plane_base[kMaxZLevels];
    int cls_base[kMaxZLevels]; // first table of the level in `raw` (tables of one level are contiguous)
    int ncls[kMaxZLevels];     // plane classes of the level
    int sm_u[kMaxZLevels], sm_f[kMaxZLevels];  // shared-memory offsets (elements of T) of the tail levels
    int sm_pitch;              // lines per plane in shared memory
    int sm_tab, sm_zc;         // offsets (elements of T) of the line tables and the plane coefficients
    int sm_tab64, sm_cls;      // offsets (bytes) of the coarsest plane's FP64 table and the class indices
    const T *f[kMaxZLevels];   // right-hand sides and iterates in global memory: [rhs][mode][plane][pitch],
    T *u[kMaxZLevels];         // levels 0 .. lt
    T *fw[kMaxZLevels];        // f, writable (levels 1 .. lt)
    const T *zc;               // [planes of all levels][8]
    const T *raw;              // [tables][sum_ny][16] line coefficients (raw_line_table)
    const double *raw64;       // the coarsest level's table in FP64
    const unsigned char *cls;  // [planes of all levels] plane class within the level
    const double *lam;         // [nmode] eigenvalues of the x-line Laplacian
};

// Line tables of one plane class: 16 values a line (raw_line_table in modal_host.cpp).
constexpr int kRawPerLine = 16;

// Lanes per plane and lines per lane for planes of ny lines.
struct ModalConfig {
    int G, K;
};
ModalConfig modal_config(int ny, bool f64);

// Shared memory the tail kernel may use, and its threads.
constexpr size_t kModalSmem = 227 * 1024 - 2048;

struct ModalPlan {
    bool f64 = false;
    int nx = 0, ny = 0, nz = 0, nb = 0, nh = 0;  // nh: odd modes (ceil(nx / 2))
    int npre = 1, npost = 0, coarse_iters = 1;
    ModalConfig cfg{8, 16};
    size_t smem = 0;              // tail kernel
    int threads = 0;
    int lt = 0, L = 0, pitch = 0;
    ModalArgs<float> a32;         // host copies of the kernel arguments
    ModalArgs<double> a64;
    void *d_args = nullptr;
    void *d_buf = nullptr;        // mode-space vectors
    void *d_tab = nullptr;        // coefficients
    void *d_sin = nullptr;        // transform matrices
    int hp = 0;                   // their padded order
};

// Tables and buffers for nb right-hand sides; 0, or a cudaError_t.
int modal_build(ModalPlan &p, const HostHierarchy &H, bool f64, int nb, int npre, int npost, int coarse_iters);
void modal_free(ModalPlan &p);

// u0 = T f0 for nb right-hand sides, in three parts: f0 (FP64, [rhs][z][y][x]) into mode space, the
// cycle there, and back into u0 (elements of type `type`).  Each adds its kernel launches to
// `launches`.  Asynchronous on st.
cudaError_t modal_transform_in(const ModalPlan &p, int nb, const double *f0, cudaStream_t st, long long &launches);
cudaError_t modal_cycle(const ModalPlan &p, int nb, cudaStream_t st, long long &launches);
cudaError_t modal_transform_out(const ModalPlan &p, int nb, Prec type, void *u0, cudaStream_t st, long long &launches);

// Kernels of one configuration (modal_inst.cu).
template <class T>
struct ModalKernels {
    cudaError_t (*tail)(const ModalArgs<T> *d_args, int nmode, int nb, int threads, size_t smem, cudaStream_t st);
    cudaError_t (*slab)(const ModalArgs<T> &a, int l, int nb, cudaStream_t st);
    cudaError_t (*relax)(const ModalArgs<T> &a, int l, int colour, int mode, int nb, cudaStream_t st);
    cudaError_t (*restrict_)(const ModalArgs<T> &a, int l, int nb, cudaStream_t st);
    int table_elems;     // of one plane class (elements of T)
    int table64_elems;   // of the coarsest plane (doubles)
    int max_threads;
    bool (*slab_fits)(const ModalArgs<T> &a, int l);
};
template <class T>
const ModalKernels<T> &modal_kernels(ModalConfig c);

}  // namespace smg
