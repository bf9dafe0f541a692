// modal.h -- the SMG V-cycle in the sine eigenvectors of the x-lines (modal.cuh has the kernels).
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "smg_internal.h"

namespace smg {

constexpr int kMaxZLevels = 13;   // nz <= 4096

// The V-cycle of one system on its mode grids, as the kernels read it (T: float or double).
// "Tail" levels are the z-levels lt .. L-1, which one CTA per mode runs in shared memory.
//
// Coefficients.  Planes of a level with equal 2D hierarchies form a class (plane_classes; two a level
// here: the planes away from the end, and the last).  Lines whose coefficients agree in every class
// form a line type (about five per 2D level: next to the ends, and even and odd between).  For each
// mode and class, modal_setup_kernel forms once the kRow multipliers of every line type and the G x G
// matrix of the y-cycle below the levels a lane holds: `blk` values, which the kernels spread over
// their lines.
struct TailOp;

template <class T>
struct ModalArgs {
    int nmode, ny, pitch;      // x-modes, lines, and lines per plane in global memory (ny rounded up to 4)
    int L, lt;                 // z-levels; first tail level
    int P, sum_ny;             // 2D levels and their lines in all
    int npre, npost;
    int ntype, nptype, ncls_all, blk;  // line types, plane types, classes of all levels, values per class
    int ny_m[kMaxPlaneLevels], line_base[kMaxPlaneLevels];
    int nz[kMaxZLevels];       // planes of each z-level
    int plane_base[kMaxZLevels];
    int cls_base[kMaxZLevels]; // first class of the level
    int ncls[kMaxZLevels];     // plane classes of the level
    int sm_u[kMaxZLevels], sm_f[kMaxZLevels];  // shared-memory offsets (elements of T) of the tail levels
    int sm_pitch;              // lines per plane in shared memory
    int sm_tab, sm_stage, sm_zt;         // offsets (elements of T): line tables, staged classes, plane types
    int sm_tab64, sm_ltype, sm_ptype, sm_pcls;  // offsets (bytes)
    const T *f[kMaxZLevels];   // right-hand sides and iterates in global memory: [rhs][mode][plane][pitch],
    T *u[kMaxZLevels];         // levels 0 .. lt
    T *fw[kMaxZLevels];        // f, writable (levels 1 .. lt)
    const T *zt;               // [plane types][8] plane coefficients
    const unsigned short *ptype;  // [planes of all levels] plane type
    const unsigned short *pcls;   // [plane types] class within the level
    const unsigned short *ltype;  // [sum_ny] line type
    const T *coef;             // [mode][class][blk]
    const double *coef64;      // [mode][blk64]: the coarsest level's class in FP64, 32 lanes
    const double *lam;         // [nmode] eigenvalues of the x-line Laplacian
    const TailOp *ops;         // the tail's steps, the last OP_END
    const double *raw;         // [class][ntype][kRawPerLine]: what the multipliers are formed from
};

// One step of the tail kernel, planned on the host (the kernel's own loop over levels, colours and sweeps spent
// 400 of a coarse step's 1800 cycles finding out what to do next).
enum : int { OP_RELAX = 1, OP_RESTRICT = 2, OP_COARSEST = 3, OP_PROLONG = 4, OP_STORE = 5, OP_TABLES = 6, OP_END = 7 };
struct alignas(16) TailOp {
    int kind;
    int level;
    int colour, mode, n;   // OP_RELAX: planes colour, colour + 2, ..; relax_plane's mode; how many
    int nz, nzc;           // planes of the level and of the next
    int u, f, uc, fc;      // shared-memory offsets of the level's vectors (f -1: in global memory) and the next's
    int ptype;             // of the level's first plane, from the tail's first
    int fetch, fetch_n;    // classes of the level relaxed next: first value, values (0: nothing to fetch)
    int spread;            // classes to spread into line tables (0: none)
    int out;               // OP_PROLONG, OP_STORE: to global memory
};
static_assert(sizeof(TailOp) == 64, "four 16-byte loads");

constexpr int kRawPerLine = 14;  // raw_line in modal.cu
constexpr int kRow = 8;          // multipliers of a line type

// Lanes per plane and lines per lane for planes of ny lines.
struct ModalConfig {
    int G, K;
};
ModalConfig modal_config(int ny, bool f64);

// Shared memory the tail kernel may use.
constexpr size_t kModalSmem = 227 * 1024 - 2048;

// The transforms of one system's x-lines into mode space and back (modal.cu).
struct SineArgs {
    int nx, ny, nz, pitch;   // pitch: lines per plane of the mode vectors (lines ny .. pitch-1 are zero)
    int nh;                  // odd modes, and pairs of points: ceil(nx / 2)
    int hp;                  // order of the stored matrices (nh rounded up to 64)
    const void *mat;         // [4][hp][hp]: by point odd, even; by mode odd, even
};

// One system's mode-space cycle as planned on the host: its kernel arguments, the bytes its modes share
// and what else it needs on the device (set by modal_place).
template <class T>
struct ModalHost {
    ModalArgs<T> a;
    ModalConfig cfg{16, 8};
    size_t smem = 0;                   // tail kernel
    std::vector<unsigned char> shared; // raw, lam, zt, ptype, pcls, ltype, ops
    size_t at[7] = {0};
    size_t coef_values = 0, coef64_values = 0, vec_bytes = 0;
    std::vector<size_t> vec_off;       // f and u of levels 0 .. lt
};
// What a hierarchy's plans of either type and any lane configuration are made of: the types and classes of its planes and
// lines.  Reads every plane's table (3 x 512 x 4096 points: 24 ms), so a handle keeps it.
struct ModalShape {
    int ntype = 0, ncls_all = 0;
    int cls_base[kMaxZLevels] = {0}, ncls[kMaxZLevels] = {0};
    std::vector<unsigned short> ptype, pcls, ltype;
    std::vector<double> zt, raw, lam;
};
ModalShape modal_shape(const HostHierarchy &H);
template <class T>
int modal_plan(ModalHost<T> &h, const HostHierarchy &H, const ModalShape &s, ModalConfig cfg, int npre, int npost);
// The vectors' sizes for nb right-hand sides (vec_off, vec_bytes).
template <class T>
void modal_vectors(ModalHost<T> &h, int nb);
template <class T>
void modal_place(ModalHost<T> &h, unsigned char *shared, T *coef, double *coef64, unsigned char *vec);
// The transforms' matrices of lines of nx points: their order as stored, the sines they are made of (host), and the
// four of them, 4 sine_order^2 values at mat, from those sines on the device.
inline int sine_order(int nx) { return ((nx + 1) / 2 + 63) / 64 * 64; }
std::vector<double> sine_table(int nx);
template <class T>
cudaError_t launch_sine_matrices(int nx, const double *sines, T *mat, cudaStream_t st);
// Threads of the tail kernel for systems that need smem bytes when ctas of them are to run: the kernel
// takes 128 registers a thread, so 512 threads fill an SM; with more CTAs than SMs the SM is shared by as
// many as the shared memory allows, else one CTA takes it whole (as far as its planes fill it).
// 1280x80x80, 1280 CTAs of 100 KB: two of 256 threads an SM 703 us an application, one of 512 809; no other size of the
// benchmark's differs by 2 %.
int modal_tail_threads(size_t smem, long long ctas, int num_sms, int most, int planes, int G);

struct ModalPlan {
    bool f64 = false;
    int nb = 0, num_sms = 0;
    ModalHost<float> h32;
    ModalHost<double> h64;
    SineArgs sine{};
    void *d_buf = nullptr;        // mode-space vectors
    void *d_tab = nullptr;        // coefficients and transform matrices, the kernels' arguments at at_args
    size_t at_args = 0;
};

// Tables, unless they are there, and vectors for nb right-hand sides; 0, or a cudaError_t (give the plan back then).
int modal_build(ModalPlan &p, const HostHierarchy &H, const ModalShape &s, bool f64, int nb, int npre, int npost);
void modal_free(ModalPlan &p);

// u0 = T f0 for nb right-hand sides, in three parts: f0 ([rhs][z][y][x], of type F64, or F32 for an FP32
// plan) into mode space, the cycle there, and back into u0 (elements of type `type`, values of a BF16 cycle rounded to
// bfloat16 in either type: value = BF16).  coarse_iters: steps on the one-plane coarsest level.  Each adds its kernel
// launches to `launches`.  Asynchronous on st.
cudaError_t modal_transform_in(const ModalPlan &p, int nb, Prec type, const void *f0, cudaStream_t st, long long &launches);
cudaError_t modal_cycle(const ModalPlan &p, int nb, int coarse_iters, cudaStream_t st, long long &launches);
cudaError_t modal_transform_out(const ModalPlan &p, int nb, Prec value, Prec type, void *u0, cudaStream_t st, long long &launches);

// Whether the FP64 cycle of nb right-hand sides is faster in mode space than on the plane kernels (form.cpp).
bool mode_space_faster(int nx, int ny, int nz, int nb, int npre, int npost);

// Many systems at once (batched.cu), FP32: their transforms and tails as one launch each, the CTAs taken
// from lists of (system, tile) and (system, mode); systems whose active flag is not 1 are skipped.
struct SineJob {
    SineArgs g;
    const float *in;       // physical right-hand side
    float *fh;             // mode-space right-hand side and result
    const float *uh;
    float *out;            // physical result
};
struct SineTile {
    int sys, line_tile, mode_tile;
};
// FP32 transforms (sine.cu) of physical vectors with elements of type `type` (forward: F32 or F64); scratch: as
// many values as out.  Backward, F64 elements hold values rounded to `value` (BF16, or no further).
cudaError_t sine_in_f32(const SineArgs &g, int nb, Prec type, const void *f, float *out, float *scratch, cudaStream_t st, long long &launches);
cudaError_t sine_out_f32(const SineArgs &g, int nb, const float *a, Prec value, Prec type, void *u, cudaStream_t st, long long &launches);
int sine_line_tiles(const SineArgs &g);
int sine_mode_tiles(const SineArgs &g);
cudaError_t launch_sine_in_batch(const SineJob *jobs, const SineTile *tiles, int ntiles, const int *active, cudaStream_t st);
cudaError_t launch_sine_out_batch(const SineJob *jobs, const SineTile *tiles, int ntiles, const int *active, cudaStream_t st);
struct ModalTask {
    int sys, mode;
};
cudaError_t launch_modal_prolong(const ModalArgs<float> &a, int l, int nb, cudaStream_t st);

// Kernels of one configuration (modal_inst.cu).
template <class T>
struct ModalKernels {
    cudaError_t (*setup)(const ModalArgs<T> &a, T *coef, double *coef64, cudaStream_t st);
    cudaError_t (*tail)(const ModalArgs<T> *d_args, int nmode, int nb, int coarse_iters, int threads, size_t smem, cudaStream_t st);
    cudaError_t (*tail_batch)(const ModalArgs<T> *d_args, const ModalTask *tasks, int ntasks, const int *active, int threads,
                              size_t smem, cudaStream_t st);
    cudaError_t (*slab)(const ModalArgs<T> &a, int l, int nb, cudaStream_t st);
    cudaError_t (*relax)(const ModalArgs<T> &a, int l, int colour, int mode, int nb, cudaStream_t st);
    cudaError_t (*restrict_)(const ModalArgs<T> &a, int l, int nb, cudaStream_t st);
    bool (*slab_fits)(const ModalArgs<T> &a, int l);
    int table_elems;     // a class's line table in shared memory (elements of T)
    int max_threads;
};
template <class T>
const ModalKernels<T> &modal_kernels(ModalConfig c);

}  // namespace smg
