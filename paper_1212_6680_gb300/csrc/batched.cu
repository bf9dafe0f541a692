// batched.cu -- krylov_solve_batched: many independent 7-point Laplacian systems on uneven
// grids solved together by Algorithm 1 of arXiv:1212.6680 (PCG eq. (1), flexible PCG eq. (2),
// PSD) with the SMG preconditioner.
//
// Per iteration, one CUDA graph:
//   1. the V-cycles of all systems in the sine eigenvectors of their x-lines (modal.cuh): one launch
//      transforms every system's residuals, one CTA per (system, mode) runs that mode's whole cycle
//      in shared memory (largest systems first; up to two launches side by side, by how many CTAs
//      share an SM), one launch transforms back.  Systems with planes too many for that run their
//      finest levels through the slab kernels first;
//   2. the FP64 Krylov kernels over all systems at once: vectors are concatenated, every CTA
//      works on one chunk of one system, per-system sums are finished by one thread per system
//      (compensated), and the per-system scalars (alpha, beta, norms) live on the device;
//   3. an 8-byte copy of the number of systems still iterating.
// A system whose recurrence residual meets the tolerance is masked out on the device (its
// CTAs return at once); when none is left, the true residuals are checked and any
// system that fails continues from its true residual with beta = 0.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <numeric>
#include <string>
#include <vector>

#include "../../include/smg.h"
#include "modal.h"
#include "plane_relax.cuh"
#include "reduce.cuh"

namespace smg {

namespace {

// ---- barrier self-test ------------------------------------------------------------------------------
__device__ __forceinline__ bool test_barrier(unsigned *count, unsigned *gen, int *err, long long limit,
                                             unsigned expected) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned g = *reinterpret_cast<volatile unsigned *>(gen);
        __threadfence();
        const unsigned arrived = atomicAdd(count, 1u);
        if (arrived == expected - 1) {
            atomicExch(count, 0u);
            __threadfence();
            atomicAdd(gen, 1u);
        } else {
            long long spins = 0;
            while (*reinterpret_cast<volatile unsigned *>(gen) == g) {
                if (*reinterpret_cast<volatile int *>(err) != 0) break;
                if (++spins > limit) {
                    atomicCAS(err, 0, SMG_ERR_TIMEOUT);
                    break;
                }
                __nanosleep(100);
            }
        }
        __threadfence();
        ok = (*reinterpret_cast<volatile int *>(err) == 0);
    }
    __syncthreads();
    return ok != 0;
}

__global__ void barrier_selftest_kernel(unsigned expected, long long limit, unsigned *count, unsigned *gen, int *err) {
    for (int s = 0; s < 4; ++s)
        if (!test_barrier(count, gen, err, limit, expected)) return;
}

// ---- batched FP64 Krylov kernels --------------------------------------------------------------------
// A CTA works on one chunk of one system; one warp per system finishes its sums.  FP64 issue bounds the
// element loops (12 FP64 operations a point and iteration), so elements are taken one by one.
constexpr int kChunk = 16384;
constexpr int kBThreads = 1024;

struct BSys {
    int nx, ny, nz;
    long long off;        // offset of this system in the concatenated vectors
    FastDiv row, plane;   // division by nx and by ny
    int c0, c1;           // its chunks [c0, c1)
};

struct BScal {
    double rho, rho_prev, beta, alpha, rr, bb;
    int restart, status, iters, pad;
};

// Per-solve controls, read from device memory so that a captured graph serves every solve.
struct BCtl {
    double tol2;  // tol^2
    int maxit;
    int variant;  // SMG_PCG, SMG_FPCG or SMG_PSD
};

struct BKrylov {
    const BSys *sys;
    const int *ch_sys;
    const long long *ch_start;  // offset of the chunk in its system
    const int *ch_len;
    double *r, *p, *q;
    float *rf;                  // r rounded to FP32 (the cycle's input)
    float *s;                   // T r of every system (the cycle's output)
    const double *const *bptr;
    double *const *xptr;
    double *part;               // 2 per chunk
    BScal *sc;
    int *active;
    int *flags;                 // [0] systems still iterating, [2] systems to restart
    const BCtl *ctl;            // tolerance, maxit, variant of the current solve (device)
    int nsys;
};

__device__ __forceinline__ double stencil_at(const double *__restrict__ v, int i, int x, int y, int z, int nx, int ny, int nz) {
    const int np = nx * ny;
    double nb = (x > 0) ? v[i - 1] : 0.0;
    if (x < nx - 1) nb += v[i + 1];
    if (y > 0) nb += v[i - nx];
    if (y < ny - 1) nb += v[i + nx];
    if (z > 0) nb += v[i - np];
    if (z < nz - 1) nb += v[i + np];
    return 6.0 * v[i] - nb;
}
__device__ __forceinline__ double stencil_of(const double *__restrict__ v, const BSys &sy, int li) {
    const int row = div_by(li, sy.row), z = div_by(row, sy.plane);
    return stencil_at(v, li, li - row * sy.nx, row - z * sy.ny, z, sy.nx, sy.ny, sy.nz);
}

template <int NV>
__device__ __forceinline__ void put_partials(const BKrylov &k, int c, double (&v)[NV]) {
    block_reduce_plain<NV>(v);
    if (threadIdx.x == 0)
        for (int i = 0; i < NV; ++i) k.part[2 * c + i] = v[i];
}

// Sums of system s's partials by one warp, the result in lane 0: a lane adds every 32nd chunk's
// (compensated), the lanes' sums are added exactly.
template <int NV>
__device__ __forceinline__ void sum_chunks(const BKrylov &k, int s, double (&tot)[NV]) {
    const int b = k.sys[s].c0, e = k.sys[s].c1;
    for (int i = 0; i < NV; ++i) {
        DSum a{0.0, 0.0};
        for (int c = b + (threadIdx.x & 31); c < e; c += 32) two_sum_acc(a, k.part[2 * c + i]);
        const double p[2] = {a.s, isfinite(a.s) ? a.c : 0.0};
        tot[i] = warp_sum_exact<2>(p);
    }
}

// r = b - A x, partial ||r||^2, ||b||^2   (mode 1: only systems whose active flag is 2)
__global__ void __launch_bounds__(kBThreads) kb_init(BKrylov k, int only_flagged) {
    const int c = blockIdx.x, s = k.ch_sys[c];
    if (c == 0 && threadIdx.x == 0) k.flags[0] = k.flags[2] = 0;  // counted by the kernel that follows
    double v[2] = {0.0, 0.0};
    if (!only_flagged || k.active[s] == 2) {
        const BSys sy = k.sys[s];
        const int l0 = static_cast<int>(k.ch_start[c]), len = k.ch_len[c];
        const double *x = k.xptr[s], *b = k.bptr[s];
        double *r = k.r + sy.off;
        float *rf = k.rf + sy.off;
#pragma unroll 2
        for (int li = l0 + threadIdx.x; li < l0 + len; li += kBThreads) {
            const double bi = b[li], ri = bi - stencil_of(x, sy, li);
            r[li] = ri;
            rf[li] = narrow_f64(ri);
            v[0] = fma(ri, ri, v[0]);
            v[1] = fma(bi, bi, v[1]);
        }
    }
    put_partials<2>(k, c, v);
}

// after kb_init: norms; mode 0 (start): every system active unless already converged;
// mode 1 (after a true-residual check): systems flagged 2 continue (restart), others stop.
__global__ void __launch_bounds__(32) kb_fin_init(BKrylov k, int mode) {
    const int s = blockIdx.x;
    double t[2];
    sum_chunks<2>(k, s, t);
    if (threadIdx.x != 0) return;
    const double rr = t[0], bb = t[1];
    BScal &q = k.sc[s];
    if (mode == 0) {
        q = BScal{0, 0, 0, 0, rr, bb, 1, 0, 0, 0};
        const double bref = bb > 0.0 ? bb : 1.0;
        k.active[s] = (rr > k.ctl->tol2 * bref) ? 1 : 0;
        if (!isfinite(rr) || !isfinite(bb)) {
            q.status = SMG_ERR_NAN;
            k.active[s] = 0;
        }
    } else if (k.active[s] == 2) {
        q.rr = rr;
        q.restart = 1;
        k.active[s] = 1;
    }
    if (k.active[s] == 1) atomicAdd(k.flags, 1);
}

// (s, r), and (s, r_k - r_{k-1}) for eq. (2): r_k - r_{k-1} = -alpha A p of the step before, still in q
__global__ void __launch_bounds__(kBThreads) kb_dots(BKrylov k) {
    const int c = blockIdx.x, s = k.ch_sys[c];
    if (k.active[s] != 1) return;
    const long long g0 = k.sys[s].off + k.ch_start[c];
    const int len = k.ch_len[c];
    const bool want = (k.ctl->variant == SMG_FPCG) && (k.sc[s].restart == 0);
    const float *sp = k.s + g0;
    const double *r = k.r + g0, *q = k.q + g0;
    double v[2] = {0.0, 0.0};
#pragma unroll 4
    for (int t = threadIdx.x; t < len; t += kBThreads) {
        const double si = widen_f32(sp[t]);
        v[0] = fma(si, r[t], v[0]);
        if (want) v[1] = fma(si, q[t], v[1]);
    }
    put_partials<2>(k, c, v);
}

// smg_batched_apply: every system's right-hand side (caller memory) rounded to the cycle's input, every
// system active.
__global__ void __launch_bounds__(kBThreads) kb_apply_in(BKrylov k) {
    const int c = blockIdx.x, s = k.ch_sys[c];
    const double *r = k.bptr[s] + k.ch_start[c];
    float *to = k.rf + k.sys[s].off + k.ch_start[c];
    for (int t = threadIdx.x; t < k.ch_len[c]; t += kBThreads) to[t] = narrow_f64(r[t]);
    if (threadIdx.x == 0 && c == k.sys[s].c0) k.active[s] = 1;
}

// smg_batched_apply: every system's T r widened exactly to FP64 into the caller's s.
__global__ void __launch_bounds__(kBThreads) kb_apply_out(BKrylov k) {
    const int c = blockIdx.x, s = k.ch_sys[c];
    double *out = k.xptr[s] + k.ch_start[c];
    const float *from = k.s + k.sys[s].off + k.ch_start[c];
    for (int t = threadIdx.x; t < k.ch_len[c]; t += kBThreads) out[t] = widen_f32(from[t]);
}

__global__ void __launch_bounds__(32) kb_fin_beta(BKrylov k) {
    const int s = blockIdx.x;
    if (k.active[s] != 1) return;
    double t[2];
    sum_chunks<2>(k, s, t);
    if (threadIdx.x != 0) return;
    BScal &q = k.sc[s];
    const double rho = t[0], sdr = -q.alpha * t[1];
    double beta = 0.0;
    if (q.restart == 0 && k.ctl->variant != SMG_PSD) {
        if (q.rho_prev == 0.0) q.status = SMG_ERR_BREAKDOWN;
        else beta = (k.ctl->variant == SMG_PCG) ? rho / q.rho_prev : sdr / q.rho_prev;
    }
    if (!isfinite(rho) || !isfinite(beta)) q.status = SMG_ERR_NAN;
    q.rho = rho;
    q.beta = beta;
}

__global__ void __launch_bounds__(kBThreads) kb_upd_p(BKrylov k) {
    const int c = blockIdx.x, s = k.ch_sys[c];
    if (k.active[s] != 1) return;
    const long long g0 = k.sys[s].off + k.ch_start[c];
    const int len = k.ch_len[c];
    const float *sp = k.s + g0;
    double *p = k.p + g0;
    const double beta = k.sc[s].beta;
#pragma unroll 4
    for (int t = threadIdx.x; t < len; t += kBThreads) {
        const double si = widen_f32(sp[t]);
        p[t] = (beta == 0.0) ? si : fma(beta, p[t], si);
    }
}

__global__ void __launch_bounds__(kBThreads) kb_spmv(BKrylov k) {
    const int c = blockIdx.x, s = k.ch_sys[c];
    if (k.active[s] != 1) return;
    const BSys sy = k.sys[s];
    const int l0 = static_cast<int>(k.ch_start[c]), len = k.ch_len[c];
    const double *p = k.p + sy.off;
    double *q = k.q + sy.off;
    double v[1] = {0.0};
#pragma unroll 2
    for (int li = l0 + threadIdx.x; li < l0 + len; li += kBThreads) {
        const double qi = stencil_of(p, sy, li);
        q[li] = qi;
        v[0] = fma(p[li], qi, v[0]);
    }
    put_partials<1>(k, c, v);
}

__global__ void __launch_bounds__(32) kb_fin_alpha(BKrylov k) {
    const int s = blockIdx.x;
    if (s == 0 && threadIdx.x == 0) k.flags[0] = 0;  // counted by kb_fin_rr
    if (k.active[s] != 1) return;
    double t[1];
    sum_chunks<1>(k, s, t);
    if (threadIdx.x != 0) return;
    BScal &q = k.sc[s];
    const double pq = t[0];
    if (!(pq > 0.0)) {
        q.status = (pq == pq) ? SMG_ERR_BREAKDOWN : SMG_ERR_NAN;
        q.alpha = 0.0;
    } else {
        q.alpha = q.rho / pq;
    }
}

__global__ void __launch_bounds__(kBThreads) kb_upd_xr(BKrylov k) {
    const int c = blockIdx.x, s = k.ch_sys[c];
    if (k.active[s] != 1) return;
    const long long g0 = k.sys[s].off + k.ch_start[c];
    const int len = k.ch_len[c];
    const double alpha = k.sc[s].alpha;
    double *x = k.xptr[s] + k.ch_start[c], *r = k.r + g0;
    float *rf = k.rf + g0;
    const double *p = k.p + g0, *q = k.q + g0;
    double v[1] = {0.0};
#pragma unroll 4
    for (int t = threadIdx.x; t < len; t += kBThreads) {
        x[t] = fma(alpha, p[t], x[t]);
        const double rn = fma(-alpha, q[t], r[t]);
        r[t] = rn;
        rf[t] = narrow_f64(rn);
        v[0] = fma(rn, rn, v[0]);
    }
    put_partials<1>(k, c, v);
}

__global__ void __launch_bounds__(32) kb_fin_rr(BKrylov k) {
    const int s = blockIdx.x;
    if (k.active[s] != 1) return;
    double t[1];
    sum_chunks<1>(k, s, t);
    if (threadIdx.x != 0) return;
    const double rr = t[0];
    BScal &q = k.sc[s];
    q.rr = rr;
    q.rho_prev = q.rho;
    q.restart = 0;
    q.iters += 1;
    const double bref = q.bb > 0.0 ? q.bb : 1.0;
    if (!isfinite(rr)) q.status = SMG_ERR_NAN;
    if (rr <= k.ctl->tol2 * bref || q.status != 0 || q.iters >= k.ctl->maxit) k.active[s] = 0;
    else atomicAdd(k.flags, 1);
}

// After the loop: true residual norms (kb_init computes r = b - A x), flag systems to restart.
__global__ void __launch_bounds__(32) kb_fin_true(BKrylov k, double *relres) {
    const int s = blockIdx.x;
    double t[2];
    sum_chunks<2>(k, s, t);
    if (threadIdx.x != 0) return;
    const double tt = t[0], bb = t[1], bref = bb > 0.0 ? bb : 1.0;
    relres[s] = sqrt(tt / bref);
    BScal &q = k.sc[s];
    if (q.status == 0 && tt > k.ctl->tol2 * bref && q.iters < k.ctl->maxit) {
        k.active[s] = 2;  // continue from the true residual
        atomicAdd(k.flags + 2, 1);
    }
}

// ---- host side ------------------------------------------------------------------------------------
thread_local std::string g_berr;

#define BCHK(call)                                                                      \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess) {                                                        \
            set_last_error(std::string("batched solver: ") + #call + ": " +       \
                           cudaGetErrorString(e_));                                     \
            return SMG_ERR_CUDA;                                                        \
        }                                                                               \
    } while (0)

struct DevBuf {
    std::vector<void *> ptrs;
    ~DevBuf() {
        for (void *p : ptrs) cudaFree(p);
    }
    template <class T>
    cudaError_t alloc(T **p, size_t n) {
        void *q = nullptr;
        cudaError_t e = cudaMalloc(&q, std::max<size_t>(n, 1) * sizeof(T));
        if (e == cudaSuccess) ptrs.push_back(q);
        *p = static_cast<T *>(q);
        return e;
    }
};

}  // namespace

cudaError_t launch_barrier_selftest(int blocks, int extra, long long spin_limit, unsigned *count, unsigned *gen,
                                    int *err, cudaStream_t st) {
    barrier_selftest_kernel<<<blocks, 32, 0, st>>>(static_cast<unsigned>(blocks + extra), spin_limit, count, gen, err);
    return cudaGetLastError();
}

}  // namespace smg

using namespace smg;

namespace {

struct SysPlan {
    int nx, ny, nz;
    long long N, off;                  // unknowns; offset into the concatenated vectors
    HostHierarchy H;
    ModalHost<float> m;                // the mode-space cycle
    double cycle_bytes;                // bytes of its vectors that one V-cycle has to move
};

// Vectors' words that one V-cycle of a system has to move.  The transforms read r and write f, read u and write s; the
// levels one CTA runs in shared memory read the first one's f and write its u; a level above them reads f and writes u and the
// next f, and on the way up reads the next u, and reads and writes its own; each further sweep there reads f and u
// and writes u.
double vcycle_words(const SysPlan &p, int npre, int npost) {
    const double np = static_cast<double>(p.nx) * p.ny;
    const int lt = p.m.a.lt;
    double w = 4.0 * np * p.nz + 2.0 * np * p.H.nz_l[lt];
    for (int l = 0; l < lt; ++l)
        w += np * ((2.0 + 2.0 + 3.0 * (npre - 1 + npost)) * p.H.nz_l[l] + 2.0 * p.H.nz_l[l + 1]);
    return w;
}

}  // namespace

// The tails that run with one number of threads (one launch): how many CTAs share an SM follows from it.
struct TailGroup {
    int threads = 0, count = 0;
    size_t smem = 0;
    ModalTask *tasks = nullptr;        // device, largest systems first
};

// Everything one set of grids needs, built once: hierarchies, mode-space plans and vectors, Krylov vectors,
// the lists of tiles and tails, and the per-iteration graph.
struct smg_batched_ctx {
    int nsys = 0, npre = 1, npost = 0, prec = SMG_FP32;
    int nsm = 0, nch = 0;
    std::vector<SysPlan> sys;
    DevBuf buf;
    BKrylov kk{};
    ModalConfig cfg{16, 8};
    ModalArgs<float> *d_args = nullptr;
    SineJob *d_jobs = nullptr;
    SineTile *d_tiles = nullptr;
    int ntiles = 0;
    TailGroup group[2];
    int *d_active = nullptr;
    BCtl *d_ctl = nullptr;
    int *d_flags = nullptr;            // [0] systems still iterating, [2] systems to restart
    double *d_relres = nullptr;
    BScal *d_sc = nullptr;
    double **d_bptr = nullptr, **d_xptr = nullptr;
    int *h_pinned = nullptr;           // pinned copy of d_flags
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};  // V-cycle start, V-cycle end, iteration end
    // profiling (smg_batched_profile_read)
    int profile = 0;
    long long prof_launches[2] = {0, 0};
    double prof_ms[2] = {0.0, 0.0}, prof_bytes[2] = {0.0, 0.0};
    long long kernel_launches = 0;
    int kernels_per_iter = 0, cycle_kernels = 0;

    ~smg_batched_ctx() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
        if (h_pinned) cudaFreeHost(h_pinned);
    }

    // s = T r of every active system.  side: a second stream for the other group of tails, with the events
    // that fork it from st and join it (null: one after the other on st).
    cudaError_t cycle(cudaStream_t st, cudaStream_t side = nullptr, cudaEvent_t fork = nullptr, cudaEvent_t join = nullptr) {
        const ModalKernels<float> &k = modal_kernels<float>(cfg);
        int n = 0;
        cudaError_t e = launch_sine_in_batch(d_jobs, d_tiles, ntiles, d_active, st);
        ++n;
        // levels whose planes do not all fit in one CTA: system by system (converged ones too: their
        // results are not used)
        for (const SysPlan &p : sys) {
            const ModalArgs<float> &a = p.m.a;
            for (int l = 0; l < a.lt && e == cudaSuccess; ++l) {
                if (npre == 1 && k.slab_fits(a, l)) {
                    e = k.slab(a, l, 1, st);
                    ++n;
                    continue;
                }
                for (int sw = 0; sw < npre && e == cudaSuccess; ++sw)
                    for (int c = 0; c < 2 && e == cudaSuccess; ++c, ++n) e = k.relax(a, l, c, sw == 0 ? c : 2, 1, st);
                if (e == cudaSuccess) e = k.restrict_(a, l, 1, st);
                ++n;
            }
        }
        const bool both = group[0].count > 0 && group[1].count > 0;
        if (both && side && e == cudaSuccess) {
            e = cudaEventRecord(fork, st);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(side, fork, 0);
        }
        for (int g = 0; g < 2; ++g) {
            if (group[g].count == 0 || e != cudaSuccess) continue;
            e = k.tail_batch(d_args, group[g].tasks, group[g].count, d_active, group[g].threads, group[g].smem,
                             (g == 1 && both && side) ? side : st);
            ++n;
        }
        if (both && side && e == cudaSuccess) {
            e = cudaEventRecord(join, side);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(st, join, 0);
        }
        for (const SysPlan &p : sys) {
            const ModalArgs<float> &a = p.m.a;
            for (int l = a.lt - 1; l >= 0 && e == cudaSuccess; --l) {
                e = launch_modal_prolong(a, l, 1, st);
                ++n;
                for (int sw = 0; sw < npost && e == cudaSuccess; ++sw)
                    for (int c = 1; c >= 0 && e == cudaSuccess; --c, ++n) e = k.relax(a, l, c, 2, 1, st);
            }
        }
        if (e == cudaSuccess) e = launch_sine_out_batch(d_jobs, d_tiles, ntiles, d_active, st);
        cycle_kernels = n + 1;
        return e;
    }
    cudaError_t init(cudaStream_t st, int mode) {
        kb_init<<<nch, kBThreads, 0, st>>>(kk, mode);
        kb_fin_init<<<nsys, 32, 0, st>>>(kk, mode);
        kernel_launches += 2;
        return cudaGetLastError();
    }
    cudaError_t krylov_tail(cudaStream_t st) {
        kb_dots<<<nch, kBThreads, 0, st>>>(kk);
        kb_fin_beta<<<nsys, 32, 0, st>>>(kk);
        kb_upd_p<<<nch, kBThreads, 0, st>>>(kk);
        kb_spmv<<<nch, kBThreads, 0, st>>>(kk);
        kb_fin_alpha<<<nsys, 32, 0, st>>>(kk);
        kb_upd_xr<<<nch, kBThreads, 0, st>>>(kk);
        kb_fin_rr<<<nsys, 32, 0, st>>>(kk);
        return cudaGetLastError();
    }
};

namespace {

int check_dims(int nsys, const int *dims) {
    if (nsys < 1 || nsys > 4096) {
        set_last_error("nsys must be in [1, 4096]");
        return SMG_ERR_ARG;
    }
    if (!dims) {
        set_last_error("null pointer");
        return SMG_ERR_ARG;
    }
    for (int s = 0; s < nsys; ++s) {
        const int nx = dims[3 * s], ny = dims[3 * s + 1], nz = dims[3 * s + 2];
        if (nx < 1 || ny < 1 || nz < 1 || nx > 128 || ny > kMaxNy || nz > kMaxNz) {
            set_last_error("each system needs 1 <= nx <= 128, 1 <= ny <= 512, 1 <= nz <= 4096");
            return SMG_ERR_ARG;
        }
    }
    return SMG_OK;
}

int batched_build(smg_batched_ctx &c, const int *dims, cudaStream_t st) {
    const int nsys = c.nsys;
    DevBuf &buf = c.buf;
    int dev = 0;
    BCHK(cudaGetDevice(&dev));
    BCHK(cudaDeviceGetAttribute(&c.nsm, cudaDevAttrMultiProcessorCount, dev));

    // ---- per-system hierarchies and mode-space plans (one lane configuration: the widest planes') ----
    c.sys.resize(nsys);
    std::vector<SysPlan> &sys = c.sys;
    int ny_max = 1;
    for (int s = 0; s < nsys; ++s) ny_max = std::max(ny_max, dims[3 * s + 1]);
    c.cfg = modal_config(ny_max, false);
    const ModalKernels<float> &k = modal_kernels<float>(c.cfg);
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    size_t b_shared = 0, b_coef = 0, b_c64 = 0, b_vec = 0;
    long long vtot = 0;
    std::map<int, std::pair<size_t, size_t>> sines;  // by nx: offsets of its sines and of its matrices
    std::vector<double> tables;
    size_t n_mats = 0;
    for (int s = 0; s < nsys; ++s) {
        SysPlan &p = sys[s];
        p.nx = dims[3 * s];
        p.ny = dims[3 * s + 1];
        p.nz = dims[3 * s + 2];
        p.N = static_cast<long long>(p.nx) * p.ny * p.nz;
        p.off = vtot;
        vtot += (p.N + 31) / 32 * 32;
        build_hierarchy(p.nx, p.ny, p.nz, p.H);
        if (modal_plan<float>(p.m, p.H, modal_shape(p.H), c.cfg, c.npre, c.npost) != 0) {
            set_last_error("batched solver: a system's planes do not fit the mode-space cycle");
            return SMG_ERR_CUDA;
        }
        modal_vectors<float>(p.m, 1);
        p.cycle_bytes = vcycle_words(p, c.npre, c.npost) * sizeof(float);
        b_shared += p.m.shared.size();
        b_coef += up(p.m.coef_values * sizeof(float));
        b_c64 += up(p.m.coef64_values * sizeof(double));
        b_vec += p.m.vec_bytes;
        if (sines.emplace(p.nx, std::make_pair(tables.size(), n_mats)).second) {
            const std::vector<double> t = sine_table(p.nx);
            tables.insert(tables.end(), t.begin(), t.end());
            n_mats += 4 * static_cast<size_t>(sine_order(p.nx)) * sine_order(p.nx);
        }
    }
    unsigned char *d_shared, *d_coef, *d_c64, *d_vec;
    float *d_mats;
    BCHK(buf.alloc(&d_shared, b_shared));
    BCHK(buf.alloc(&d_coef, b_coef));
    BCHK(buf.alloc(&d_c64, b_c64));
    BCHK(buf.alloc(&d_vec, b_vec));
    BCHK(buf.alloc(&d_mats, n_mats));
    double *d_tables;
    BCHK(buf.alloc(&d_tables, tables.size()));
    BCHK(buf.alloc(&c.kk.r, vtot));
    BCHK(buf.alloc(&c.kk.p, vtot));
    BCHK(buf.alloc(&c.kk.q, vtot));
    BCHK(buf.alloc(&c.kk.rf, vtot));
    BCHK(buf.alloc(&c.kk.s, vtot));
    BCHK(cudaMemsetAsync(c.kk.p, 0, vtot * sizeof(double), st));
    BCHK(cudaMemsetAsync(c.kk.q, 0, vtot * sizeof(double), st));
    BCHK(cudaMemcpyAsync(d_tables, tables.data(), tables.size() * sizeof(double), cudaMemcpyHostToDevice, st));
    for (const auto &e : sines) BCHK(launch_sine_matrices<float>(e.first, d_tables + e.second.first, d_mats + e.second.second, st));
    std::vector<unsigned char> shared;
    shared.reserve(b_shared);
    {
        size_t o_s = 0, o_c = 0, o_6 = 0, o_v = 0;
        for (SysPlan &p : sys) {
            modal_place<float>(p.m, d_shared + o_s, reinterpret_cast<float *>(d_coef + o_c), reinterpret_cast<double *>(d_c64 + o_6), d_vec + o_v);
            shared.insert(shared.end(), p.m.shared.begin(), p.m.shared.end());
            o_s += p.m.shared.size();
            o_c += up(p.m.coef_values * sizeof(float));
            o_6 += up(p.m.coef64_values * sizeof(double));
            o_v += p.m.vec_bytes;
        }
    }
    BCHK(cudaMemcpyAsync(d_shared, shared.data(), shared.size(), cudaMemcpyHostToDevice, st));
    for (SysPlan &p : sys)
        BCHK(k.setup(p.m.a, const_cast<float *>(p.m.a.coef), const_cast<double *>(p.m.a.coef64), st));

    // ---- lists: transform tiles, and the tails by threads per CTA (an SM holds 512 threads of them: one
    // CTA of 512, or two of 256 where the shared memory allows), largest planes first ----
    std::vector<int> by_size(nsys);
    std::iota(by_size.begin(), by_size.end(), 0);
    std::stable_sort(by_size.begin(), by_size.end(), [&](int a, int b) {
        return static_cast<long long>(sys[a].ny) * sys[a].nz > static_cast<long long>(sys[b].ny) * sys[b].nz;
    });
    std::vector<ModalArgs<float>> args(nsys);
    std::vector<SineJob> jobs(nsys);
    std::vector<SineTile> tiles;
    std::vector<ModalTask> tasks[2];
    for (int s : by_size) {
        SysPlan &p = sys[s];
        args[s] = p.m.a;
        SineArgs g{p.nx, p.ny, p.nz, p.m.a.pitch, (p.nx + 1) / 2, sine_order(p.nx), d_mats + sines[p.nx].second};
        jobs[s] = SineJob{g, c.kk.rf + p.off, p.m.a.fw[0], p.m.a.u[0], c.kk.s + p.off};
        for (int m = 0; m < sine_mode_tiles(g); ++m)
            for (int t = 0; t < sine_line_tiles(g); ++t) tiles.push_back(SineTile{s, t, m});
        const int gi = 2 * (p.m.smem + 2048) <= kModalSmem ? 1 : 0;
        c.group[gi].threads = gi ? 256 : k.max_threads;
        c.group[gi].smem = std::max(c.group[gi].smem, p.m.smem);
        for (int m = 0; m < p.nx; ++m) tasks[gi].push_back(ModalTask{s, m});
    }
    BCHK(buf.alloc(&c.d_args, nsys));
    BCHK(buf.alloc(&c.d_jobs, nsys));
    BCHK(buf.alloc(&c.d_tiles, tiles.size()));
    BCHK(cudaMemcpyAsync(c.d_args, args.data(), nsys * sizeof(args[0]), cudaMemcpyHostToDevice, st));
    BCHK(cudaMemcpyAsync(c.d_jobs, jobs.data(), nsys * sizeof(jobs[0]), cudaMemcpyHostToDevice, st));
    BCHK(cudaMemcpyAsync(c.d_tiles, tiles.data(), tiles.size() * sizeof(tiles[0]), cudaMemcpyHostToDevice, st));
    c.ntiles = static_cast<int>(tiles.size());
    for (int g = 0; g < 2; ++g) {
        c.group[g].count = static_cast<int>(tasks[g].size());
        BCHK(buf.alloc(&c.group[g].tasks, tasks[g].size()));
        BCHK(cudaMemcpyAsync(c.group[g].tasks, tasks[g].data(), tasks[g].size() * sizeof(ModalTask), cudaMemcpyHostToDevice, st));
    }

    // ---- Krylov data ----
    std::vector<BSys> hsys(nsys);
    std::vector<int> ch_sys, ch_len;
    std::vector<long long> ch_start;
    for (int s = 0; s < nsys; ++s) {
        BSys &q = hsys[s];
        q.nx = sys[s].nx;
        q.ny = sys[s].ny;
        q.nz = sys[s].nz;
        q.off = sys[s].off;
        q.row = fast_div(q.nx);
        q.plane = fast_div(q.ny);
        q.c0 = static_cast<int>(ch_sys.size());
        for (long long cc = 0; cc < sys[s].N; cc += kChunk) {
            ch_sys.push_back(s);
            ch_start.push_back(cc);
            ch_len.push_back(static_cast<int>(std::min<long long>(kChunk, sys[s].N - cc)));
        }
        q.c1 = static_cast<int>(ch_sys.size());
    }
    c.nch = static_cast<int>(ch_sys.size());
    const int nch = c.nch;
    BSys *d_sys;
    int *d_ch_sys, *d_ch_len;
    long long *d_ch_start;
    BCHK(buf.alloc(&d_sys, nsys));
    BCHK(buf.alloc(&d_ch_sys, nch));
    BCHK(buf.alloc(&d_ch_len, nch));
    BCHK(buf.alloc(&d_ch_start, nch));
    BCHK(buf.alloc(&c.kk.part, 2 * static_cast<size_t>(nch)));
    BCHK(buf.alloc(&c.d_active, nsys));
    BCHK(buf.alloc(&c.d_flags, 4));
    BCHK(buf.alloc(&c.d_ctl, 1));
    BCHK(buf.alloc(&c.d_relres, nsys));
    BCHK(buf.alloc(&c.d_sc, nsys));
    BCHK(buf.alloc(&c.d_bptr, nsys));
    BCHK(buf.alloc(&c.d_xptr, nsys));
    BCHK(cudaMemsetAsync(c.d_flags, 0, 4 * sizeof(int), st));
    BCHK(cudaMemcpyAsync(d_sys, hsys.data(), nsys * sizeof(BSys), cudaMemcpyHostToDevice, st));
    BCHK(cudaMemcpyAsync(d_ch_sys, ch_sys.data(), nch * sizeof(int), cudaMemcpyHostToDevice, st));
    BCHK(cudaMemcpyAsync(d_ch_len, ch_len.data(), nch * sizeof(int), cudaMemcpyHostToDevice, st));
    BCHK(cudaMemcpyAsync(d_ch_start, ch_start.data(), nch * sizeof(long long), cudaMemcpyHostToDevice, st));
    BKrylov &kk = c.kk;
    kk.sys = d_sys;
    kk.ch_sys = d_ch_sys;
    kk.ch_start = d_ch_start;
    kk.ch_len = d_ch_len;
    kk.bptr = c.d_bptr;
    kk.xptr = c.d_xptr;
    kk.sc = c.d_sc;
    kk.active = c.d_active;
    kk.flags = c.d_flags;
    kk.ctl = c.d_ctl;
    kk.nsys = nsys;
    BCHK(cudaMallocHost(&c.h_pinned, 4 * sizeof(int)));
    for (cudaEvent_t &e : c.ev) BCHK(cudaEventCreate(&e));
    BCHK(cudaStreamSynchronize(st));  // the copies above read this function's vectors

    // ---- capture one iteration into a CUDA graph ----
    struct Capture {
        cudaStream_t s = nullptr, side = nullptr;
        cudaEvent_t fork = nullptr, join = nullptr;
        ~Capture() {
            if (fork) cudaEventDestroy(fork);
            if (join) cudaEventDestroy(join);
            if (s) cudaStreamDestroy(s);
            if (side) cudaStreamDestroy(side);
        }
    } cap;
    BCHK(cudaStreamCreateWithFlags(&cap.s, cudaStreamNonBlocking));
    BCHK(cudaStreamCreateWithFlags(&cap.side, cudaStreamNonBlocking));
    BCHK(cudaEventCreateWithFlags(&cap.fork, cudaEventDisableTiming));
    BCHK(cudaEventCreateWithFlags(&cap.join, cudaEventDisableTiming));
    {
        cudaStream_t cs = cap.s;
        BCHK(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        // the events become event-record nodes, so the V-cycle and the Krylov part of every
        // replay can be timed
        cudaError_t e = cudaEventRecordWithFlags(c.ev[0], cs, cudaEventRecordExternal);
        if (e == cudaSuccess) e = c.cycle(cs, cap.side, cap.fork, cap.join);
        if (e == cudaSuccess) e = cudaEventRecordWithFlags(c.ev[1], cs, cudaEventRecordExternal);
        if (e == cudaSuccess) e = c.krylov_tail(cs);
        if (e == cudaSuccess) e = cudaEventRecordWithFlags(c.ev[2], cs, cudaEventRecordExternal);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(c.h_pinned, c.d_flags, sizeof(int), cudaMemcpyDeviceToHost, cs);
        cudaError_t e2 = cudaStreamEndCapture(cs, &c.graph);
        if (e != cudaSuccess || e2 != cudaSuccess) {
            set_last_error(std::string("batched solver: graph capture: ") +
                           cudaGetErrorString(e != cudaSuccess ? e : e2));
            return SMG_ERR_CUDA;
        }
        BCHK(cudaGraphInstantiate(&c.exec, c.graph, 0));
    }
    c.kernels_per_iter = c.cycle_kernels + 7;
    return SMG_OK;
}

int batched_solve(smg_batched_ctx &c, int variant, const double *const *b, double *const *x, double tol, int maxit,
                  int *iters, double *relres, cudaStream_t st) {
    const int nsys = c.nsys;
    for (int s = 0; s < nsys; ++s) iters[s] = 0;
    const BCtl ctl{tol * tol, maxit, variant};
    BCHK(cudaMemcpyAsync(c.d_ctl, &ctl, sizeof(BCtl), cudaMemcpyHostToDevice, st));
    BCHK(cudaMemcpyAsync(c.d_bptr, b, nsys * sizeof(double *), cudaMemcpyHostToDevice, st));
    BCHK(cudaMemcpyAsync(c.d_xptr, x, nsys * sizeof(double *), cudaMemcpyHostToDevice, st));
    BCHK(c.init(st, 0));
    BCHK(cudaMemcpyAsync(c.h_pinned, c.d_flags, sizeof(int), cudaMemcpyDeviceToHost, st));
    BCHK(cudaStreamSynchronize(st));
    int nact = c.h_pinned[0];
    for (int round = 0; round < 8; ++round) {
        for (int it = 0; it < maxit && nact > 0; ++it) {
            BCHK(cudaGraphLaunch(c.exec, st));
            BCHK(cudaStreamSynchronize(st));
            c.kernel_launches += c.kernels_per_iter;
            nact = c.h_pinned[0];
            if (c.profile) {
                float m0 = 0.0f, m1 = 0.0f;
                if (cudaEventElapsedTime(&m0, c.ev[0], c.ev[1]) == cudaSuccess &&
                    cudaEventElapsedTime(&m1, c.ev[1], c.ev[2]) == cudaSuccess) {
                    c.prof_launches[0] += 1;
                    c.prof_ms[0] += m0;
                    c.prof_launches[1] += 1;
                    c.prof_ms[1] += m1;
                }
            }
        }
        // true residuals; systems that fail continue from them
        kb_init<<<c.nch, kBThreads, 0, st>>>(c.kk, 0);
        kb_fin_true<<<nsys, 32, 0, st>>>(c.kk, c.d_relres);
        BCHK(cudaGetLastError());
        c.kernel_launches += 2;
        BCHK(cudaMemcpyAsync(c.h_pinned + 2, c.d_flags + 2, sizeof(int), cudaMemcpyDeviceToHost, st));
        BCHK(cudaStreamSynchronize(st));
        if (c.h_pinned[2] == 0) break;
        kb_fin_init<<<nsys, 32, 0, st>>>(c.kk, 1);
        c.kernel_launches += 1;
        BCHK(cudaMemcpyAsync(c.h_pinned, c.d_flags, sizeof(int), cudaMemcpyDeviceToHost, st));
        BCHK(cudaStreamSynchronize(st));
        nact = c.h_pinned[0];
    }
    std::vector<BScal> hs(nsys);
    std::vector<double> rel(nsys);
    BCHK(cudaMemcpy(hs.data(), c.d_sc, nsys * sizeof(BScal), cudaMemcpyDeviceToHost));
    BCHK(cudaMemcpy(rel.data(), c.d_relres, nsys * sizeof(double), cudaMemcpyDeviceToHost));
    int result = SMG_OK;
    for (int s = 0; s < nsys; ++s) {
        iters[s] = hs[s].iters;
        if (relres) relres[s] = rel[s];
        if (c.profile) c.prof_bytes[0] += hs[s].iters * c.sys[s].cycle_bytes;
        if (hs[s].status != 0 && result == SMG_OK) result = hs[s].status;
        if (result == SMG_OK && !(rel[s] <= tol)) result = SMG_ERR_NOCONV;
    }
    if (result == SMG_ERR_NOCONV) set_last_error("batched solver: a system did not converge within maxit");
    else if (result != SMG_OK) set_last_error("batched solver: breakdown or NaN in a system");
    return result;
}

}  // namespace

extern "C" int smg_batched_setup(int nsys, const int *dims, int npre, int npost, int prec, smg_batched_handle *out,
                                 void *stream) {
    if (!out) {
        set_last_error("null pointer");
        return SMG_ERR_ARG;
    }
    *out = nullptr;
    int rc = check_dims(nsys, dims);
    if (rc != SMG_OK) return rc;
    if (npre < 1 || npost < 0 || npre > 8 || npost > 8) {
        set_last_error("1 <= npre <= 8 and 0 <= npost <= 8 required");
        return SMG_ERR_ARG;
    }
    if (prec != SMG_FP32) {
        set_last_error("the batched solver runs the FP32 cycle (SMG_FP32) only");
        return SMG_ERR_ARG;
    }
    auto *c = new smg_batched_ctx();
    c->nsys = nsys;
    c->npre = npre;
    c->npost = npost;
    c->prec = prec;
    rc = batched_build(*c, dims, static_cast<cudaStream_t>(stream));
    if (rc != SMG_OK) {
        const std::string msg = smg_last_error();
        delete c;
        set_last_error(msg);
        return rc;
    }
    *out = c;
    return SMG_OK;
}

extern "C" int smg_batched_solve(smg_batched_handle h, int variant, const double *const *b, double *const *x,
                                 double tol, int maxit, int *iters, double *relres, void *stream) {
    if (!h || !b || !x || !iters) {
        set_last_error("null pointer");
        return SMG_ERR_ARG;
    }
    if (variant != SMG_PCG && variant != SMG_FPCG && variant != SMG_PSD) {
        set_last_error("variant must be SMG_PCG, SMG_FPCG or SMG_PSD");
        return SMG_ERR_ARG;
    }
    if (!(tol > 0.0) || maxit < 0) {
        set_last_error("tol > 0 and maxit >= 0 required");
        return SMG_ERR_ARG;
    }
    for (int s = 0; s < h->nsys; ++s) {
        if (!b[s] || !x[s]) {
            set_last_error("null vector pointer");
            return SMG_ERR_ARG;
        }
    }
    return batched_solve(*h, variant, b, x, tol, maxit, iters, relres, static_cast<cudaStream_t>(stream));
}

extern "C" int smg_batched_apply(smg_batched_handle h, const double *const *r, double *const *out, void *stream) {
    if (!h || !r || !out) {
        set_last_error("null pointer");
        return SMG_ERR_ARG;
    }
    for (int s = 0; s < h->nsys; ++s) {
        if (!r[s] || !out[s]) {
            set_last_error("null vector pointer");
            return SMG_ERR_ARG;
        }
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    smg_batched_ctx &c = *h;
    BCHK(cudaMemcpyAsync(c.d_bptr, r, c.nsys * sizeof(double *), cudaMemcpyHostToDevice, st));
    BCHK(cudaMemcpyAsync(c.d_xptr, out, c.nsys * sizeof(double *), cudaMemcpyHostToDevice, st));
    kb_apply_in<<<c.nch, kBThreads, 0, st>>>(c.kk);
    BCHK(cudaGetLastError());
    BCHK(c.cycle(st));
    kb_apply_out<<<c.nch, kBThreads, 0, st>>>(c.kk);
    BCHK(cudaGetLastError());
    c.kernel_launches += c.cycle_kernels + 2;
    BCHK(cudaStreamSynchronize(st));
    return SMG_OK;
}

extern "C" int smg_batched_destroy(smg_batched_handle h) {
    if (h) {
        cudaDeviceSynchronize();
        delete h;
    }
    return SMG_OK;
}

extern "C" int smg_batched_info(smg_batched_handle h, int *threads, int *order, int *blocks, long long *tasks,
                                long long *launches, int *rows_per_lane) {
    if (!h || !threads || !order || !blocks || !tasks || !launches || !rows_per_lane) {
        set_last_error("null pointer");
        return SMG_ERR_ARG;
    }
    // the group of tails with the larger planes
    const TailGroup &g = h->group[0].count > 0 ? h->group[0] : h->group[1];
    int nx = 1;
    for (const SysPlan &p : h->sys) nx = std::max(nx, p.nx);
    *threads = g.threads;
    *order = 1;
    *rows_per_lane = (nx + 31) / 32;
    *blocks = h->nsm * (g.threads == 256 ? 2 : 1);
    *tasks = h->group[0].count + h->group[1].count;
    *launches = h->kernel_launches;
    return SMG_OK;
}

extern "C" int smg_batched_set_profile(smg_batched_handle h, int on) {
    if (!h || on < 0 || on > 1) {
        set_last_error("a handle and on in {0, 1} required");
        return SMG_ERR_ARG;
    }
    h->profile = on;
    return SMG_OK;
}

extern "C" int smg_batched_profile_read(smg_batched_handle h, int which, long long *launches, double *ms,
                                        double *bytes) {
    if (!h || which < 0 || which > 1 || !launches || !ms || !bytes) {
        set_last_error("bad arguments");
        return SMG_ERR_ARG;
    }
    *launches = h->prof_launches[which];
    *ms = h->prof_ms[which];
    *bytes = h->prof_bytes[which];
    h->prof_launches[which] = 0;
    h->prof_ms[which] = 0.0;
    h->prof_bytes[which] = 0.0;
    return SMG_OK;
}

extern "C" int krylov_solve_batched(int nsys, const int *dims, int npre, int npost, int prec, const double *const *b,
                                    double *const *x, double tol, int maxit, int *iters, void *stream) {
    if (!b || !x || !iters || !dims) {
        set_last_error("null pointer");
        return SMG_ERR_ARG;
    }
    if (!(tol > 0.0) || maxit < 0) {
        set_last_error("npre >= 1, npost >= 0, tol > 0, maxit >= 0 required");
        return SMG_ERR_ARG;
    }
    if (nsys >= 1 && nsys <= 4096)
        for (int s = 0; s < nsys; ++s) iters[s] = 0;
    smg_batched_handle h = nullptr;
    int rc = smg_batched_setup(nsys, dims, npre, npost, prec, &h, stream);
    if (rc != SMG_OK) return rc;
    rc = smg_batched_solve(h, SMG_FPCG, b, x, tol, maxit, iters, nullptr, stream);
    const std::string msg = rc != SMG_OK ? std::string(smg_last_error()) : std::string();
    smg_batched_destroy(h);
    if (rc != SMG_OK) set_last_error(msg);
    return rc;
}

extern "C" int smg_barrier_selftest(int extra_blocks, double limit_seconds, int *status, void *stream) {
    if (!status || extra_blocks < 0 || !(limit_seconds > 0.0) || limit_seconds > 10.0) {
        set_last_error("status must be non-null, extra_blocks >= 0, 0 < limit_seconds <= 10");
        return SMG_ERR_ARG;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned *d = nullptr;
    cudaError_t e = cudaMalloc(&d, 4 * sizeof(unsigned));
    if (e != cudaSuccess) {
        set_last_error(std::string("smg_barrier_selftest: ") + cudaGetErrorString(e));
        return SMG_ERR_CUDA;
    }
    cudaMemsetAsync(d, 0, 4 * sizeof(unsigned), st);
    // one poll takes at least the 100 ns sleep: the limit is a lower bound on the wait
    const long long spins = static_cast<long long>(limit_seconds * 1e7);
    e = launch_barrier_selftest(4, extra_blocks, spins, d, d + 1, reinterpret_cast<int *>(d + 2), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(status, d + 2, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(d);
    if (e != cudaSuccess) {
        set_last_error(std::string("smg_barrier_selftest: ") + cudaGetErrorString(e));
        return SMG_ERR_CUDA;
    }
    return SMG_OK;
}
