// krylov_kernels.cu -- FP64 kernels of Algorithm 1 (section "PSD and PCG methods" of
// arXiv:1212.6680): s_k = T r_k, p_k = s_k + beta_k p_{k-1}, alpha_k = (s_k, r_k)/(p_k, A p_k),
// x_{k+1} = x_k + alpha_k p_k, r_{k+1} = r_k - alpha_k A p_k, with beta_k from eq. (1)
// (standard PCG), eq. (2) (flexible PCG, extra vector r_k - r_{k-1}) or 0 (PSD).
//
// The scalars live on the device (KrylovScalars); the last CTA of each reduction kernel
// combines the per-CTA partial sums and computes the scalar the next kernel needs, so one
// iteration runs without the host.  Inner products: each thread accumulates its products
// with FMA, then the CTAs' partials are added exactly (reduce.cuh).  With T = I, rho is the ||r||^2 of the step before
// and no kernel forms it.
// The preconditioned residual s is read straight from the V-cycle's level-0 storage
// (FP64, FP32 or BF16): widening it to FP64 is exact, so no FP64 copy of s is made.
#include <cuda_bf16.h>

#include "grid_sync.cuh"
#include "krylov.h"
#include "plane_relax.cuh"
#include "reduce.cuh"

namespace smg {

// Write this block's partials; the last block to finish sums all of them (rounded once) into
// tot[] (thread 0's is the sum).  Returns true in every thread of the last block.
template <int NV>
__device__ __forceinline__ bool grid_reduce(double (&v)[NV], DSum *part, unsigned *counter, double (&tot)[NV]) {
    __shared__ bool last;
    __shared__ double res[NV];
    block_reduce_plain<NV>(v);
    if (threadIdx.x == 0) {
        for (int k = 0; k < NV; ++k) part[static_cast<size_t>(blockIdx.x) * NV + k].s = v[k];
        unsigned t;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return false;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int k = w; k < NV; k += nw) {
        constexpr int kPer = (kMaxReduceBlocks + 31) / 32;
        double p[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const unsigned b = lane + 32 * i;
            p[i] = b < gridDim.x ? __ldcg(&part[static_cast<size_t>(b) * NV + k].s) : 0.0;
        }
        const double t = warp_sum_exact<kPer>(p);
        if (lane == 0) res[k] = t;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) tot[k] = res[k];
    if (threadIdx.x == 0) *counter = 0u;
    return true;
}

// This CTA's share of n items: contiguous (a grid-wide stride leaves some CTAs a whole trip more than
// others: 4 against 3 at 128^3, and takes a CTA's rows apart), walked with the CTA's threads.
// A grid may have 2^32 points: the share's place in the vectors is a 64-bit base, and its items are counted from
// there in 32 bits (64-bit counts in the loops: solve-101x75x53 855 -> 867 us).
struct Share {
    long long base;
    int begin, end;
};
__device__ __forceinline__ Share cta_share(long long n) {
    const long long base = n * blockIdx.x / gridDim.x;
    return Share{base, static_cast<int>(threadIdx.x), static_cast<int>(n * (blockIdx.x + 1) / gridDim.x - base)};
}
struct GridDiv {  // rows of nx values (or nx / 4 chunks), ny rows a plane
    FastDiv row, plane;
};
// The row of the share's item i and its place in that row of `len` items.
struct RowOf {
    int row0, x0;
    __device__ __forceinline__ RowOf(const Share &sh, int len, const FastDiv &by) {
        row0 = div_by_wide(static_cast<unsigned>(sh.base), by);
        x0 = static_cast<int>(sh.base - static_cast<long long>(row0) * len);
    }
    __device__ __forceinline__ void at(int i, int len, const FastDiv &by, int &row, int &x) const {
        const int t = x0 + i, dr = div_by(t, by);
        row = row0 + dr;
        x = t - dr * len;
    }
};

__device__ __forceinline__ double stencil7(const double *__restrict__ u, long long i, int x, int y, int z, int nx,
                                           int ny, int nz, long long np) {
    double nb = (x > 0) ? u[i - 1] : 0.0;
    if (x < nx - 1) nb += u[i + 1];
    if (y > 0) nb += u[i - nx];
    if (y < ny - 1) nb += u[i + nx];
    if (z > 0) nb += u[i - np];
    if (z < nz - 1) nb += u[i + np];
    return 6.0 * u[i] - nb;
}

// After the x/r update (last CTA, one thread): rr = ||r_new||^2, the iteration count, the residual
// history and, inside the CUDA graph that repeats the iteration, its loop condition.
__device__ __forceinline__ void finish_update(KrylovScalars *sc, double rr, cudaGraphConditionalHandle cond,
                                              int use_cond) {
    const int it = sc->it + 1;
    const double bb = sc->bb > 0.0 ? sc->bb : 1.0;
    int status = sc->status;
    if (!isfinite(rr)) sc->status = status = -6;
    if (use_cond) {
        const bool go = status == 0 && !(rr <= sc->tol2 * bb) && it < sc->maxit;
        cudaGraphSetConditional(cond, go ? 1u : 0u);
    }
    sc->rr = rr;
    sc->rho_prev = sc->rho;
    sc->restart = 0;
    sc->it = it;
    if (sc->hist != nullptr) sc->hist[it] = rr;  // the host takes sqrt(rr / bb)
}

// r = b - A x ; f0 = (S) r ; rr = ||r||^2 ; bb = ||b||^2 ; restart = 1.
template <class S>
__global__ void __launch_bounds__(kMaxThreads) k_init_residual(int nx, int ny, int nz, const double *__restrict__ b, const double *__restrict__ x,
                                double *__restrict__ r, S *__restrict__ f0, KrylovScalars *sc, DSum *part,
                                unsigned *counter, GridDiv gd) {
    const long long np = static_cast<long long>(nx) * ny;
    double a0 = 0.0, a1 = 0.0;
    const Share sh = cta_share(np * nz);
    const RowOf rows(sh, nx, gd.row);
    b += sh.base;
    x += sh.base;
    r += sh.base;
    if (f0 != nullptr) f0 += sh.base;
    for (int i = sh.begin; i < sh.end; i += blockDim.x) {
        int row, xx;
        rows.at(i, nx, gd.row, row, xx);
        const int zz = div_by(row, gd.plane), yy = row - zz * ny;
        const double bi = b[i];
        const double ri = bi - stencil7(x, i, xx, yy, zz, nx, ny, nz, np);
        r[i] = ri;
        if (f0 != nullptr) stv<S, double>(f0 + i, ri);
        a0 = fma(ri, ri, a0);
        a1 = fma(bi, bi, a1);
    }
    double v[2] = {a0, a1};
    double tot[2];
    if (grid_reduce<2>(v, part, counter, tot) && threadIdx.x == 0) {
        sc->rr = tot[0];
        sc->bb = tot[1];
        sc->restart = 1;
        sc->rho = tot[0];  // T = I: the first step's scalars
        sc->beta = 0.0;
        if (!isfinite(tot[0]) || !isfinite(tot[1])) sc->status = -6;
    }
}

// tt = ||b - A x||^2 (true residual).
__global__ void __launch_bounds__(kMaxThreads) k_true_residual(int nx, int ny, int nz, const double *__restrict__ b, const double *__restrict__ x,
                                KrylovScalars *sc, DSum *part, unsigned *counter, GridDiv gd) {
    const long long np = static_cast<long long>(nx) * ny;
    double a0 = 0.0;
    const Share sh = cta_share(np * nz);
    const RowOf rows(sh, nx, gd.row);
    b += sh.base;
    x += sh.base;
    for (int i = sh.begin; i < sh.end; i += blockDim.x) {
        int row, xx;
        rows.at(i, nx, gd.row, row, xx);
        const int zz = div_by(row, gd.plane), yy = row - zz * ny;
        const double ri = b[i] - stencil7(x, i, xx, yy, zz, nx, ny, nz, np);
        a0 = fma(ri, ri, a0);
    }
    double v[1] = {a0};
    double tot[1];
    if (grid_reduce<1>(v, part, counter, tot) && threadIdx.x == 0) sc->tt = tot[0];
}

// rho = (s, r), sdr = (s, r_k - r_{k-1}); beta by eq. (1), eq. (2) or 0.  r_k - r_{k-1} = -alpha A p of the
// step before, still in q: eq. (2)'s extra vector needs no storage of its own.
template <class S>
__global__ void __launch_bounds__(kMaxThreads) k_dots_beta(long long n, const S *__restrict__ s, const double *__restrict__ r,
                            const double *__restrict__ q, KrylovScalars *sc, DSum *part, unsigned *counter) {
    pdl_trigger();
    pdl_wait();
    const int variant = sc->variant;
    const bool need_sdr = (variant == 1) && (sc->restart == 0);
    double a0 = 0.0, a1 = 0.0;
    const Share sh = cta_share(n);
    s += sh.base;
    r += sh.base;
    q += sh.base;
    for (int i = sh.begin; i < sh.end; i += blockDim.x) {
        const double si = ldv<double>(s + i);
        a0 = fma(si, r[i], a0);
        if (need_sdr) a1 = fma(si, q[i], a1);
    }
    double v[2] = {a0, a1};
    double tot[2];
    if (grid_reduce<2>(v, part, counter, tot) && threadIdx.x == 0) finish_dots(sc, tot[0], tot[1]);
}

// T = I: after the x/r update, whose rr is the next rho and sq = (r, q) (flexible variant only), the next
// step's beta.  It is judged when that step begins (ident_status): the solve may be over.
__device__ __forceinline__ void ident_dots(KrylovScalars *sc, double sq) {
    const double rho = sc->rr, sdr = -sc->alpha * sq;
    sc->rho = rho;
    sc->sdr = sdr;
    sc->beta = sc->variant == 2 || sc->rho_prev == 0.0 ? 0.0 : (sc->variant == 0 ? rho : sdr) / sc->rho_prev;
}
__device__ __forceinline__ void ident_status(KrylovScalars *sc) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    if (sc->restart == 0 && sc->variant != 2 && sc->rho_prev == 0.0) sc->status = -4;
    if (!isfinite(sc->rho) || !isfinite(sc->beta)) sc->status = -6;
}

// p = s + beta p
template <class S, bool IDENT>
__global__ void __launch_bounds__(kMaxThreads) k_update_p(long long n, const S *__restrict__ s, double *__restrict__ p, KrylovScalars *sc) {
    pdl_trigger();
    pdl_wait();
    if constexpr (IDENT) ident_status(sc);
    const double beta = sc->beta;
    const Share sh = cta_share(n);
    s += sh.base;
    p += sh.base;
    for (int i = sh.begin; i < sh.end; i += blockDim.x) {
        const double si = ldv<double>(s + i);
        p[i] = (beta == 0.0) ? si : fma(beta, p[i], si);
    }
}

// q = A p ; pq = (p, q) ; alpha = rho / pq
__global__ void __launch_bounds__(kMaxThreads) k_spmv_alpha(int nx, int ny, int nz, const double *__restrict__ p, double *__restrict__ q,
                             KrylovScalars *sc, DSum *part, unsigned *counter, GridDiv gd) {
    pdl_trigger();
    pdl_wait();
    const long long np = static_cast<long long>(nx) * ny;
    double a0 = 0.0;
    const Share sh = cta_share(np * nz);
    const RowOf rows(sh, nx, gd.row);
    p += sh.base;
    q += sh.base;
    for (int i = sh.begin; i < sh.end; i += blockDim.x) {
        int row, xx;
        rows.at(i, nx, gd.row, row, xx);
        const int zz = div_by(row, gd.plane), yy = row - zz * ny;
        const double qi = stencil7(p, i, xx, yy, zz, nx, ny, nz, np);
        q[i] = qi;
        a0 = fma(p[i], qi, a0);
    }
    double v[1] = {a0};
    double tot[1];
    if (grid_reduce<1>(v, part, counter, tot) && threadIdx.x == 0) {
        const double pq = tot[0];
        sc->pq = pq;
        if (!(pq > 0.0)) {
            sc->status = (pq == pq) ? -4 : -6;
            sc->alpha = 0.0;
        } else {
            sc->alpha = sc->rho / pq;
        }
    }
}

// The x/r update's sums: rr, and for T = I (r, q).
template <bool IDENT>
__device__ __forceinline__ void finish_xr(double a0, double a1, KrylovScalars *sc, DSum *part, unsigned *counter,
                                          cudaGraphConditionalHandle cond, int use_cond) {
    if constexpr (IDENT) {
        double v[2] = {a0, a1}, tot[2];
        if (!grid_reduce<2>(v, part, counter, tot) || threadIdx.x != 0) return;
        finish_update(sc, tot[0], cond, use_cond);
        ident_dots(sc, tot[1]);
    } else {
        double v[1] = {a0}, tot[1];
        if (grid_reduce<1>(v, part, counter, tot) && threadIdx.x == 0) finish_update(sc, tot[0], cond, use_cond);
    }
}

// x += alpha p ; r_new = r - alpha q ; r = r_new ; f0 = (S) r_new ; rr = ||r_new||^2
template <class S, bool IDENT>
__global__ void __launch_bounds__(kMaxThreads) k_update_xr(long long n, double *__restrict__ x, const double *__restrict__ p, double *__restrict__ r,
                            const double *__restrict__ q, S *__restrict__ f0,
                            KrylovScalars *sc, DSum *part, unsigned *counter, cudaGraphConditionalHandle cond,
                            int use_cond) {
    pdl_trigger();
    pdl_wait();
    const double alpha = sc->alpha;
    const bool sq = IDENT && sc->variant == 1;
    double a0 = 0.0, a1 = 0.0;
    const Share sh = cta_share(n);
    x += sh.base;
    p += sh.base;
    r += sh.base;
    q += sh.base;
    if (f0 != nullptr) f0 += sh.base;
    for (int i = sh.begin; i < sh.end; i += blockDim.x) {
        x[i] = fma(alpha, p[i], x[i]);
        const double qi = q[i], rn = fma(-alpha, qi, r[i]);
        r[i] = rn;
        if (f0 != nullptr) stv<S, double>(f0 + i, rn);
        a0 = fma(rn, rn, a0);
        if (sq) a1 = fma(rn, qi, a1);
    }
    finish_xr<IDENT>(a0, a1, sc, part, counter, cond, use_cond);
}

// ---- the same four kernels on 4-element chunks ---------------------------------------------------
// Used when nx % 4 == 0 and every vector is 16-byte aligned: each thread moves four consecutive
// elements of a vector with 16-byte loads and stores (the element values, the operations on them
// and the order of the six neighbour terms of A p are those of the scalar kernels; only the
// assignment of elements to threads, and so the partial sums' grouping, differs).
__device__ __forceinline__ void ld4(double (&v)[4], const double *p) {
    const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4(double *p, const double (&v)[4]) {
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}
template <class S> __device__ __forceinline__ void lds4(double (&v)[4], const S *p);
template <> __device__ __forceinline__ void lds4<double>(double (&v)[4], const double *p) { ld4(v, p); }
template <> __device__ __forceinline__ void lds4<float>(double (&v)[4], const float *p) {
    const float4 a = reinterpret_cast<const float4 *>(p)[0];
    v[0] = widen_f32(a.x); v[1] = widen_f32(a.y); v[2] = widen_f32(a.z); v[3] = widen_f32(a.w);
}
template <> __device__ __forceinline__ void lds4<__nv_bfloat16>(double (&v)[4], const __nv_bfloat16 *p) {
    const uint2 a = reinterpret_cast<const uint2 *>(p)[0];
    const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162 *>(&a.x), hi = *reinterpret_cast<const __nv_bfloat162 *>(&a.y);
    v[0] = widen_f32(__low2float(lo)); v[1] = widen_f32(__high2float(lo));
    v[2] = widen_f32(__low2float(hi)); v[3] = widen_f32(__high2float(hi));
}
template <class S> __device__ __forceinline__ void sts4(S *p, const double (&v)[4]);
template <> __device__ __forceinline__ void sts4<double>(double *p, const double (&v)[4]) { st4(p, v); }
template <> __device__ __forceinline__ void sts4<float>(float *p, const double (&v)[4]) {
    reinterpret_cast<float4 *>(p)[0] = make_float4(narrow_f64(v[0]), narrow_f64(v[1]), narrow_f64(v[2]), narrow_f64(v[3]));
}
template <> __device__ __forceinline__ void sts4<__nv_bfloat16>(__nv_bfloat16 *p, const double (&v)[4]) {
    __nv_bfloat162 lo, hi;
    lo.x = __float2bfloat16_rn(narrow_f64(v[0])); lo.y = __float2bfloat16_rn(narrow_f64(v[1]));
    hi.x = __float2bfloat16_rn(narrow_f64(v[2])); hi.y = __float2bfloat16_rn(narrow_f64(v[3]));
    uint2 a;
    a.x = *reinterpret_cast<unsigned *>(&lo);
    a.y = *reinterpret_cast<unsigned *>(&hi);
    reinterpret_cast<uint2 *>(p)[0] = a;
}

// One chunk as stored: 16-byte words.
template <class S>
struct RawChunk {
    static constexpr int W = static_cast<int>(sizeof(S)) * 4 / 16 > 0 ? static_cast<int>(sizeof(S)) * 4 / 16 : 1;
    uint4 w[W];
};
template <>
struct RawChunk<__nv_bfloat16> {
    uint2 w[1];
};
template <class S>
__device__ __forceinline__ RawChunk<S> raw4(const S *p) {
    RawChunk<S> r;
    using Q = std::remove_reference_t<decltype(r.w[0])>;
#pragma unroll
    for (int i = 0; i < static_cast<int>(sizeof(r) / sizeof(Q)); ++i) r.w[i] = reinterpret_cast<const Q *>(p)[i];
    return r;
}
template <class S>
__device__ __forceinline__ void widen4(double (&v)[4], const RawChunk<S> &r) {
    lds4<S>(v, reinterpret_cast<const S *>(&r));
}

// (s, r) and, when wanted, (s, q) over this CTA's chunks; the next chunk is on its way while one is
// summed (3.4 chunks a thread at 128^3: a load's latency each otherwise).
template <class S>
__device__ __forceinline__ void dots_share(double &a0, double &a1, const Share &sh, const S *s, const double *r, const double *q,
                                           bool with_q) {
    if (sh.begin >= sh.end) return;
    s += 4 * sh.base;
    r += 4 * sh.base;
    q += 4 * sh.base;
    RawChunk<S> ns = raw4<S>(s + 4 * sh.begin);
    RawChunk<double> nr = raw4<double>(r + 4 * sh.begin), nq;
    if (with_q) nq = raw4<double>(q + 4 * sh.begin);
    for (int c = sh.begin; c < sh.end; c += blockDim.x) {
        const RawChunk<S> cs = ns;
        const RawChunk<double> cr = nr, cq = nq;
        const int n = c + static_cast<int>(blockDim.x);
        if (n < sh.end) {
            ns = raw4<S>(s + 4 * n);
            nr = raw4<double>(r + 4 * n);
            if (with_q) nq = raw4<double>(q + 4 * n);
        }
        double sv[4], v[4];
        widen4<S>(sv, cs);
        widen4<double>(v, cr);
#pragma unroll
        for (int k = 0; k < 4; ++k) a0 = fma(sv[k], v[k], a0);
        if (with_q) {
            widen4<double>(v, cq);
#pragma unroll
            for (int k = 0; k < 4; ++k) a1 = fma(sv[k], v[k], a1);
        }
    }
}

// p = s + beta p over this CTA's chunks (p = s when beta is 0: p may hold anything then).
template <class S>
__device__ __forceinline__ void update_p_share(const Share &sh, const S *s, double *p, double beta) {
    if (sh.begin >= sh.end) return;
    const bool keep = beta != 0.0;
    s += 4 * sh.base;
    p += 4 * sh.base;
    RawChunk<S> ns = raw4<S>(s + 4 * sh.begin);
    RawChunk<double> np;
    if (keep) np = raw4<double>(p + 4 * sh.begin);
    for (int c = sh.begin; c < sh.end; c += blockDim.x) {
        const RawChunk<S> cs = ns;
        const RawChunk<double> cp = np;
        const int n = c + static_cast<int>(blockDim.x);
        if (n < sh.end) {
            ns = raw4<S>(s + 4 * n);
            if (keep) np = raw4<double>(p + 4 * n);
        }
        double sv[4], pv[4];
        widen4<S>(sv, cs);
        if (keep) {
            widen4<double>(pv, cp);
#pragma unroll
            for (int k = 0; k < 4; ++k) sv[k] = fma(beta, pv[k], sv[k]);
        }
        st4(p + 4 * c, sv);
    }
}

template <class S>
__global__ void __launch_bounds__(kMaxThreads) k_dots_beta4(int nc, const S *__restrict__ s, const double *__restrict__ r,
                             const double *__restrict__ q, KrylovScalars *sc, DSum *part, unsigned *counter) {
    pdl_trigger();
    pdl_wait();
    const Share sh = cta_share(nc);
    const int variant = sc->variant;
    const bool need_sdr = (variant == 1) && (sc->restart == 0);
    double a0 = 0.0, a1 = 0.0;
    dots_share<S>(a0, a1, sh, s, r, q, need_sdr);
    double v[2] = {a0, a1};
    double tot[2];
    if (grid_reduce<2>(v, part, counter, tot) && threadIdx.x == 0) finish_dots(sc, tot[0], tot[1]);
}

template <class S, bool IDENT>
__global__ void __launch_bounds__(kMaxThreads) k_update_p4(int nc, const S *__restrict__ s, double *__restrict__ p, KrylovScalars *sc) {
    pdl_trigger();
    pdl_wait();
    if constexpr (IDENT) ident_status(sc);
    const Share sh = cta_share(nc);
    const double beta = sc->beta;
    update_p_share<S>(sh, s, p, beta);
}

// q = A p on four consecutive points of an x-row (nx % 4 == 0), the neighbour terms summed in the
// order of stencil7.
__global__ void __launch_bounds__(kMaxThreads) k_spmv_alpha4(int nx, int ny, int nz, const double *__restrict__ p, double *__restrict__ q,
                              KrylovScalars *sc, DSum *part, unsigned *counter, GridDiv gd) {
    pdl_trigger();
    pdl_wait();
    const int nq = nx >> 2, npi = nx * ny, nc = (npi >> 2) * nz;
    const Share sh = cta_share(nc);
    const RowOf rows(sh, nq, gd.row);
    p += 4 * sh.base;
    q += 4 * sh.base;
    double a0 = 0.0;
#pragma unroll 2
    for (int c = sh.begin; c < sh.end; c += blockDim.x) {
        int row, xq;
        rows.at(c, nq, gd.row, row, xq);
        const int zz = div_by(row, gd.plane), yy = row - zz * ny, xx = 4 * xq;
        const int i = 4 * c;
        double pc[4];
        ld4(pc, p + i);
        const double pl = (xx > 0) ? p[i - 1] : 0.0, pr = (xx + 4 < nx) ? p[i + 4] : 0.0;
        double nb[4] = {pl + pc[1], pc[0] + pc[2], pc[1] + pc[3], pc[2] + pr};
        double t[4];
        if (yy > 0) {
            ld4(t, p + i - nx);
#pragma unroll
            for (int k = 0; k < 4; ++k) nb[k] += t[k];
        }
        if (yy < ny - 1) {
            ld4(t, p + i + nx);
#pragma unroll
            for (int k = 0; k < 4; ++k) nb[k] += t[k];
        }
        if (zz > 0) {
            ld4(t, p + i - npi);
#pragma unroll
            for (int k = 0; k < 4; ++k) nb[k] += t[k];
        }
        if (zz < nz - 1) {
            ld4(t, p + i + npi);
#pragma unroll
            for (int k = 0; k < 4; ++k) nb[k] += t[k];
        }
        double qv[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            qv[k] = 6.0 * pc[k] - nb[k];
            a0 = fma(pc[k], qv[k], a0);
        }
        st4(q + i, qv);
    }
    double v[1] = {a0};
    double tot[1];
    if (grid_reduce<1>(v, part, counter, tot) && threadIdx.x == 0) {
        const double pq = tot[0];
        sc->pq = pq;
        if (!(pq > 0.0)) {
            sc->status = (pq == pq) ? -4 : -6;
            sc->alpha = 0.0;
        } else {
            sc->alpha = sc->rho / pq;
        }
    }
}

template <class S, bool IDENT>
__global__ void __launch_bounds__(kMaxThreads) k_update_xr4(int nc, double *__restrict__ x, const double *__restrict__ p, double *__restrict__ r,
                             const double *__restrict__ q, S *__restrict__ f0,
                             KrylovScalars *sc, DSum *part, unsigned *counter, cudaGraphConditionalHandle cond,
                             int use_cond) {
    pdl_trigger();
    pdl_wait();
    const Share sh = cta_share(nc);
    x += 4 * sh.base;
    p += 4 * sh.base;
    r += 4 * sh.base;
    q += 4 * sh.base;
    if (f0 != nullptr) f0 += 4 * sh.base;
    const double alpha = sc->alpha;
    const bool sq = IDENT && sc->variant == 1;
    double a0 = 0.0, a1 = 0.0;
#pragma unroll 2
    for (int c = sh.begin; c < sh.end; c += blockDim.x) {
        const int i = 4 * c;
        double xv[4], pv[4], ro[4], qv[4], rn[4];
        ld4(xv, x + i);
        ld4(pv, p + i);
        ld4(ro, r + i);
        ld4(qv, q + i);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            xv[k] = fma(alpha, pv[k], xv[k]);
            rn[k] = fma(-alpha, qv[k], ro[k]);
            a0 = fma(rn[k], rn[k], a0);
            if (sq) a1 = fma(rn[k], qv[k], a1);
        }
        st4(x + i, xv);
        st4(r + i, rn);
        if (f0 != nullptr) sts4<S>(f0 + i, rn);
    }
    finish_xr<IDENT>(a0, a1, sc, part, counter, cond, use_cond);
}

// ---- the four kernels above as one cooperative kernel ---------------------------------------------
// The iteration tail with three grid-wide barriers in place of three kernel boundaries: dots and
// beta | p update | q = A p and alpha | x, r update.  Same grid, same 4-element chunks per thread
// and the same last-CTA reductions as the separate kernels, so every value (partial sums
// included) is bit-identical to theirs.  Neighbour values of p are written by other CTAs in the
// p phase, so the stencil phase reads p through L2 (ld.global.cg).
__device__ __forceinline__ void ld4cg(double (&v)[4], const double *p) {
    const double2 a = __ldcg(reinterpret_cast<const double2 *>(p)), b = __ldcg(reinterpret_cast<const double2 *>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

template <class S>
__global__ void __launch_bounds__(kMaxThreads) k_tail_fused(int nx, int ny, int nz, const S *__restrict__ s, double *x,
                                                    double *r, double *p, double *q, S *f0,
                                                    KrylovScalars *sc, DSum *part, unsigned *counter, unsigned *bar,
                                                    long long spin_limit, cudaGraphConditionalHandle cond,
                                                    int use_cond, GridDiv gd) {
    const int nq = nx >> 2, npi = nx * ny, nc = (npi >> 2) * nz;
    const Share sh = cta_share(nc);
    unsigned *bcount = bar, *bgen = bar + 1;
    int *berr = reinterpret_cast<int *>(bar + 2);
    const unsigned nblk = gridDim.x;
    // A barrier wait that gave up ends this launch and stops the solve: the first CTA to see it
    // records SMG_ERR_TIMEOUT and ends the graph's loop (no x/r update completes then, so nothing
    // else sets the loop condition in this launch).
    auto give_up = [&]() {
        if (threadIdx.x == 0 && atomicCAS(bar + 3, 0u, 1u) == 0u) {
            sc->status = SMG_ERR_TIMEOUT;
            if (use_cond) cudaGraphSetConditional(cond, 0u);
        }
    };
    if (*reinterpret_cast<volatile int *>(berr) != 0) {  // an earlier launch of this solve gave up
        give_up();
        return;
    }
    // ---- rho = (s, r), sdr = (s, r - r_prev); beta ----
    {
        const int variant = sc->variant;
        const bool need_sdr = (variant == 1) && (sc->restart == 0);
        double a0 = 0.0, a1 = 0.0;
        dots_share<S>(a0, a1, sh, s, r, q, need_sdr);
        double v[2] = {a0, a1};
        double tot[2];
        if (grid_reduce<2>(v, part, counter, tot) && threadIdx.x == 0) finish_dots(sc, tot[0], tot[1]);
    }
    if (!grid_barrier(bcount, bgen, berr, spin_limit, nblk)) {
        give_up();
        return;
    }
    // ---- p = s + beta p ----
    {
        const double beta = __ldcg(&sc->beta);
        update_p_share<S>(sh, s, p, beta);
    }
    if (!grid_barrier(bcount, bgen, berr, spin_limit, nblk)) {
        give_up();
        return;
    }
    // ---- q = A p, pq = (p, q), alpha ----
    {
        const RowOf rows(sh, nq, gd.row);
        const long long to = 4 * sh.base;
        double a0 = 0.0;
#pragma unroll 2
        for (int c = sh.begin; c < sh.end; c += blockDim.x) {
            int row, xq;
            rows.at(c, nq, gd.row, row, xq);
            const int zz = div_by(row, gd.plane), yy = row - zz * ny, xx = 4 * xq;
            const long long i = to + 4 * c;
            double pc[4];
            ld4cg(pc, p + i);
            const double pl = (xx > 0) ? __ldcg(p + i - 1) : 0.0, pr = (xx + 4 < nx) ? __ldcg(p + i + 4) : 0.0;
            double nb[4] = {pl + pc[1], pc[0] + pc[2], pc[1] + pc[3], pc[2] + pr};
            double t[4];
            if (yy > 0) {
                ld4cg(t, p + i - nx);
#pragma unroll
                for (int k = 0; k < 4; ++k) nb[k] += t[k];
            }
            if (yy < ny - 1) {
                ld4cg(t, p + i + nx);
#pragma unroll
                for (int k = 0; k < 4; ++k) nb[k] += t[k];
            }
            if (zz > 0) {
                ld4cg(t, p + i - npi);
#pragma unroll
                for (int k = 0; k < 4; ++k) nb[k] += t[k];
            }
            if (zz < nz - 1) {
                ld4cg(t, p + i + npi);
#pragma unroll
                for (int k = 0; k < 4; ++k) nb[k] += t[k];
            }
            double qv[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                qv[k] = 6.0 * pc[k] - nb[k];
                a0 = fma(pc[k], qv[k], a0);
            }
            st4(q + i, qv);
        }
        double v[1] = {a0};
        double tot[1];
        if (grid_reduce<1>(v, part, counter, tot) && threadIdx.x == 0) {
            const double pq = tot[0];
            sc->pq = pq;
            if (!(pq > 0.0)) {
                sc->status = (pq == pq) ? -4 : -6;
                sc->alpha = 0.0;
            } else {
                sc->alpha = sc->rho / pq;
            }
        }
    }
    if (!grid_barrier(bcount, bgen, berr, spin_limit, nblk)) {
        give_up();
        return;
    }
    // ---- x += alpha p, r_new = r - alpha q, f0 = (S) r_new, rr ----
    {
        const double alpha = __ldcg(&sc->alpha);
        const long long to = 4 * sh.base;
        double a0 = 0.0;
#pragma unroll 2
        for (int c = sh.begin; c < sh.end; c += blockDim.x) {
            const long long i = to + 4 * c;
            double xv[4], pv[4], ro[4], qv[4], rn[4];
            ld4(xv, x + i);
            ld4(pv, p + i);
            ld4(ro, r + i);
            ld4(qv, q + i);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                xv[k] = fma(alpha, pv[k], xv[k]);
                rn[k] = fma(-alpha, qv[k], ro[k]);
                a0 = fma(rn[k], rn[k], a0);
            }
            st4(x + i, xv);
            st4(r + i, rn);
            if (f0 != nullptr) sts4<S>(f0 + i, rn);
        }
        double v[1] = {a0};
        double tot[1];
        if (grid_reduce<1>(v, part, counter, tot) && threadIdx.x == 0) finish_update(sc, tot[0], cond, use_cond);
    }
}

// ---- launchers --------------------------------------------------------------------------------
// Grid of the Krylov kernels over `items` elements or chunks: one CTA per SM, of as many threads as
// give every SM work (an FP64 unit serves its SM alone, so small grids are spread thin), 64 to 1024.
struct RedGrid {
    int blocks, threads;
};
RedGrid reduction_grid(long long items) {
    constexpr int kSMs = 152;
    long long t = (items + kSMs - 1) / kSMs;
    t = std::min<long long>(kMaxThreads, std::max<long long>(64, (t + 63) / 64 * 64));
    const long long b = std::max<long long>(1, std::min<long long>(kSMs, (items + t - 1) / t));
    return RedGrid{static_cast<int>(b), static_cast<int>(t)};
}

// Polls of a grid-barrier wait in the fused tail before it gives up (about a second).
constexpr long long kTailSpinLimit = 10000000;

// True when nb CTAs of the fused tail can all be resident on this device (cached per device).
template <class S>
bool fused_tail_fits(int nb) {
    static int per_sm[64] = {0};
    static int sms[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (per_sm[dev] == 0) {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_tail_fused<S>, kMaxThreads, 0) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        per_sm[dev] = b > 0 ? b : -1;
    }
    return per_sm[dev] > 0 && static_cast<long long>(per_sm[dev]) * sms[dev] >= nb;
}

#define SMG_PREC_SWITCH(storage, ...)                               \
    switch (storage) {                                              \
    case Prec::F64: { using S = double; __VA_ARGS__; break; }       \
    case Prec::F32: { using S = float; __VA_ARGS__; break; }        \
    case Prec::BF16: { using S = __nv_bfloat16; __VA_ARGS__; break; } \
    }

cudaError_t kry_init_residual(Prec st_prec, int nx, int ny, int nz, const double *b, const double *x, double *r,
                              void *f0, KrylovWork &w, cudaStream_t st) {
    const long long n = static_cast<long long>(nx) * ny * nz;
    const RedGrid g = reduction_grid(n);
    SMG_PREC_SWITCH(st_prec, k_init_residual<S><<<g.blocks, g.threads, 0, st>>>(nx, ny, nz, b, x, r, static_cast<S *>(f0),
                                                                      w.sc, w.part, w.counter, GridDiv{fast_div(nx), fast_div(ny)}));
    return cudaGetLastError();
}

cudaError_t kry_true_residual(int nx, int ny, int nz, const double *b, const double *x, KrylovWork &w,
                              cudaStream_t st) {
    const long long n = static_cast<long long>(nx) * ny * nz;
    const RedGrid g = reduction_grid(n);
    k_true_residual<<<g.blocks, g.threads, 0, st>>>(nx, ny, nz, b, x, w.sc, w.part, w.counter,
                                                        GridDiv{fast_div(nx), fast_div(ny)});
    return cudaGetLastError();
}

cudaError_t kry_iteration_tail(Prec st_prec, int nx, int ny, int nz, const void *s, double *x, double *r, double *p,
                               double *q, void *f0, KrylovWork &w, Dots dots, cudaStream_t st,
                               cudaGraphConditionalHandle cond, int use_cond) {
    const bool ident = dots == Dots::Ident;
    const long long n = static_cast<long long>(nx) * ny * nz;
    const RedGrid g1 = reduction_grid(n);
    cudaError_t e = cudaSuccess;
    auto al16 = [](const void *v) { return v == nullptr || (reinterpret_cast<uintptr_t>(v) & 15u) == 0; };
    if (nx % 4 == 0 && al16(s) && al16(x) && al16(r) && al16(p) && al16(q) && al16(f0)) {
        const int nc = static_cast<int>(n / 4);
        const RedGrid g4 = reduction_grid(nc);
        const GridDiv gd4{fast_div(nx / 4), fast_div(ny)};
        SMG_PREC_SWITCH(st_prec, {
            const S *sp = static_cast<const S *>(s);
            S *f0p = static_cast<S *>(f0);
            if (w.fused && dots == Dots::Kernel && w.bar != nullptr && fused_tail_fits<S>(g4.blocks)) {
                // one cooperative launch: the runtime refuses it unless every CTA is resident
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3(g4.blocks);
                cfg.blockDim = dim3(g4.threads);
                cfg.stream = st;
                cudaLaunchAttribute attr[1];
                attr[0].id = cudaLaunchAttributeCooperative;
                attr[0].val.cooperative = 1;
                cfg.attrs = attr;
                cfg.numAttrs = 1;
                e = cudaLaunchKernelEx(&cfg, k_tail_fused<S>, nx, ny, nz, sp, x, r, p, q, f0p, w.sc, w.part, w.counter,
                                       w.bar, static_cast<long long>(kTailSpinLimit), cond, use_cond, gd4);
                return e != cudaSuccess ? e : cudaGetLastError();
            }
            if (e == cudaSuccess && dots == Dots::Kernel) e = launch_pdl(k_dots_beta4<S>, dim3(g4.blocks), dim3(g4.threads), 0, st, nc, sp, r, q, w.sc, w.part, w.counter);
            if (e == cudaSuccess) e = launch_pdl(ident ? k_update_p4<S, true> : k_update_p4<S, false>, dim3(g4.blocks), dim3(g4.threads), 0, st, nc, sp, p, w.sc);
            if (e == cudaSuccess)
                e = launch_pdl(k_spmv_alpha4, dim3(g4.blocks), dim3(g4.threads), 0, st, nx, ny, nz, p, q, w.sc, w.part, w.counter, gd4);
            if (e == cudaSuccess)
                e = launch_pdl(ident ? k_update_xr4<S, true> : k_update_xr4<S, false>, dim3(g4.blocks), dim3(g4.threads), 0, st, nc, x, p, r, q, f0p, w.sc, w.part, w.counter,
                               cond, use_cond);
        });
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    const GridDiv gd{fast_div(nx), fast_div(ny)};
    SMG_PREC_SWITCH(st_prec, {
        const S *sp = static_cast<const S *>(s);
        S *f0p = static_cast<S *>(f0);
        if (e == cudaSuccess && dots == Dots::Kernel) e = launch_pdl(k_dots_beta<S>, dim3(g1.blocks), dim3(g1.threads), 0, st, n, sp, r, q, w.sc, w.part, w.counter);
        if (e == cudaSuccess) e = launch_pdl(ident ? k_update_p<S, true> : k_update_p<S, false>, dim3(g1.blocks), dim3(g1.threads), 0, st, n, sp, p, w.sc);
        if (e == cudaSuccess)
            e = launch_pdl(k_spmv_alpha, dim3(g1.blocks), dim3(g1.threads), 0, st, nx, ny, nz, p, q, w.sc, w.part, w.counter, gd);
        if (e == cudaSuccess)
            e = launch_pdl(ident ? k_update_xr<S, true> : k_update_xr<S, false>, dim3(g1.blocks), dim3(g1.threads), 0, st, n, x, p, r, q, f0p, w.sc, w.part, w.counter, cond,
                           use_cond);
    });
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace smg
