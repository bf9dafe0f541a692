// modal.cu -- the transforms of the x-lines into their sine eigenvectors and back, the prolongation in
// mode space, and the host side of the mode-space V-cycle (modal.cuh).
//
// Transform.  The orthonormal eigenvectors of tridiag(-1, 2, -1) of order n are
// s_k(x) = sqrt(2 / (n + 1)) sin(pi k x / (n + 1)), x, k = 1 .. n.  s_k is symmetric about the middle for
// odd k and antisymmetric for even k, so the line is folded first (x with n + 1 - x: sum and
// difference) and each parity is a product of half the order: n / 2 multiply-adds a point and
// transform, as two dense products over all lines.  No fast sine transform: n + 1 is 129, 257 or 1281
// for the sizes in use (few small factors), and at n <= 256 the product costs less than the passes
// over memory of a factored transform.
//
// A CTA of 128 threads forms TM x 16 lines by 32 modes of each parity; a thread holds TM lines x 4 modes
// of both parities.  FP32: bound by FFMA issue (64 FMAs to 12 shared-memory reads a step).
#include <cmath>
#include <cstring>

#include "modal.cuh"

namespace smg {

// ---- transforms -------------------------------------------------------------------------------------

constexpr int kBK = 16;      // lines of the product's inner dimension per stage
constexpr int kBN = 32;      // modes (or pairs of points) of a parity per CTA

template <class T> constexpr int tm_lines() { return 4; }

template <class T> __device__ __forceinline__ T in_val(double v);
template <> __device__ __forceinline__ float in_val<float>(double v) { return narrow_f64(v); }
template <> __device__ __forceinline__ double in_val<double>(double v) { return v; }
template <class S, class T> __device__ __forceinline__ S out_val(T v);
template <> __device__ __forceinline__ float out_val<float, float>(float v) { return v; }
template <> __device__ __forceinline__ double out_val<double, float>(float v) { return widen_f32(v); }
template <> __device__ __forceinline__ __nv_bfloat16 out_val<__nv_bfloat16, float>(float v) { return __float2bfloat16_rn(v); }
template <> __device__ __forceinline__ double out_val<double, double>(double v) { return v; }

struct SineArgs {
    int nx, ny, nz, pitch;   // pitch: lines per plane of the mode vectors (lines ny .. pitch-1 are zero)
    int nh;                  // odd modes, and pairs of points: ceil(nx / 2)
    int hp;                  // order of the stored matrices (nh rounded up to 32)
    const void *mat;         // [4][hp][hp]: by point odd, even; by mode odd, even
};

// One stage: acc[p][i][j] += sum_k A_p[k][line i] B_p[k][mode j] for both parities p.  In FP32 the stage's
// sum is formed apart and added once, which keeps the rounding error of a long line that of a short
// sum (128 points: 0.94e-7 of the result's norm instead of 1.5e-7, 1280: 1.5e-7).
template <class T, int TM>
__device__ __forceinline__ void sine_stage(T (&sum)[2][TM][4], const T *a0, const T *a1, const T *b0, const T *b1) {
    constexpr int LD = 16 * TM + 4;
    constexpr bool kApart = sizeof(T) == 4;
    T part[2][TM][4];
    T (&acc)[2][TM][4] = kApart ? part : sum;
    if constexpr (kApart) {
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) part[p][i][j] = T(0);
    }
#pragma unroll 4
    for (int k = 0; k < kBK; ++k) {
        T a[2][TM], b[2][4];
#pragma unroll
        for (int q = 0; q < TM / 4; ++q) {
            const V4<T> u = ld4(a0 + k * LD + 4 * q), v = ld4(a1 + k * LD + 4 * q);
            a[0][4 * q] = u.x, a[0][4 * q + 1] = u.y, a[0][4 * q + 2] = u.z, a[0][4 * q + 3] = u.w;
            a[1][4 * q] = v.x, a[1][4 * q + 1] = v.y, a[1][4 * q + 2] = v.z, a[1][4 * q + 3] = v.w;
        }
        const V4<T> u = ld4(b0 + k * kBN), v = ld4(b1 + k * kBN);
        b[0][0] = u.x, b[0][1] = u.y, b[0][2] = u.z, b[0][3] = u.w;
        b[1][0] = v.x, b[1][1] = v.y, b[1][2] = v.z, b[1][3] = v.w;
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[p][i][j] = fma(a[p][i], b[p][j], acc[p][i][j]);
    }
    if constexpr (kApart) {
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) sum[p][i][j] += part[p][i][j];
    }
}

template <class T, int TM>
struct SineSmem {
    static constexpr int BM = 16 * TM, LD = BM + 4;
    T a[2][2][kBK * LD];     // [buffer][parity]
    T b[2][2][kBK * kBN];
    long long off[BM];       // first element of each line in the physical vector, -1: none
};

template <class T, int TM>
__device__ __forceinline__ void line_offsets(SineSmem<T, TM> &s, const SineArgs &g, long long p0) {
    constexpr int BM = SineSmem<T, TM>::BM;
    for (int i = threadIdx.x; i < BM; i += blockDim.x) {
        const long long p = p0 + i;
        const unsigned z = static_cast<unsigned>(p / g.pitch), y = static_cast<unsigned>(p - static_cast<long long>(z) * g.pitch);
        s.off[i] = (p < static_cast<long long>(g.nz) * g.pitch && y < static_cast<unsigned>(g.ny))
                       ? (static_cast<long long>(z) * g.ny + y) * g.nx : -1;
    }
}

// Stage rows k0 .. k0+kBK-1 of both parities' matrices, columns c0 .. c0+kBN-1.
template <class T>
__device__ __forceinline__ void stage_matrix(T *b0, T *b1, const T *m0, const T *m1, int hp, int k0, int c0) {
    constexpr int PER = 16 / sizeof(T);
    for (int i = threadIdx.x; i < kBK * kBN / PER; i += blockDim.x) {
        const int r = i / (kBN / PER), c = (i % (kBN / PER)) * PER;
        const long long o = static_cast<long long>(k0 + r) * hp + c0 + c;
        *reinterpret_cast<uint4 *>(b0 + r * kBN + c) = *reinterpret_cast<const uint4 *>(m0 + o);
        *reinterpret_cast<uint4 *>(b1 + r * kBN + c) = *reinterpret_cast<const uint4 *>(m1 + o);
    }
}

// fhat[rhs][mode][line] = sum_x s_mode(x) f[rhs][line][x]; modes in the order odd, even.
template <class T>
__global__ void __launch_bounds__(128) sine_in_kernel(const __grid_constant__ SineArgs g, const double *__restrict__ f, T *__restrict__ out) {
    constexpr int TM = tm_lines<T>(), BM = 16 * TM, LD = BM + 4, NL = BM * kBK / 128;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SineSmem<T, TM> &s = *reinterpret_cast<SineSmem<T, TM> *>(smem_raw);
    pdl_trigger();
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const long long lines = static_cast<long long>(g.nz) * g.pitch, p0 = static_cast<long long>(blockIdx.x) * BM;
    const int c0 = blockIdx.y * kBN, ne = g.nx / 2;
    const T *m0 = static_cast<const T *>(g.mat), *m1 = m0 + static_cast<long long>(g.hp) * g.hp;
    const double *fr = f + static_cast<long long>(blockIdx.z) * g.nx * g.ny * g.nz;
    line_offsets(s, g, p0);
    stage_matrix(s.b[0][0], s.b[0][1], m0, m1, g.hp, 0, c0);
    pdl_wait();
    __syncthreads();
    const int lx = tid % kBK, ll = tid / kBK;   // this thread's point of a stage, first line of a stage
    double ra[NL], rb[NL];
    auto fetch = [&](int k0) {
        const int x = k0 + lx, xm = g.nx - 1 - x;
        const bool in = x < g.nh, two = in && xm != x;
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const long long o = s.off[ll + i * (128 / kBK)];
            ra[i] = (in && o >= 0) ? fr[o + x] : 0.0;
            rb[i] = (two && o >= 0) ? fr[o + xm] : 0.0;
        }
    };
    auto fold = [&](int buf, int k0) {
        const bool two = k0 + lx < ne;  // the middle point of an odd line has no partner: odd modes only
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const T u = in_val<T>(ra[i]), v = in_val<T>(rb[i]);
            s.a[buf][0][lx * LD + ll + i * (128 / kBK)] = u + v;
            s.a[buf][1][lx * LD + ll + i * (128 / kBK)] = two ? u - v : T(0);
        }
    };
    T acc[2][TM][4];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[p][i][j] = T(0);
    const int nk = (g.nh + kBK - 1) / kBK;
    fetch(0);
    fold(0, 0);
    __syncthreads();
    for (int kt = 0; kt < nk; ++kt) {
        const int cur = kt & 1;
        const bool more = kt + 1 < nk;
        if (more) {
            fetch((kt + 1) * kBK);
            stage_matrix(s.b[cur ^ 1][0], s.b[cur ^ 1][1], m0, m1, g.hp, (kt + 1) * kBK, c0);
        }
        sine_stage<T, TM>(acc, s.a[cur][0] + ty * TM, s.a[cur][1] + ty * TM, s.b[cur][0] + tx * 4, s.b[cur][1] + tx * 4);
        if (more) fold(cur ^ 1, (kt + 1) * kBK);
        __syncthreads();
    }
    T *o = out + static_cast<long long>(blockIdx.z) * g.nx * lines;
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = c0 + tx * 4 + j;
            if (c >= (p ? ne : g.nh)) continue;
            T *row = o + static_cast<long long>(p ? g.nh + c : c) * lines;
#pragma unroll
            for (int q = 0; q < TM / 4; ++q) {
                const long long ln = p0 + ty * TM + 4 * q;
                if (ln < lines) st4(row + ln, acc[p][4 * q][j], acc[p][4 * q + 1][j], acc[p][4 * q + 2][j], acc[p][4 * q + 3][j]);
            }
        }
}

// u[rhs][line][x] = sum_mode s_mode(x) uhat[rhs][mode][line]: both parities' sums for 32 points and their
// mirror images, sum and difference staged in shared memory so that lines are written whole words in x order.
template <class T, class S>
__global__ void __launch_bounds__(128) sine_out_kernel(const __grid_constant__ SineArgs g, const T *__restrict__ uh, S *__restrict__ u) {
    constexpr int TM = tm_lines<T>(), BM = 16 * TM, LD = BM + 4;
    constexpr int PER = 16 / sizeof(T), NA = kBK * BM / PER / 128;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SineSmem<T, TM> &s = *reinterpret_cast<SineSmem<T, TM> *>(smem_raw);
    pdl_trigger();
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const long long lines = static_cast<long long>(g.nz) * g.pitch, p0 = static_cast<long long>(blockIdx.x) * BM;
    const int c0 = blockIdx.y * kBN, ne = g.nx / 2;
    const long long hh = static_cast<long long>(g.hp) * g.hp;
    const T *m0 = static_cast<const T *>(g.mat) + 2 * hh, *m1 = m0 + hh;
    const T *in = uh + static_cast<long long>(blockIdx.z) * g.nx * lines;
    line_offsets(s, g, p0);
    stage_matrix(s.b[0][0], s.b[0][1], m0, m1, g.hp, 0, c0);
    pdl_wait();
    uint4 r[2][NA];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int e = tid + i * 128, k = k0 + e / (BM / PER);
            const long long ln = p0 + (e % (BM / PER)) * PER;
            const uint4 z = make_uint4(0u, 0u, 0u, 0u);
            r[0][i] = (k < g.nh && ln < lines) ? *reinterpret_cast<const uint4 *>(in + static_cast<long long>(k) * lines + ln) : z;
            r[1][i] = (k < ne && ln < lines) ? *reinterpret_cast<const uint4 *>(in + static_cast<long long>(g.nh + k) * lines + ln) : z;
        }
    };
    auto put = [&](int buf) {
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int e = tid + i * 128, at = (e / (BM / PER)) * LD + (e % (BM / PER)) * PER;
            *reinterpret_cast<uint4 *>(&s.a[buf][0][at]) = r[0][i];
            *reinterpret_cast<uint4 *>(&s.a[buf][1][at]) = r[1][i];
        }
    };
    T acc[2][TM][4];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[p][i][j] = T(0);
    const int nk = (g.nh + kBK - 1) / kBK;
    fetch(0);
    put(0);
    __syncthreads();
    for (int kt = 0; kt < nk; ++kt) {
        const int cur = kt & 1;
        const bool more = kt + 1 < nk;
        if (more) {
            fetch((kt + 1) * kBK);
            stage_matrix(s.b[cur ^ 1][0], s.b[cur ^ 1][1], m0, m1, g.hp, (kt + 1) * kBK, c0);
        }
        sine_stage<T, TM>(acc, s.a[cur][0] + ty * TM, s.a[cur][1] + ty * TM, s.b[cur][0] + tx * 4, s.b[cur][1] + tx * 4);
        if (more) put(cur ^ 1);
        __syncthreads();
    }
    // stage [line][x and mirror image] over the operand buffers (the last stage's reads are done)
    constexpr int LS = 2 * kBN + 1;
    static_assert(sizeof(T) * BM * LS <= sizeof(s.a), "the result tile fits over the operand buffers");
    T *w = &s.a[0][0][0];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            w[(ty * TM + i) * LS + tx * 4 + j] = acc[0][i][j] + acc[1][i][j];
            w[(ty * TM + i) * LS + kBN + tx * 4 + j] = acc[0][i][j] - acc[1][i][j];
        }
    __syncthreads();
    S *ur = u + static_cast<long long>(blockIdx.z) * g.nx * g.ny * g.nz;
    const int lane = tid & 31, x = c0 + lane;
    for (int i = tid >> 5; i < BM; i += 4) {
        const long long o = s.off[i];
        if (o < 0) continue;
        if (x < g.nh) ur[o + x] = out_val<S, T>(w[i * LS + lane]);
        if (x < ne) ur[o + g.nx - 1 - x] = out_val<S, T>(w[i * LS + kBN + lane]);
    }
}

// ---- prolongation and correction on a level above the tail -------------------------------------------

// u_l += P u_{l+1}, four lines a thread.  HBM: reads u_l and u_{l+1} once, writes u_l.
template <class T>
__global__ void __launch_bounds__(256) modal_prolong_kernel(const __grid_constant__ ModalArgs<T> A, int l) {
    pdl_trigger();
    pdl_wait();
    const int nz = A.nz[l], nzc = A.nz[l + 1], q = A.pitch / 4;
    const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= static_cast<long long>(nz) * q) return;
    const int z = static_cast<int>(i / q), y = static_cast<int>(i - static_cast<long long>(z) * q) * 4;
    const long long vec = static_cast<long long>(blockIdx.z) * A.nmode + blockIdx.y;
    T *u = A.u[l] + (vec * nz + z) * A.pitch + y;
    const T *uc = A.u[l + 1] + vec * nzc * A.pitch + y;
    V4<T> v = ld4(u);
    auto add = [&](int Z, T w) {
        const V4<T> c = ld4(uc + static_cast<long long>(Z) * A.pitch);
        v.x = fma(w, c.x, v.x);
        v.y = fma(w, c.y, v.y);
        v.z = fma(w, c.z, v.z);
        v.w = fma(w, c.w, v.w);
    };
    if (z & 1) {
        add(z >> 1, T(1));
    } else {
        const T *zc = A.zc + (A.plane_base[l] + z) * kCoefPerPlane;
        if (z > 0) add(z / 2 - 1, zc[6]);
        if (z / 2 < nzc) add(z / 2, zc[7]);
    }
    st4(u, v.x, v.y, v.z, v.w);
}

// ---- host -------------------------------------------------------------------------------------------

#define SMG_MODAL_CFG(MT, GG, KK) extern const ModalKernels<std::conditional_t<MT == 0, float, double>> modal_kernels_##MT##_##GG##_##KK
SMG_MODAL_CFG(0, 8, 4);
SMG_MODAL_CFG(0, 8, 8);
SMG_MODAL_CFG(0, 8, 16);
SMG_MODAL_CFG(0, 16, 16);
SMG_MODAL_CFG(0, 32, 16);
SMG_MODAL_CFG(1, 8, 4);
SMG_MODAL_CFG(1, 8, 8);
SMG_MODAL_CFG(1, 16, 8);
SMG_MODAL_CFG(1, 32, 8);
SMG_MODAL_CFG(1, 32, 16);

ModalConfig modal_config(int ny, bool f64) {
    if (ny <= 32) return {8, 4};
    if (ny <= 64) return {8, 8};
    if (ny <= 128) return f64 ? ModalConfig{16, 8} : ModalConfig{8, 16};
    if (ny <= 256) return f64 ? ModalConfig{32, 8} : ModalConfig{16, 16};
    return {32, 16};
}

template <>
const ModalKernels<float> &modal_kernels<float>(ModalConfig c) {
    if (c.K == 4) return modal_kernels_0_8_4;
    if (c.K == 8) return modal_kernels_0_8_8;
    if (c.G == 8) return modal_kernels_0_8_16;
    return c.G == 16 ? modal_kernels_0_16_16 : modal_kernels_0_32_16;
}
template <>
const ModalKernels<double> &modal_kernels<double>(ModalConfig c) {
    if (c.K == 4) return modal_kernels_1_8_4;
    if (c.K == 16) return modal_kernels_1_32_16;
    if (c.G == 8) return modal_kernels_1_8_8;
    return c.G == 16 ? modal_kernels_1_16_8 : modal_kernels_1_32_8;
}

// The 16 coefficients of line y of 2D level m of the plane with coefficient table pc (pairs (s, t) stand
// for s lambda + t): the diagonal, the couplings to lines y-1 and y+1, then for an even line its
// interpolation weights, for an odd line 2j+1 the restriction's multipliers of lines 2j-1, 2j+1, 2j+3 and
// the diagonal of coarse line j.
static void raw_line(const HostHierarchy &H, const double *pc, int m, int y, double *r) {
    auto line = [&](int mm, int yy) { return pc + static_cast<size_t>(H.line_base[mm] + yy) * kCoefPerLine; };
    const double *c = line(m, y);
    for (int i = 0; i < kRawPerLine; ++i) r[i] = 0.0;
    r[0] = c[1], r[1] = c[4], r[2] = c[0], r[3] = c[3], r[4] = c[2], r[5] = c[5];
    if (y % 2 == 0) {
        r[6] = c[6], r[7] = c[7];
        return;
    }
    const double *e0 = line(m, y - 1), *d = line(m + 1, y / 2);
    double w1 = 0.0;
    const double *e1 = nullptr;
    if (y + 1 < H.ny_m[m]) {
        e1 = line(m, y + 1);
        w1 = e1[6];
    }
    const double w0 = e0[7];
    r[6] = -w0 * e0[0], r[7] = -w0 * e0[3];
    r[8] = -(w0 * e0[2] + (e1 ? w1 * e1[0] : 0.0)), r[9] = -(w0 * e0[5] + (e1 ? w1 * e1[3] : 0.0));
    r[10] = e1 ? -w1 * e1[2] : 0.0, r[11] = e1 ? -w1 * e1[5] : 0.0;
    r[12] = d[1], r[13] = d[4];
}

void modal_free(ModalPlan &p) {
    cudaFree(p.d_args);
    cudaFree(p.d_buf);
    cudaFree(p.d_tab);
    cudaFree(p.d_sin);
    p = ModalPlan();
}

#define MCHK(call)                                \
    do {                                          \
        const cudaError_t e_ = (call);            \
        if (e_ != cudaSuccess) return static_cast<int>(e_); \
    } while (0)

namespace {

size_t up(size_t v, size_t to) { return (v + to - 1) / to * to; }

// Shared memory of the tail from level lt on (offsets into a), 0 when it does not fit.
template <class T>
size_t plan_tail(ModalArgs<T> &a, int lt, const ModalKernels<T> &k) {
    const size_t row = a.sm_pitch;
    size_t o = 0;
    int cls = 1;
    a.lt = lt;
    for (int l = lt; l < a.L; ++l) {
        a.sm_u[l] = static_cast<int>(o);
        o += row * a.nz[l];
        a.sm_f[l] = static_cast<int>(o);
        if (l > lt) o += row * a.nz[l];
        if (l + 1 < a.L) cls = std::max(cls, a.ncls[l]);
        if (o * sizeof(T) > kModalSmem) return 0;
    }
    a.sm_tab = static_cast<int>(up(o, 4));
    o = a.sm_tab + static_cast<size_t>(cls) * k.table_elems;
    const size_t planes = a.plane_base[a.L - 1] + 1 - a.plane_base[lt];
    a.sm_zc = static_cast<int>(o);
    o += planes * kCoefPerPlane;
    size_t b = up(o * sizeof(T), 16);
    a.sm_tab64 = static_cast<int>(b);
    b += static_cast<size_t>(k.table64_elems) * 8;
    a.sm_cls = static_cast<int>(b);
    b += up(planes, 16);
    return b <= kModalSmem ? b : 0;
}

template <class T>
int build(ModalPlan &p, ModalArgs<T> &a, const HostHierarchy &H) {
    const int nx = H.nx, L = H.L, nb = p.nb;
    const ModalKernels<T> &k = modal_kernels<T>(p.cfg);
    std::memset(&a, 0, sizeof(a));
    a.nmode = nx;
    a.ny = H.ny;
    a.pitch = p.pitch;
    a.L = L;
    a.P = H.P;
    a.sum_ny = H.sum_ny;
    a.npre = p.npre;
    a.npost = p.npost;
    a.coarse_iters = p.coarse_iters;
    for (int m = 0; m < H.P; ++m) a.ny_m[m] = H.ny_m[m], a.line_base[m] = H.line_base[m];
    a.sm_pitch = static_cast<int>(up(H.ny, p.cfg.K));
    // plane classes and their line coefficients
    std::vector<unsigned char> cls(H.nplanes_total);
    std::vector<T> raw, zc(H.zcoef.begin(), H.zcoef.end());
    std::vector<double> raw64(static_cast<size_t>(H.sum_ny) * kRawPerLine), lam(nx);
    int base = 0;
    for (int l = 0; l < L; ++l) {
        std::vector<int> slot, rep;
        a.nz[l] = H.nz_l[l];
        a.plane_base[l] = H.plane_base[l];
        a.cls_base[l] = base;
        a.ncls[l] = plane_classes(H, l, slot, rep);
        if (a.ncls[l] > 255) return static_cast<int>(cudaErrorNotSupported);
        base += a.ncls[l];
        for (int z = 0; z < a.nz[l]; ++z) cls[H.plane_base[l] + z] = static_cast<unsigned char>(slot[z]);
        for (int z : rep) {
            const double *pc = &H.pcoef[static_cast<size_t>(H.plane_base[l] + z) * H.sum_ny * kCoefPerLine];
            for (int m = 0; m < H.P; ++m)
                for (int y = 0; y < H.ny_m[m]; ++y) {
                    double r[kRawPerLine];
                    raw_line(H, pc, m, y, r);
                    for (double v : r) raw.push_back(static_cast<T>(v));
                    if (l == L - 1)
                        std::memcpy(&raw64[static_cast<size_t>(H.line_base[m] + y) * kRawPerLine], r, sizeof(r));
                }
        }
    }
    const double pi = 3.14159265358979323846;
    for (int q = 0; q < nx; ++q) {
        const int kk = q < p.nh ? 2 * q + 1 : 2 * (q - p.nh) + 2;
        const double s = std::sin(pi * kk / (2.0 * (nx + 1)));
        lam[q] = 4.0 * s * s;
    }
    // coefficients on the device
    const size_t b_zc = up(zc.size() * sizeof(T), 256), b_raw = up(raw.size() * sizeof(T), 256),
                 b_r64 = up(raw64.size() * 8, 256), b_lam = up(lam.size() * 8, 256), b_cls = up(cls.size(), 256);
    MCHK(cudaMalloc(&p.d_tab, b_zc + b_raw + b_r64 + b_lam + b_cls));
    unsigned char *d = static_cast<unsigned char *>(p.d_tab);
    auto put = [&](const void *src, size_t bytes, size_t room) {
        const cudaError_t e = cudaMemcpy(d, src, bytes, cudaMemcpyHostToDevice);
        d += room;
        return e;
    };
    a.zc = reinterpret_cast<const T *>(d);
    MCHK(put(zc.data(), zc.size() * sizeof(T), b_zc));
    a.raw = reinterpret_cast<const T *>(d);
    MCHK(put(raw.data(), raw.size() * sizeof(T), b_raw));
    a.raw64 = reinterpret_cast<const double *>(d);
    MCHK(put(raw64.data(), raw64.size() * 8, b_r64));
    a.lam = reinterpret_cast<const double *>(d);
    MCHK(put(lam.data(), lam.size() * 8, b_lam));
    a.cls = d;
    MCHK(put(cls.data(), cls.size(), b_cls));
    // transform matrices: by point (odd, even modes), then by mode
    const size_t hp = p.hp;
    std::vector<T> mat(4 * hp * hp, T(0));
    const double sc = std::sqrt(2.0 / (nx + 1));
    std::vector<double> sines(2 * (nx + 1));
    for (int i = 0; i < 2 * (nx + 1); ++i) sines[i] = sc * std::sin(pi * i / (nx + 1));
    for (int x = 0; x < p.nh; ++x)
        for (int q = 0; q < p.nh; ++q)
            for (int par = 0; par < 2; ++par) {
                if (par == 1 && (q >= nx / 2 || x >= nx / 2)) continue;
                const long long ph = static_cast<long long>(x + 1) * (2 * q + 1 + par) % (2 * (nx + 1));
                const T v = static_cast<T>(sines[ph]);
                mat[par * hp * hp + x * hp + q] = v;
                mat[(2 + par) * hp * hp + q * hp + x] = v;
            }
    MCHK(cudaMalloc(&p.d_sin, mat.size() * sizeof(T)));
    MCHK(cudaMemcpy(p.d_sin, mat.data(), mat.size() * sizeof(T), cudaMemcpyHostToDevice));
    // the first level whose coarser levels all fit in one CTA's shared memory
    p.smem = 0;
    for (p.lt = 0; p.lt < L; ++p.lt)
        if ((p.smem = plan_tail(a, p.lt, k)) != 0) break;
    if (p.smem == 0) return static_cast<int>(cudaErrorNotSupported);
    const int groups = (a.nz[p.lt] + 1) / 2, want = groups * p.cfg.G;
    p.threads = std::min(k.max_threads, std::max(128, (want + 31) / 32 * 32));
    // mode vectors: f and u of levels 0 .. lt
    size_t total = 0;
    std::vector<size_t> off;
    for (int l = 0; l <= p.lt; ++l)
        for (int t = 0; t < 2; ++t) {
            off.push_back(total);
            total += up(static_cast<size_t>(nb) * nx * a.nz[l] * a.pitch * sizeof(T), 256);
        }
    MCHK(cudaMalloc(&p.d_buf, total));
    unsigned char *bb = static_cast<unsigned char *>(p.d_buf);
    for (int l = 0; l <= p.lt; ++l) {
        a.fw[l] = reinterpret_cast<T *>(bb + off[2 * l]);
        a.f[l] = a.fw[l];
        a.u[l] = reinterpret_cast<T *>(bb + off[2 * l + 1]);
    }
    MCHK(cudaMalloc(&p.d_args, sizeof(a)));
    MCHK(cudaMemcpy(p.d_args, &a, sizeof(a), cudaMemcpyHostToDevice));
    return 0;
}

template <class T>
cudaError_t cycle(const ModalPlan &p, const ModalArgs<T> &a, int nb, cudaStream_t st, long long &launches) {
    const ModalKernels<T> &k = modal_kernels<T>(p.cfg);
    cudaError_t e;
    for (int l = 0; l < p.lt; ++l) {
        if (a.npre == 1 && k.slab_fits(a, l)) {
            if ((e = k.slab(a, l, nb, st)) != cudaSuccess) return e;
            launches += 1;
            continue;
        }
        for (int s = 0; s < a.npre; ++s)
            for (int c = 0; c < 2; ++c) {
                if ((e = k.relax(a, l, c, s == 0 ? c : 2, nb, st)) != cudaSuccess) return e;
                launches += 1;
            }
        if ((e = k.restrict_(a, l, nb, st)) != cudaSuccess) return e;
        launches += 1;
    }
    if ((e = k.tail(static_cast<const ModalArgs<T> *>(p.d_args), a.nmode, nb, p.threads, p.smem, st)) != cudaSuccess) return e;
    launches += 1;
    for (int l = p.lt - 1; l >= 0; --l) {
        const long long n = static_cast<long long>(a.nz[l]) * (a.pitch / 4);
        e = launch_pdl(modal_prolong_kernel<T>, dim3(static_cast<unsigned>((n + 255) / 256), a.nmode, nb), dim3(256), 0, st, a, l);
        if (e != cudaSuccess) return e;
        launches += 1;
        for (int s = 0; s < a.npost; ++s)
            for (int c = 1; c >= 0; --c) {
                if ((e = k.relax(a, l, c, 2, nb, st)) != cudaSuccess) return e;
                launches += 1;
            }
    }
    return cudaSuccess;
}

SineArgs sine_args(const ModalPlan &p) { return SineArgs{p.nx, p.ny, p.nz, p.pitch, p.nh, p.hp, p.d_sin}; }

template <class T>
dim3 sine_grid(const ModalPlan &p, int nb) {
    const long long lines = static_cast<long long>(p.nz) * p.pitch;
    constexpr int BM = 16 * tm_lines<T>();
    return dim3(static_cast<unsigned>((lines + BM - 1) / BM), (p.nh + kBN - 1) / kBN, nb);
}

template <class T>
cudaError_t sine_in(const ModalPlan &p, int nb, const double *f, T *out, cudaStream_t st) {
    constexpr size_t smem = sizeof(SineSmem<T, tm_lines<T>()>);
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&sine_in_kernel<T>), smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(sine_in_kernel<T>, sine_grid<T>(p, nb), dim3(128), smem, st, sine_args(p), f, out);
}
template <class T, class S>
cudaError_t sine_out(const ModalPlan &p, int nb, const T *uh, void *u, cudaStream_t st) {
    constexpr size_t smem = sizeof(SineSmem<T, tm_lines<T>()>);
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&sine_out_kernel<T, S>), smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(sine_out_kernel<T, S>, sine_grid<T>(p, nb), dim3(128), smem, st, sine_args(p), uh, static_cast<S *>(u));
}

}  // namespace

int modal_build(ModalPlan &p, const HostHierarchy &H, bool f64, int nb, int npre, int npost, int coarse_iters) {
    modal_free(p);
    p.f64 = f64;
    p.nx = H.nx, p.ny = H.ny, p.nz = H.nz, p.nb = nb, p.L = H.L;
    p.nh = (H.nx + 1) / 2;
    p.hp = static_cast<int>(up(p.nh, 32));
    p.npre = npre, p.npost = npost, p.coarse_iters = coarse_iters;
    p.pitch = static_cast<int>(up(H.ny, 4));
    p.cfg = modal_config(H.ny, f64);
    return f64 ? build<double>(p, p.a64, H) : build<float>(p, p.a32, H);
}

cudaError_t modal_transform_in(const ModalPlan &p, int nb, const double *f0, cudaStream_t st, long long &launches) {
    launches += 1;
    return p.f64 ? sine_in<double>(p, nb, f0, p.a64.fw[0], st) : sine_in<float>(p, nb, f0, p.a32.fw[0], st);
}

cudaError_t modal_cycle(const ModalPlan &p, int nb, cudaStream_t st, long long &launches) {
    return p.f64 ? cycle<double>(p, p.a64, nb, st, launches) : cycle<float>(p, p.a32, nb, st, launches);
}

cudaError_t modal_transform_out(const ModalPlan &p, int nb, Prec type, void *u0, cudaStream_t st, long long &launches) {
    launches += 1;
    if (p.f64) return sine_out<double, double>(p, nb, p.a64.u[0], u0, st);
    if (type == Prec::F64) return sine_out<float, double>(p, nb, p.a32.u[0], u0, st);
    if (type == Prec::BF16) return sine_out<float, __nv_bfloat16>(p, nb, p.a32.u[0], u0, st);
    return sine_out<float, float>(p, nb, p.a32.u[0], u0, st);
}

}  // namespace smg
