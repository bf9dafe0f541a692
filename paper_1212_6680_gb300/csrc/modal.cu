// modal.cu -- the transforms of the x-lines into their sine eigenvectors and back, the prolongation in
// mode space, and the host side of the mode-space V-cycle (modal.cuh).
//
// The FP32 transforms are in sine.cu; the FP64 ones here hold 4 lines by 4 modes of each parity a thread and are
// bound by FP64 issue.
#include <cmath>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "modal.cuh"

namespace smg {

// ---- transforms -------------------------------------------------------------------------------------

constexpr int kBK = 16;      // lines of the product's inner dimension per stage
constexpr int kBN = 32;      // modes (or pairs of points) of a parity per CTA

template <class T> constexpr int tm_lines() { return 4; }


// One stage: acc[p][i][j] += sum_k A_p[k][line i] B_p[k][mode j] for both parities p.
template <class T, int TM>
__device__ __forceinline__ void sine_stage(T (&acc)[2][TM][4], const T *a0, const T *a1, const T *b0, const T *b1) {
    constexpr int LD = 16 * TM + 4;
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
__device__ __forceinline__ void sine_in_body(const SineArgs &g, const double *__restrict__ fr, T *__restrict__ o, int line_tile, int mode_tile,
                                             unsigned char *smem_raw) {
    constexpr int TM = tm_lines<T>(), BM = 16 * TM, LD = BM + 4, NL = BM * kBK / 128;
    SineSmem<T, TM> &s = *reinterpret_cast<SineSmem<T, TM> *>(smem_raw);
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const long long lines = static_cast<long long>(g.nz) * g.pitch, p0 = static_cast<long long>(line_tile) * BM;
    const int c0 = mode_tile * kBN, ne = g.nx / 2;
    const T *m0 = static_cast<const T *>(g.mat), *m1 = m0 + static_cast<long long>(g.hp) * g.hp;
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
            const T u = ra[i], v = rb[i];
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

template <class T>
__global__ void __launch_bounds__(128) sine_in_kernel(const __grid_constant__ SineArgs g, const double *__restrict__ f, T *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_trigger();
    const long long rhs = blockIdx.z;
    sine_in_body<T>(g, f + rhs * g.nx * g.ny * g.nz, out + rhs * g.nx * g.nz * g.pitch, blockIdx.x, blockIdx.y, smem_raw);
}

// u[rhs][line][x] = sum_mode s_mode(x) uhat[rhs][mode][line]: both parities' sums for 32 points and their
// mirror images, sum and difference staged in shared memory so that lines are written whole words in x order.
template <class T, class S>
__device__ __forceinline__ void sine_out_body(const SineArgs &g, const T *__restrict__ in, S *__restrict__ ur, int line_tile, int mode_tile,
                                              unsigned char *smem_raw) {
    constexpr int TM = tm_lines<T>(), BM = 16 * TM, LD = BM + 4;
    constexpr int PER = 16 / sizeof(T), NA = kBK * BM / PER / 128;
    SineSmem<T, TM> &s = *reinterpret_cast<SineSmem<T, TM> *>(smem_raw);
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const long long lines = static_cast<long long>(g.nz) * g.pitch, p0 = static_cast<long long>(line_tile) * BM;
    const int c0 = mode_tile * kBN, ne = g.nx / 2;
    const long long hh = static_cast<long long>(g.hp) * g.hp;
    const T *m0 = static_cast<const T *>(g.mat) + 2 * hh, *m1 = m0 + hh;
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
    const int lane = tid & 31, x = c0 + lane;
    for (int i = tid >> 5; i < BM; i += 4) {
        const long long o = s.off[i];
        if (o < 0) continue;
        if (x < g.nh) ur[o + x] = static_cast<S>(w[i * LS + lane]);
        if (x < ne) ur[o + g.nx - 1 - x] = static_cast<S>(w[i * LS + kBN + lane]);
    }
}

template <class T, class S>
__global__ void __launch_bounds__(128) sine_out_kernel(const __grid_constant__ SineArgs g, const T *__restrict__ uh, S *__restrict__ u) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_trigger();
    const long long rhs = blockIdx.z;
    sine_out_body<T, S>(g, uh + rhs * g.nx * g.nz * g.pitch, u + rhs * g.nx * g.ny * g.nz, blockIdx.x, blockIdx.y, smem_raw);
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
        const T *zc = A.zt + A.ptype[A.plane_base[l] + z] * kCoefPerPlane;
        if (z > 0) add(z / 2 - 1, zc[6]);
        if (z / 2 < nzc) add(z / 2, zc[7]);
    }
    st4(u, v.x, v.y, v.z, v.w);
}

// ---- host -------------------------------------------------------------------------------------------

#define SMG_MODAL_CFG(MT, GG, KK) extern const ModalKernels<std::conditional_t<MT == 0, float, double>> modal_kernels_##MT##_##GG##_##KK
SMG_MODAL_CFG(0, 8, 4);
SMG_MODAL_CFG(0, 8, 8);
SMG_MODAL_CFG(0, 16, 8);
SMG_MODAL_CFG(0, 16, 16);
SMG_MODAL_CFG(0, 32, 16);
SMG_MODAL_CFG(1, 8, 4);
SMG_MODAL_CFG(1, 8, 8);
SMG_MODAL_CFG(1, 16, 8);
SMG_MODAL_CFG(1, 32, 8);
SMG_MODAL_CFG(1, 32, 16);

// Few lanes a plane leave more planes to a warp and fewer shuffles, few lines a lane a shorter chain and fewer
// registers: up to 128 lines 8 and 16 lanes.  The two splits of 129 to 256 lines, applications in us: FP32 16 x 16 / 32 x 8
// 256^3 645 / 669, 64x160x100 77 / 78, 64x256x64 71 / 70, 128x200x64 (1,1) 113 / 108; FP64 32 x 8 / 16 x 16 64x256x64 455 /
// 500, 100x256x200 2562 / 2485, 64x160x100 552 / 513, 128x200x64 (1,1) 1296 / 1218.
ModalConfig modal_config(int ny, bool f64) {
    if (ny <= 32) return {8, 4};
    if (ny <= 64) return {8, 8};
    if (ny <= 128) return {16, 8};
    if (ny <= 256) return f64 ? ModalConfig{32, 8} : ModalConfig{16, 16};
    return {32, 16};
}

template <>
const ModalKernels<float> &modal_kernels<float>(ModalConfig c) {
    if (c.K == 4) return modal_kernels_0_8_4;
    if (c.K == 8) return c.G == 8 ? modal_kernels_0_8_8 : modal_kernels_0_16_8;
    return c.G == 16 ? modal_kernels_0_16_16 : modal_kernels_0_32_16;
}
template <>
const ModalKernels<double> &modal_kernels<double>(ModalConfig c) {
    if (c.K == 4) return modal_kernels_1_8_4;
    if (c.K == 16) return modal_kernels_1_32_16;
    if (c.G == 8) return modal_kernels_1_8_8;
    return c.G == 16 ? modal_kernels_1_16_8 : modal_kernels_1_32_8;
}

// The coefficients of line y of 2D level m of the plane with coefficient table pc (pairs (s, t) stand for
// s lambda + t): the diagonal, the couplings to lines y-1 and y+1, then for an even line its
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
    cudaFree(p.d_buf);
    cudaFree(p.d_tab);
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
size_t plan_tail(ModalArgs<T> &a, int lt, ModalConfig cfg, const ModalKernels<T> &k) {
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
    auto elems = [&](int &at, size_t n) {
        at = static_cast<int>(o = up(o, 4));
        o += n;
    };
    elems(a.sm_tab, static_cast<size_t>(cls) * k.table_elems);
    elems(a.sm_stage, static_cast<size_t>(cls) * a.blk);
    elems(a.sm_zt, static_cast<size_t>(a.nptype) * kCoefPerPlane);
    size_t b = o * sizeof(T);
    auto bytes = [&](int &at, size_t n) {
        at = static_cast<int>(b = up(b, 16));
        b += n;
    };
    const int k6 = cfg.G * cfg.K / 32;  // Tab<32, k6>::kElems, and the level-0 couplings with one line a lane
    bytes(a.sm_tab64, sizeof(double) * (9 * 32 * (k6 - 1) + 1024 + 32 * k6 + (k6 == 1 ? 64 : 0)));
    bytes(a.sm_ltype, 2 * static_cast<size_t>(a.sum_ny));
    bytes(a.sm_ptype, 2 * static_cast<size_t>(a.plane_base[a.L - 1] + 1 - a.plane_base[lt]));
    bytes(a.sm_pcls, 2 * static_cast<size_t>(a.nptype));
    return b <= kModalSmem ? b : 0;
}

}  // namespace

// The tail's steps in order: tables of level lt; down, each level relaxed (npre sweeps of both colours) and
// restricted; the last level solved; up, each level corrected and relaxed (npost sweeps).  A level's classes are
// fetched while the step before its tables are spread runs.
template <class T>
std::vector<TailOp> tail_ops(const ModalArgs<T> &a) {
    const int L = a.L, lt = a.lt;
    std::vector<TailOp> ops;
    auto add = [&](int kind, int l) -> TailOp & {
        TailOp o{};
        const int c = l + 1 < L ? l + 1 : L - 1;
        o.kind = kind;
        o.level = l;
        o.nz = a.nz[l];
        o.nzc = a.nz[c];
        o.u = a.sm_u[l];
        o.f = l == lt ? -1 : a.sm_f[l];
        o.uc = a.sm_u[c];
        o.fc = a.sm_f[c];
        o.ptype = a.plane_base[l] - a.plane_base[lt];
        ops.push_back(o);
        return ops.back();
    };
    auto fetch = [&](TailOp &o, int l) {
        if (l < lt || l >= L - 1) return;
        o.fetch = a.cls_base[l] * a.blk;
        o.fetch_n = a.ncls[l] * a.blk;
    };
    auto relax = [&](int l, int colour, int mode) -> TailOp & {
        TailOp &o = add(OP_RELAX, l);
        o.colour = colour;
        o.mode = mode;
        o.n = colour ? a.nz[l] / 2 : (a.nz[l] + 1) / 2;
        return o;
    };
    TailOp &t = add(OP_TABLES, lt);
    if (lt < L - 1) t.spread = a.ncls[lt];
    for (int l = lt; l < L - 1; ++l) {
        for (int s = 0; s < a.npre; ++s)
            for (int c = 0; c < 2; ++c) {
                TailOp &o = relax(l, c, s == 0 ? c : 2);
                if (s == 0 && c == 0) fetch(o, l + 1);
            }
        TailOp &o = add(OP_RESTRICT, l);
        if (l + 1 < L - 1) o.spread = a.ncls[l + 1];
    }
    TailOp &solve = add(OP_COARSEST, L - 1);
    if (a.npost > 0) fetch(solve, L - 2);
    for (int l = L - 2; l >= lt; --l) {
        TailOp &o = add(OP_PROLONG, l);
        o.out = l == lt && a.npost == 0;
        if (a.npost > 0) o.spread = a.ncls[l];
        for (int s = 0; s < a.npost; ++s)
            for (int c = 1; c >= 0; --c) {
                TailOp &r = relax(l, c, 2);
                if (s == 0 && c == 1) fetch(r, l - 1);
            }
        if (l == lt && a.npost > 0) add(OP_STORE, l).out = 1;
    }
    add(OP_END, lt);
    return ops;
}

ModalShape modal_shape(const HostHierarchy &H) {
    ModalShape s;
    // plane classes; plane types: planes with equal coefficients and class
    s.ptype.resize(H.nplanes_total);
    std::vector<const double *> reps;  // each class's plane table
    std::map<std::string, int> seen;
    for (int l = 0; l < H.L; ++l) {
        std::vector<int> slot, rep;
        s.cls_base[l] = static_cast<int>(reps.size());
        s.ncls[l] = plane_classes(H, l, slot, rep);
        for (int z = 0; z < H.nz_l[l]; ++z) {
            const double *zc = &H.zcoef[static_cast<size_t>(H.plane_base[l] + z) * kCoefPerPlane];
            std::string key(reinterpret_cast<const char *>(zc), sizeof(double) * kCoefPerPlane);
            key.append(reinterpret_cast<const char *>(&slot[z]), sizeof(int));
            const auto it = seen.emplace(key, static_cast<int>(seen.size()));
            if (it.second) {
                s.zt.insert(s.zt.end(), zc, zc + kCoefPerPlane);
                s.pcls.push_back(static_cast<unsigned short>(slot[z]));
            }
            s.ptype[H.plane_base[l] + z] = static_cast<unsigned short>(it.first->second);
        }
        for (int z : rep) reps.push_back(&H.pcoef[static_cast<size_t>(H.plane_base[l] + z) * H.sum_ny * kCoefPerLine]);
    }
    s.ncls_all = static_cast<int>(reps.size());
    // line types: lines with equal coefficients in every class
    s.ltype.resize(H.sum_ny);
    std::vector<std::vector<double>> rows;  // [type][class][kRawPerLine]
    seen.clear();
    for (int m = 0; m < H.P; ++m)
        for (int y = 0; y < H.ny_m[m]; ++y) {
            std::vector<double> r(reps.size() * kRawPerLine);
            for (size_t c = 0; c < reps.size(); ++c) raw_line(H, reps[c], m, y, &r[c * kRawPerLine]);
            const auto it = seen.emplace(std::string(reinterpret_cast<const char *>(r.data()), r.size() * sizeof(double)),
                                         static_cast<int>(rows.size()));
            if (it.second) rows.push_back(std::move(r));
            s.ltype[H.line_base[m] + y] = static_cast<unsigned short>(it.first->second);
        }
    s.ntype = static_cast<int>(rows.size());
    s.raw.resize(static_cast<size_t>(s.ncls_all) * s.ntype * kRawPerLine);
    for (int t = 0; t < s.ntype; ++t)
        for (int c = 0; c < s.ncls_all; ++c)
            std::memcpy(&s.raw[(static_cast<size_t>(c) * s.ntype + t) * kRawPerLine], &rows[t][static_cast<size_t>(c) * kRawPerLine],
                        kRawPerLine * sizeof(double));
    const double pi = 3.14159265358979323846;
    const int nh = (H.nx + 1) / 2;
    s.lam.resize(H.nx);
    for (int q = 0; q < H.nx; ++q) {
        const int kk = q < nh ? 2 * q + 1 : 2 * (q - nh) + 2;
        const double v = std::sin(pi * kk / (2.0 * (H.nx + 1)));
        s.lam[q] = 4.0 * v * v;
    }
    return s;
}

template <class T>
void modal_vectors(ModalHost<T> &h, int nb) {
    const ModalArgs<T> &a = h.a;
    h.vec_bytes = 0;
    h.vec_off.clear();
    for (int l = 0; l <= a.lt; ++l)
        for (int t = 0; t < 2; ++t) {
            h.vec_off.push_back(h.vec_bytes);
            h.vec_bytes += up(static_cast<size_t>(nb) * a.nmode * a.nz[l] * a.pitch * sizeof(T), 256);
        }
}

template <class T>
int modal_plan(ModalHost<T> &h, const HostHierarchy &H, const ModalShape &s, ModalConfig cfg, int npre, int npost) {
    const int L = H.L;
    h.cfg = cfg;
    ModalArgs<T> &a = h.a;
    std::memset(&a, 0, sizeof(a));
    a.nmode = H.nx;
    a.ny = H.ny;
    a.pitch = static_cast<int>(up(H.ny, 4));
    a.L = L;
    a.P = H.P;
    a.sum_ny = H.sum_ny;
    a.npre = npre;
    a.npost = npost;
    for (int m = 0; m < H.P; ++m) a.ny_m[m] = H.ny_m[m], a.line_base[m] = H.line_base[m];
    a.sm_pitch = static_cast<int>(up(H.ny, cfg.K));
    for (int l = 0; l < L; ++l) {
        a.nz[l] = H.nz_l[l];
        a.plane_base[l] = H.plane_base[l];
        a.cls_base[l] = s.cls_base[l];
        a.ncls[l] = s.ncls[l];
    }
    a.ncls_all = s.ncls_all;
    a.nptype = static_cast<int>(s.pcls.size());
    a.ntype = s.ntype;
    a.blk = a.ntype * kRow + cfg.G * cfg.G;
    const std::vector<T> zt(s.zt.begin(), s.zt.end());
    const size_t sizes[] = {s.raw.size() * 8, s.lam.size() * 8, zt.size() * sizeof(T), s.ptype.size() * 2, s.pcls.size() * 2, s.ltype.size() * 2};
    const void *const src[] = {s.raw.data(), s.lam.data(), zt.data(), s.ptype.data(), s.pcls.data(), s.ltype.data()};
    size_t o = 0;
    for (int i = 0; i < 6; ++i) {
        h.at[i] = o;
        o += up(sizes[i], 256);
    }
    h.shared.assign(o, 0);
    for (int i = 0; i < 6; ++i) std::memcpy(h.shared.data() + h.at[i], src[i], sizes[i]);
    h.coef_values = static_cast<size_t>(a.nmode) * a.ncls_all * a.blk;
    h.coef64_values = static_cast<size_t>(a.nmode) * (a.ntype * kRow + 1024);
    // the first level whose coarser levels all fit in one CTA's shared memory
    const ModalKernels<T> &k = modal_kernels<T>(cfg);
    h.smem = 0;
    for (int lt = 0; lt < L && h.smem == 0; ++lt) h.smem = plan_tail(a, lt, cfg, k);
    if (h.smem == 0) return static_cast<int>(cudaErrorNotSupported);
    const std::vector<TailOp> ops = tail_ops(a);
    h.at[6] = h.shared.size();
    h.shared.resize(h.at[6] + up(ops.size() * sizeof(TailOp), 256), 0);
    std::memcpy(h.shared.data() + h.at[6], ops.data(), ops.size() * sizeof(TailOp));
    return 0;
}

template <class T>
void modal_place(ModalHost<T> &h, unsigned char *shared, T *coef, double *coef64, unsigned char *vec) {
    ModalArgs<T> &a = h.a;
    a.raw = reinterpret_cast<const double *>(shared + h.at[0]);
    a.lam = reinterpret_cast<const double *>(shared + h.at[1]);
    a.zt = reinterpret_cast<const T *>(shared + h.at[2]);
    a.ptype = reinterpret_cast<const unsigned short *>(shared + h.at[3]);
    a.pcls = reinterpret_cast<const unsigned short *>(shared + h.at[4]);
    a.ltype = reinterpret_cast<const unsigned short *>(shared + h.at[5]);
    a.ops = reinterpret_cast<const TailOp *>(shared + h.at[6]);
    a.coef64 = coef64;
    a.coef = coef;
    for (int l = 0; l <= a.lt; ++l) {
        a.fw[l] = reinterpret_cast<T *>(vec + h.vec_off[2 * l]);
        a.f[l] = a.fw[l];
        a.u[l] = reinterpret_cast<T *>(vec + h.vec_off[2 * l + 1]);
    }
}

std::vector<double> sine_table(int nx) {
    const double pi = 3.14159265358979323846, sc = std::sqrt(2.0 / (nx + 1));
    std::vector<double> sines(2 * (nx + 1));
    for (int i = 0; i < 2 * (nx + 1); ++i) sines[i] = sc * std::sin(pi * i / (nx + 1));
    return sines;
}

// The four matrices from the sines of one period, zero in the padding.  HBM: writes them once (on the host they took
// 6.5 ms at 2048 points, and their copy as long again).
template <class T>
__global__ void __launch_bounds__(256) sine_matrices_kernel(int nx, int nh, int hp, const double *__restrict__ sines, T *__restrict__ mat) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y, par = blockIdx.z & 1;
    if (c >= hp) return;
    const int x = blockIdx.z < 2 ? r : c, q = blockIdx.z < 2 ? c : r;  // by point, then by mode
    const int n = par ? nx / 2 : nh;
    T v = T(0);
    if (x < n && q < n) v = static_cast<T>(sines[(x + 1) * (2 * q + 1 + par) % (2 * (nx + 1))]);
    mat[(static_cast<long long>(blockIdx.z) * hp + r) * hp + c] = v;
}
template <class T>
cudaError_t launch_sine_matrices(int nx, const double *sines, T *mat, cudaStream_t st) {
    const int nh = (nx + 1) / 2, hp = sine_order(nx);
    sine_matrices_kernel<T><<<dim3((hp + 255) / 256, hp, 4), 256, 0, st>>>(nx, nh, hp, sines, mat);
    return cudaGetLastError();
}

int modal_tail_threads(size_t smem, long long ctas, int num_sms, int most, int planes, int G) {
    if (ctas > num_sms) {
        if (4 * (smem + 2048) <= kModalSmem) most = std::min(most, 128);
        else if (2 * (smem + 2048) <= kModalSmem) most = std::min(most, 256);
    }
    const int want = (planes + 1) / 2 * G;
    return std::min(most, std::max(128, (want + 31) / 32 * 32));
}

template int modal_plan<float>(ModalHost<float> &, const HostHierarchy &, const ModalShape &, ModalConfig, int, int);
template void modal_vectors<float>(ModalHost<float> &, int);
template void modal_place<float>(ModalHost<float> &, unsigned char *, float *, double *, unsigned char *);
template cudaError_t launch_sine_matrices<float>(int, const double *, float *, cudaStream_t);

namespace {

// Vectors for nb right-hand sides in place of those there are, and the tables unless they are there: one block with
// what is copied (shared data, arguments, sines) first, then what is formed there (coefficients, transform matrices).
template <class T>
int build(ModalPlan &p, ModalHost<T> &h, const HostHierarchy &H, const ModalShape &s, int nb, int npre, int npost) {
    const bool fresh = p.d_tab == nullptr;
    if (fresh)
        if (int e = modal_plan<T>(h, H, s, modal_config(H.ny, sizeof(T) == 8), npre, npost)) return e;
    p.nb = 0;
    cudaFree(p.d_buf);
    p.d_buf = nullptr;
    modal_vectors<T>(h, nb);
    MCHK(cudaMalloc(&p.d_buf, h.vec_bytes));
    unsigned char *const vec = static_cast<unsigned char *>(p.d_buf);
    if (fresh) {
        const std::vector<double> sines = sine_table(H.nx);
        const int hp = sine_order(H.nx);
        p.at_args = h.shared.size();
        const size_t at_sines = p.at_args + up(sizeof(h.a), 256), at_64 = at_sines + up(sines.size() * sizeof(double), 256);
        const size_t at_coef = at_64 + up(h.coef64_values * 8, 256), at_mat = at_coef + up(h.coef_values * sizeof(T), 256);
        MCHK(cudaMalloc(&p.d_tab, at_mat + 4 * sizeof(T) * hp * hp));
        unsigned char *const d = static_cast<unsigned char *>(p.d_tab);
        double *const c64 = reinterpret_cast<double *>(d + at_64);
        T *const coef = reinterpret_cast<T *>(d + at_coef), *const mat = reinterpret_cast<T *>(d + at_mat);
        modal_place<T>(h, d, coef, c64, vec);
        h.shared.resize(at_64, 0);
        std::memcpy(h.shared.data() + p.at_args, &h.a, sizeof(h.a));
        std::memcpy(h.shared.data() + at_sines, sines.data(), sines.size() * sizeof(double));
        MCHK(cudaMemcpy(d, h.shared.data(), h.shared.size(), cudaMemcpyHostToDevice));
        MCHK(launch_sine_matrices<T>(H.nx, reinterpret_cast<const double *>(d + at_sines), mat, 0));
        const ModalKernels<T> &k = modal_kernels<T>(h.cfg);
        MCHK(k.setup(h.a, coef, c64, 0));
        p.sine = SineArgs{H.nx, H.ny, H.nz, h.a.pitch, (H.nx + 1) / 2, hp, mat};
        int dev = 0;
        MCHK(cudaGetDevice(&dev));
        MCHK(cudaDeviceGetAttribute(&p.num_sms, cudaDevAttrMultiProcessorCount, dev));
    } else {
        unsigned char *const d = static_cast<unsigned char *>(p.d_tab);
        modal_place<T>(h, d, const_cast<T *>(h.a.coef), const_cast<double *>(h.a.coef64), vec);
        MCHK(cudaMemcpy(d + p.at_args, &h.a, sizeof(h.a), cudaMemcpyHostToDevice));
    }
    MCHK(cudaStreamSynchronize(0));  // the set-up kernels: callers' streams need not wait for the default one
    p.nb = nb;
    return 0;
}

template <class T>
cudaError_t prolong(const ModalArgs<T> &a, int l, int nb, cudaStream_t st) {
    const long long n = static_cast<long long>(a.nz[l]) * (a.pitch / 4);
    return launch_pdl(modal_prolong_kernel<T>, dim3(static_cast<unsigned>((n + 255) / 256), a.nmode, nb), dim3(256), 0, st, a, l);
}

template <class T>
cudaError_t cycle(const ModalPlan &p, const ModalHost<T> &h, int nb, int coarse_iters, cudaStream_t st, long long &launches) {
    const ModalArgs<T> &a = h.a;
    const ModalKernels<T> &k = modal_kernels<T>(h.cfg);
    cudaError_t e;
    for (int l = 0; l < a.lt; ++l) {
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
    const int threads = modal_tail_threads(h.smem, static_cast<long long>(a.nmode) * nb, p.num_sms, k.max_threads, a.nz[a.lt], h.cfg.G);
    if ((e = k.tail(reinterpret_cast<const ModalArgs<T> *>(static_cast<const unsigned char *>(p.d_tab) + p.at_args), a.nmode, nb, coarse_iters, threads, h.smem, st)) != cudaSuccess)
        return e;
    launches += 1;
    for (int l = a.lt - 1; l >= 0; --l) {
        if ((e = prolong(a, l, nb, st)) != cudaSuccess) return e;
        launches += 1;
        for (int s = 0; s < a.npost; ++s)
            for (int c = 1; c >= 0; --c) {
                if ((e = k.relax(a, l, c, 2, nb, st)) != cudaSuccess) return e;
                launches += 1;
            }
    }
    return cudaSuccess;
}

template <class T>
dim3 sine_grid(const ModalPlan &p, int nb) {
    const long long lines = static_cast<long long>(p.sine.nz) * p.sine.pitch;
    constexpr int BM = 16 * tm_lines<T>();
    return dim3(static_cast<unsigned>((lines + BM - 1) / BM), (p.sine.nh + kBN - 1) / kBN, nb);
}

// Shared memory of a transform's CTAs: so much that no SM takes more of them than its share.  Launched beside the
// kernel before it, they settle on the SMs that come free first, three or four together, and there share an
// FP64 unit that one of them already fills (applications at 294x11x30 923 -> 415 us, 570x13x16 1643 -> 744 us, 255x90x10
// 829 -> 369 us).  Not for few tiles of one or two stages, where it matters more that they can start
// beside the kernel before (46x79x16 (1,1) 238 us, 261 spread).
size_t sine_smem(const ModalPlan &p, dim3 g, size_t need) {
    constexpr size_t kPerSm = 228 * 1024, kPerCta = 1024;  // of an SM; reserved with each CTA
    const size_t tiles = static_cast<size_t>(g.x) * g.y * g.z, sms = p.num_sms;
    if (p.sine.nh <= 2 * kBK && 4 * tiles <= sms) return need;
    return std::max<size_t>(need, kPerSm / ((tiles + sms - 1) / sms + 1) - kPerCta + 128);
}

template <class T>
cudaError_t sine_in(const ModalPlan &p, int nb, const double *f, T *out, cudaStream_t st) {
    const size_t smem = sine_smem(p, sine_grid<T>(p, nb), sizeof(SineSmem<T, tm_lines<T>()>));
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&sine_in_kernel<T>), smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(sine_in_kernel<T>, sine_grid<T>(p, nb), dim3(128), smem, st, p.sine, f, out);
}
template <class T, class S>
cudaError_t sine_out(const ModalPlan &p, int nb, const T *uh, void *u, cudaStream_t st) {
    const size_t smem = sine_smem(p, sine_grid<T>(p, nb), sizeof(SineSmem<T, tm_lines<T>()>));
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&sine_out_kernel<T, S>), smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(sine_out_kernel<T, S>, sine_grid<T>(p, nb), dim3(128), smem, st, p.sine, uh, static_cast<S *>(u));
}

}  // namespace

int modal_build(ModalPlan &p, const HostHierarchy &H, const ModalShape &s, bool f64, int nb, int npre, int npost) {
    if (p.d_tab != nullptr && p.f64 != f64) modal_free(p);
    p.f64 = f64;
    return f64 ? build<double>(p, p.h64, H, s, nb, npre, npost) : build<float>(p, p.h32, H, s, nb, npre, npost);
}

cudaError_t modal_transform_in(const ModalPlan &p, int nb, Prec type, const void *f0, cudaStream_t st, long long &launches) {
    // long lines are folded into the iterate's place first: nothing of it is needed yet
    if (!p.f64) return sine_in_f32(p.sine, nb, type, f0, p.h32.a.fw[0], p.h32.a.u[0], st, launches);
    launches += 1;
    return sine_in<double>(p, nb, static_cast<const double *>(f0), p.h64.a.fw[0], st);
}

cudaError_t modal_cycle(const ModalPlan &p, int nb, int coarse_iters, cudaStream_t st, long long &launches) {
    return p.f64 ? cycle<double>(p, p.h64, nb, coarse_iters, st, launches) : cycle<float>(p, p.h32, nb, coarse_iters, st, launches);
}

cudaError_t modal_transform_out(const ModalPlan &p, int nb, Prec value, Prec type, void *u0, cudaStream_t st, long long &launches) {
    if (!p.f64) return sine_out_f32(p.sine, nb, p.h32.a.u[0], value, type, u0, st, launches);
    launches += 1;
    return sine_out<double, double>(p, nb, p.h64.a.u[0], u0, st);
}

cudaError_t launch_modal_prolong(const ModalArgs<float> &a, int l, int nb, cudaStream_t st) { return prolong(a, l, nb, st); }

}  // namespace smg
