// modal.cuh -- the SMG V-cycle (section "Preconditioning with SMG" of arXiv:1212.6680) in the sine
// eigenvectors of the x-lines.
//
// Every x-line matrix of the cycle is S Lx + T I with one and the same Lx = tridiag(-1, 2, -1), and
// every coupling between lines and planes is of that form too.  In the orthonormal sine basis of the
// x-direction (Lx v_k = lambda_k v_k) an exact line solve is a division by S lambda_k + T, a coupling
// a multiplication, and the modes k do not couple at all: the V-cycle is nx independent 2D (y, z)
// cycles between two dense transforms of the x-lines (modal.cu).  The same linear operator as the
// plane kernels' in exact arithmetic, step by step the same relaxations.  What it removes is the
// serial chain of a line solve (elimination, five rounds of cyclic reduction, back substitution) in
// each of a plane's 4P - 3 dependent steps, and the CTA barrier between them.  One application at
// 128^3: 672 -> 119 us (FP32), 2352 -> 1018 us (FP64); 256^3 FP32 2154 -> 829 us; 1280x80x80 FP32
// 3802 -> 1441 us; 24x20x16 FP32 135 -> 27 us.
//
// One CTA runs the whole cycle of one mode in shared memory (modal_tail); levels whose planes do
// not fit there run as launches over global memory first (modal_slab, or the single steps).
//
// One plane of one mode is a vector of ny values.  G lanes hold K consecutive lines each
// (G K >= ny, both powers of two), and the plane's y-cycle runs in registers:
//   * coarse line i of level m+1 is line 2i+1 of level m, so a lane's K lines hold K/2 lines of the
//     next level, and so on: the first log2 K levels need a shuffle only at the lane borders, the
//     rest has one line per lane (level log2 K + t at lanes 2^t - 1 (mod 2^t));
//   * right-hand sides are kept divided by the line's diagonal (gi = g / (S lambda + T)), which
//     turns each relaxation into two FMAs a line and makes the first even sweep the identity;
//   * the lines' multipliers come from a table in shared memory, laid out so that a group's lanes
//     read consecutive words; planes with equal coefficients (plane_classes) share one.
// Lines past the end have zero multipliers, so no step tests for them.
#pragma once

#include "modal.h"
#include "plane_relax.cuh"

namespace smg {

template <class T> struct V4 { T x, y, z, w; };
__device__ __forceinline__ V4<float> ld4(const float *p) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    return V4<float>{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ V4<double> ld4(const double *p) {
    const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    return V4<double>{a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ void st4(float *p, float x, float y, float z, float w) {
    *reinterpret_cast<float4 *>(p) = make_float4(x, y, z, w);
}
__device__ __forceinline__ void st4(double *p, double x, double y, double z, double w) {
    reinterpret_cast<double2 *>(p)[0] = make_double2(x, y);
    reinterpret_cast<double2 *>(p)[1] = make_double2(z, w);
}

constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n / 2); }

// Layout of one plane class's line table (elements of T).  In-register level m (K >> m lines a lane):
// per even line {a-, a+, wm, wp}, per odd line {a-, a+, ca, cc} and cb; level log2 K + t: the same per
// lane.  a-, a+: couplings over the diagonal; wm, wp: interpolation weights; ca, cb, cc: the
// restriction from lines 2j-1, 2j+1, 2j+3 to coarse line j, over the coarse line's diagonal.
template <int G, int K>
struct Tab {
    static constexpr int M0 = ilog2(K), TM = ilog2(G);
    static constexpr int quad(int m) { return m == 0 ? 0 : quad(m - 1) + (K >> (m - 1)) * G; }
    static constexpr int even(int m) { return 4 * quad(m); }
    static constexpr int odd(int m) { return 4 * (quad(m) + (K >> m) / 2 * G); }
    static constexpr int cross(int t) { return 4 * (quad(M0) + t * G); }
    static constexpr int kScal = 4 * (quad(M0) + (TM + 1) * G);
    static constexpr int scal(int m) { return m == 0 ? kScal : scal(m - 1) + (K >> (m - 1)) / 2 * G; }
    static constexpr int xscal(int t) { return scal(M0) + t * G; }
    static constexpr int kInv = kScal + (scal(M0) - kScal) + (TM + 1) * G;
    static constexpr int kElems = (kInv + K * G + 3) / 4 * 4;
    static constexpr int kEntries = quad(M0) + (TM + 1) * G;
    // reciprocal diagonal of line lane K + j of level 0: four lines of a lane together
    __host__ __device__ static constexpr int inv(int lane, int j) {
        return kInv + (K >= 4 ? ((j / 4) * G + lane) * 4 + (j & 3) : j * G + lane);
    }
};

// Entry e of the table of one plane class for the mode with eigenvalue lam.
template <class T, int G, int K>
__device__ __forceinline__ void table_entry(T *tab, const T *__restrict__ raw, const T lam, const int *ny_m,
                                            const int *line_base, const int P, int e) {
    using L = Tab<G, K>;
    int m = 0, n = K, lane, j = 0, y, t = -1;
    while (n > 1 && e >= n * G) {
        e -= n * G;
        ++m;
        n >>= 1;
    }
    bool line = true;
    if (n > 1) {
        y = e;
        lane = e / n;
        j = e - lane * n;
    } else {
        t = e / G;
        lane = e - t * G;
        m += t;
        line = ((lane + 1) & ((1 << t) - 1)) == 0;
        y = ((lane + 1) >> t) - 1;
    }
    T inv = T(0), am = T(0), ap = T(0), p = T(0), q = T(0), cb = T(0);
    const bool is_odd = (y & 1) != 0;
    if (line && m < P && y < ny_m[m]) {
        const T *r = raw + static_cast<long long>(line_base[m] + y) * kRawPerLine;
        const V4<T> r0 = ld4(r), r1 = ld4(r + 4);
        inv = T(1) / fma(r0.x, lam, r0.y);
        am = fma(r0.z, lam, r0.w) * inv;
        ap = fma(r1.x, lam, r1.y) * inv;
        if (is_odd) {
            const V4<T> r2 = ld4(r + 8), r3 = ld4(r + 12);
            const T ic = T(1) / fma(r3.x, lam, r3.y);
            p = fma(r1.z, lam, r1.w) * ic;
            cb = fma(r2.x, lam, r2.y) * ic;
            q = fma(r2.z, lam, r2.w) * ic;
        } else {
            p = r1.z;
            q = r1.w;
        }
    }
    if (t < 0) {
        const int i = j >> 1;
        const int base4 = 4 * ((m == 0 ? 0 : 2 * G * (K - (K >> m))) + ((j & 1) ? n / 2 * G : 0) + i * G + lane);
        st4(tab + base4, am, ap, p, q);
        if (j & 1) tab[L::kScal + G * (K - (K >> m)) + i * G + lane] = cb;
    } else {
        st4(tab + L::cross(0) + 4 * (t * G + lane), am, ap, p, q);
        tab[L::xscal(0) + t * G + lane] = cb;
    }
    if (m == 0) tab[L::inv(lane, j)] = inv;
}

// Shuffles within a group of G lanes; at the group's ends they return the lane's own value, which the
// zero multiplier of the missing neighbour removes.
template <class T, int G>
__device__ __forceinline__ T up(T v, int s) { return __shfl_up_sync(0xffffffffu, v, s, G); }
template <class T, int G>
__device__ __forceinline__ T dn(T v, int s) { return __shfl_down_sync(0xffffffffu, v, s, G); }

// The y-cycle from level log2 K on (one line per lane): gi in, the correction out.
template <class T, int G, int K>
__device__ __forceinline__ T ycycle_cross(T gi0, const T *tab, int ln) {
    using L = Tab<G, K>;
    T gi[L::TM + 1];
    gi[0] = gi0;
#pragma unroll
    for (int t = 0; t < L::TM; ++t) {
        const int s = 1 << t;
        const V4<T> c = ld4(tab + L::cross(t) + 4 * ln);
        const T cb = tab[L::xscal(t) + ln];
        const T o = gi[t] - c.x * up<T, G>(gi[t], s) - c.y * dn<T, G>(gi[t], s);
        gi[t + 1] = c.z * up<T, G>(o, 2 * s) + cb * o + c.w * dn<T, G>(o, 2 * s);
    }
    T c = gi[L::TM];
#pragma unroll
    for (int t = L::TM - 1; t >= 0; --t) {
        const int s = 1 << t;
        const V4<T> k = ld4(tab + L::cross(t) + 4 * ln);
        const T v = gi[t] + k.z * up<T, G>(c, s) + k.w * dn<T, G>(c, s);       // even lines + P c
        const T o = gi[t] - k.x * up<T, G>(v, s) - k.y * dn<T, G>(v, s);       // odd lines
        const T e = gi[t] - k.x * up<T, G>(o, s) - k.y * dn<T, G>(o, s);       // even lines again
        c = (((ln + 1) >> t) & 1) ? e : o;
    }
    return c;
}

// The y-cycle from in-register level M on: g (right-hand sides over the diagonals) in, the
// correction out.  Down: even lines (zero neighbours), odd lines, restriction (the residual is zero on
// odd lines); up: odd lines against the corrected even ones, then even lines.
template <class T, int G, int K, int M>
__device__ __forceinline__ void ycycle(T (&g)[(K >> M)], const T *tab, int ln) {
    using L = Tab<G, K>;
    constexpr int N = K >> M;
    if constexpr (N == 1) {
        g[0] = ycycle_cross<T, G, K>(g[0], tab, ln);
    } else {
        constexpr int H = N / 2;
        T c[H];
        {
            T o[H];
            const T nx = dn<T, G>(g[0], 1);
            T ca[H], cc[H];
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const V4<T> k = ld4(tab + L::odd(M) + 4 * (i * G + ln));
                o[i] = g[2 * i + 1] - k.x * g[2 * i] - k.y * (i + 1 < H ? g[(2 * i + 2) % N] : nx);
                ca[i] = k.z;
                cc[i] = k.w;
            }
            const T po = up<T, G>(o[H - 1], 1), no = dn<T, G>(o[0], 1);
#pragma unroll
            for (int i = 0; i < H; ++i)
                c[i] = ca[i] * (i > 0 ? o[(i + H - 1) % H] : po) + tab[L::scal(M) + i * G + ln] * o[i] +
                       cc[i] * (i + 1 < H ? o[(i + 1) % H] : no);
        }
        ycycle<T, G, K, M + 1>(c, tab, ln);
        T v[H];
        {
            const T pc = up<T, G>(c[H - 1], 1);
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const V4<T> k = ld4(tab + L::even(M) + 4 * (i * G + ln));
                v[i] = g[2 * i] + k.z * (i > 0 ? c[(i + H - 1) % H] : pc) + k.w * c[i];
            }
            const T nv = dn<T, G>(v[0], 1);
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const V4<T> k = ld4(tab + L::odd(M) + 4 * (i * G + ln));
                g[2 * i + 1] = g[2 * i + 1] - k.x * v[i] - k.y * (i + 1 < H ? v[(i + 1) % H] : nv);
            }
            const T po = up<T, G>(g[N - 1], 1);
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const V4<T> k = ld4(tab + L::even(M) + 4 * (i * G + ln));
                g[2 * i] = g[2 * i] - k.x * (i > 0 ? g[(2 * i + N - 1) % N] : po) - k.y * g[2 * i + 1];
            }
        }
    }
}

// A plane's row of lines in shared memory keeps lane ln's 16-byte chunks at positions XOR-ed with
// bits of ln, so that the eight lanes of a load phase touch every bank once (a lane's K lines are
// K sizeof(T) bytes apart from the next lane's).
template <class T, int K>
struct RowMap {
    static constexpr int CH = 16 / static_cast<int>(sizeof(T));
    static constexpr int CPL = K / CH;   // chunks a lane
    __device__ static __forceinline__ int chunk(int c) { return c ^ ((c >> 3) & (CPL - 1)); }
    __device__ static __forceinline__ int elem(int y) { return chunk(y / CH) * CH + y % CH; }
};

template <class T, int K, bool SM>
__device__ __forceinline__ void load_row(T (&v)[K], const T *row, int ln, int pitch) {
    using R = RowMap<T, K>;
    union U { uint4 c; T t[R::CH]; };
#pragma unroll
    for (int q = 0; q < R::CPL; ++q) {
        const int c = ln * R::CPL + q;
        U u;
        u.c = make_uint4(0u, 0u, 0u, 0u);
        if (c * R::CH < pitch) u.c = reinterpret_cast<const uint4 *>(row)[SM ? R::chunk(c) : c];
#pragma unroll
        for (int j = 0; j < R::CH; ++j) v[q * R::CH + j] = u.t[j];
    }
}
template <class T, int K, bool SM>
__device__ __forceinline__ void store_row(T *row, const T (&v)[K], int ln, int pitch) {
    using R = RowMap<T, K>;
    union U { uint4 c; T t[R::CH]; };
#pragma unroll
    for (int q = 0; q < R::CPL; ++q) {
        const int c = ln * R::CPL + q;
        U u;
#pragma unroll
        for (int j = 0; j < R::CH; ++j) u.t[j] = v[q * R::CH + j];
        if (c * R::CH < pitch) reinterpret_cast<uint4 *>(row)[SM ? R::chunk(c) : c] = u.c;
    }
}

// The vectors of one mode a step works on: u and f rows in shared (SM) or global memory.
template <class T>
struct Rows {
    T *p;
    int pitch, z0;   // lines per row; the plane the first row holds
    __device__ __forceinline__ T *at(int z) const { return p + static_cast<long long>(z - z0) * pitch; }
};

// One plane's part of f - sum (M (lambda + Ly) + Kc) u, on a row u (zero where the plane is absent).
// Ly u is formed from first differences, which are exact where u is smooth, before it meets M: on
// coarse z-levels M / Kc grows like 4^l while u is dominated by smooth lines, and M (4 u) - M (u + u) - ...
// would leave a rounding error of eps M u, white over the lines of this one mode, in a residual of
// size Kc u (FP32, 128^3: a cycle's error against FP64 1.4e-6 instead of 2.6e-7).  For the same reason
// lambda is not merged into the other coefficients, which are dyadic away from the boundary.
template <class T, int G, int K>
__device__ __forceinline__ void couple(T (&g)[K], const T (&u)[K], T M, T Kc, T lam, bool in_plane, int ln) {
#pragma unroll
    for (int j = 0; j < K; ++j) g[j] = fma(-Kc, u[j], g[j]);
    if (!in_plane) return;  // M = 0 on every plane of the launch
    T ul = up<T, G>(u[K - 1], 1), ur = dn<T, G>(u[0], 1);
    if (ln == 0) ul = T(0);
    if (ln == G - 1) ur = T(0);
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const T d = (u[j] - (j > 0 ? u[(j + K - 1) % K] : ul)) + (u[j] - (j + 1 < K ? u[(j + 1) % K] : ur));
        g[j] = fma(-M, fma(lam, u[j], d), g[j]);
    }
}
template <class T, int K>
__device__ __forceinline__ void zero_row(T (&v)[K]) {
#pragma unroll
    for (int j = 0; j < K; ++j) v[j] = T(0);
}

// Relaxation of plane z: u_z = C_z (f - A u)_z (modes 0 and 1: the own plane is zero, mode 0: all
// planes are) or u_z += (mode 2).  cross: the couplings between planes have an in-plane part (all
// levels but the finest).  The result stays in g.
template <class T, int G, int K, bool SMU, bool SMF>
__device__ __forceinline__ void relax_plane(T (&g)[K], const Rows<T> &u, const Rows<T> &f, int z, int nz, const T *zc,
                                            const T *tab, T lam, int mode, bool cross, int ln) {
    load_row<T, K, SMF>(g, f.at(z), ln, f.pitch);
    if (mode > 0) {
        T v[K];
        if (z > 0) load_row<T, K, SMU>(v, u.at(z - 1), ln, u.pitch);
        else zero_row<T, K>(v);
        couple<T, G, K>(g, v, zc[0], zc[3], lam, cross, ln);
        if (z + 1 < nz) load_row<T, K, SMU>(v, u.at(z + 1), ln, u.pitch);
        else zero_row<T, K>(v);
        couple<T, G, K>(g, v, zc[2], zc[5], lam, cross, ln);
        if (mode == 2) {
            load_row<T, K, SMU>(v, u.at(z), ln, u.pitch);
            couple<T, G, K>(g, v, zc[1], zc[4], lam, true, ln);
        }
    }
    using L = Tab<G, K>;
#pragma unroll
    for (int q = 0; q < K / 4; ++q) {
        const V4<T> i4 = ld4(tab + L::kInv + (q * G + ln) * 4);
        g[4 * q] *= i4.x;
        g[4 * q + 1] *= i4.y;
        g[4 * q + 2] *= i4.z;
        g[4 * q + 3] *= i4.w;
    }
    ycycle<T, G, K, 0>(g, tab, ln);
    if (mode == 2) {
        T v[K];
        load_row<T, K, SMU>(v, u.at(z), ln, u.pitch);
#pragma unroll
        for (int j = 0; j < K; ++j) g[j] += v[j];
    }
}

// Coarse plane Z's right-hand side P^T (f - A u): the residuals of planes 2Z, 2Z+1 and 2Z+2 with the
// weights of P, as one combination of five planes of u and three of f.  zc_level: plane 0's row.
template <class T, int G, int K, bool SMU, bool SMF>
__device__ __forceinline__ void restrict_plane(T (&g)[K], const Rows<T> &u, const Rows<T> &f, int Z, int nz,
                                               const T *zc_level, T lam, bool cross, int ln) {
    const int o = 2 * Z + 1;
    const T *zo = zc_level + o * kCoefPerPlane, *z0 = zo - kCoefPerPlane, *z1 = zo + kCoefPerPlane;
    const bool h1 = o + 1 < nz;
    const T w0 = z0[7], w1 = h1 ? z1[6] : T(0);
    T v[K];
    load_row<T, K, SMF>(g, f.at(o), ln, f.pitch);
    load_row<T, K, SMF>(v, f.at(o - 1), ln, f.pitch);
#pragma unroll
    for (int j = 0; j < K; ++j) g[j] = fma(w0, v[j], g[j]);
    if (h1) {
        load_row<T, K, SMF>(v, f.at(o + 1), ln, f.pitch);
#pragma unroll
        for (int j = 0; j < K; ++j) g[j] = fma(w1, v[j], g[j]);
    }
    if (Z > 0) load_row<T, K, SMU>(v, u.at(o - 2), ln, u.pitch);
    else zero_row<T, K>(v);
    couple<T, G, K>(g, v, w0 * z0[0], w0 * z0[3], lam, cross, ln);
    load_row<T, K, SMU>(v, u.at(o - 1), ln, u.pitch);
    couple<T, G, K>(g, v, fma(w0, z0[1], zo[0]), fma(w0, z0[4], zo[3]), lam, true, ln);
    load_row<T, K, SMU>(v, u.at(o), ln, u.pitch);
    couple<T, G, K>(g, v, zo[1] + w0 * z0[2] + (h1 ? w1 * z1[0] : T(0)), zo[4] + w0 * z0[5] + (h1 ? w1 * z1[3] : T(0)),
                    lam, true, ln);
    if (h1) load_row<T, K, SMU>(v, u.at(o + 1), ln, u.pitch);
    else zero_row<T, K>(v);
    couple<T, G, K>(g, v, h1 ? fma(w1, z1[1], zo[2]) : T(0), h1 ? fma(w1, z1[4], zo[5]) : T(0), lam, true, ln);
    const bool h2 = o + 2 < nz;
    if (h2) load_row<T, K, SMU>(v, u.at(o + 2), ln, u.pitch);
    else zero_row<T, K>(v);
    couple<T, G, K>(g, v, h2 ? w1 * z1[2] : T(0), h2 ? w1 * z1[5] : T(0), lam, cross, ln);
}

// The coarsest level: its one plane in FP64 by one warp (C steps of u += C (f - A u)).
template <class T, int G, int K, bool SM>
__device__ __forceinline__ void coarsest(const T *frow, T *urow, int ny, int iters, const double *tab, int lane) {
    constexpr int K6 = G * K / 32;
    using L = Tab<32, K6>;
    double fi[K6], u[K6], g[K6];
#pragma unroll
    for (int j = 0; j < K6; ++j) {
        const int y = lane * K6 + j;
        double v = 0.0;
        if (y < ny) v = ldv<double>(frow + (SM ? RowMap<T, K>::elem(y) : y));
        fi[j] = v * tab[L::inv(lane, j)];
        u[j] = 0.0;
    }
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int j = 0; j < K6; ++j) g[j] = fi[j];
        if (it > 0) {
            const double ul = up<double, 32>(u[K6 - 1], 1), ur = dn<double, 32>(u[0], 1);
#pragma unroll
            for (int j = 0; j < K6; ++j) {
                const double *k = K6 == 1 ? tab + L::cross(0) + 4 * lane
                                          : tab + ((j & 1) ? L::odd(0) : L::even(0)) + 4 * ((j >> 1) * 32 + lane);
                g[j] = fi[j] - u[j] - k[0] * (j > 0 ? u[(j + K6 - 1) % K6] : ul) - k[1] * (j + 1 < K6 ? u[(j + 1) % K6] : ur);
            }
        }
        ycycle<double, 32, K6, 0>(g, tab, lane);
#pragma unroll
        for (int j = 0; j < K6; ++j) u[j] += g[j];
    }
#pragma unroll
    for (int j = 0; j < K6; ++j) {
        const int y = lane * K6 + j;
        if (y < ny) stv<T, double>(urow + (SM ? RowMap<T, K>::elem(y) : y), u[j]);
    }
}

// Runs body(plane, active) for the planes first, first + step, ... (count of them), one per group of G
// lanes; every lane of a warp takes the same number of trips (groups past the end repeat the last
// plane with active = false).
template <int G, class F>
__device__ __forceinline__ void for_planes(int count, int first, int step, F body) {
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5, sub = (threadIdx.x & 31) / G;
    constexpr int GPW = 32 / G;
    for (int p0 = warp * GPW; p0 < count; p0 += nw * GPW) {
        const int p = p0 + sub;
        body(first + step * min(p, count - 1), p < count);
    }
}

template <class T, int G, int K>
__device__ __forceinline__ void build_tables(T *tab, const ModalArgs<T> &A, int l, T lam, int tid, int nt) {
    const T *raw = A.raw + static_cast<long long>(A.cls_base[l]) * A.sum_ny * kRawPerLine;
    const int per = Tab<G, K>::kEntries;
    for (int e = tid; e < per * A.ncls[l]; e += nt) {
        const int c = e / per;
        table_entry<T, G, K>(tab + c * Tab<G, K>::kElems, raw + static_cast<long long>(c) * A.sum_ny * kRawPerLine, lam,
                             A.ny_m, A.line_base, A.P, e - c * per);
    }
}

template <class T>
constexpr int modal_threads() { return sizeof(T) == 8 ? 256 : 512; }

// The cycle of one mode (blockIdx.x) and right-hand side (blockIdx.y) on the tail levels.
template <class T, int G, int K>
__device__ __forceinline__ void tail_body(const ModalArgs<T> &A, int mode_idx, int rhs, unsigned char *smem) {
    T *sm = reinterpret_cast<T *>(smem);
    const int tid = threadIdx.x, nt = blockDim.x, ln = (tid & 31) % G;
    const int L = A.L, lt = A.lt, sp = A.sm_pitch;
    T *tab = sm + A.sm_tab, *zcs = sm + A.sm_zc;
    double *tab64 = reinterpret_cast<double *>(smem + A.sm_tab64);
    unsigned char *cls = smem + A.sm_cls;
    const double lam64 = A.lam[mode_idx];
    const T lam = static_cast<T>(lam64);
    const int pb = A.plane_base[lt], np = A.plane_base[L - 1] + 1 - pb;
    for (int i = tid; i < np * kCoefPerPlane; i += nt) zcs[i] = A.zc[pb * kCoefPerPlane + i];
    for (int i = tid; i < np; i += nt) cls[i] = A.cls[pb + i];
    constexpr int K6 = G * K / 32;
    auto build64 = [&](int t0, int n) {
        for (int e = t0; e < Tab<32, K6>::kEntries; e += n)
            table_entry<double, 32, K6>(tab64, A.raw64, lam64, A.ny_m, A.line_base, A.P, e);
    };
    if (lt < L - 1) build_tables<T, G, K>(tab, A, lt, lam, tid, nt);
    build64(tid, nt);
    pdl_wait();
    __syncthreads();
    const long long vec = static_cast<long long>(rhs) * A.nmode + mode_idx;
    const Rows<T> fg{const_cast<T *>(A.f[lt]) + vec * A.nz[lt] * A.pitch, A.pitch, 0};
    T *ug = A.u[lt] + vec * A.nz[lt] * A.pitch;
    auto U = [&](int l) { return Rows<T>{sm + A.sm_u[l], sp, 0}; };
    auto F = [&](int l) { return Rows<T>{sm + A.sm_f[l], sp, 0}; };
    auto relax = [&](int l, int colour, int mode) {
        const int nz = A.nz[l], n = colour ? nz / 2 : (nz + 1) / 2;
        const T *zl = zcs + (A.plane_base[l] - pb) * kCoefPerPlane;
        const unsigned char *cl = cls + A.plane_base[l] - pb;
        const Rows<T> u = U(l);
        for_planes<G>(n, colour, 2, [&](int z, bool act) {
            T g[K];
            const T *tb = tab + cl[z] * Tab<G, K>::kElems;
            if (l == lt) relax_plane<T, G, K, true, false>(g, u, fg, z, nz, zl + z * kCoefPerPlane, tb, lam, mode, l > 0, ln);
            else relax_plane<T, G, K, true, true>(g, u, F(l), z, nz, zl + z * kCoefPerPlane, tb, lam, mode, true, ln);
            if (act) store_row<T, K, true>(u.at(z), g, ln, sp);
        });
        __syncthreads();
    };
    for (int l = lt; l + 1 < L; ++l) {
        for (int s = 0; s < A.npre; ++s) {
            relax(l, 0, s == 0 ? 0 : 2);
            relax(l, 1, s == 0 ? 1 : 2);
        }
        const T *zl = zcs + (A.plane_base[l] - pb) * kCoefPerPlane;
        const Rows<T> fc = F(l + 1);
        if (l + 2 < L) build_tables<T, G, K>(tab, A, l + 1, lam, tid, nt);
        for_planes<G>(A.nz[l + 1], 0, 1, [&](int Z, bool act) {
            T g[K];
            if (l == lt) restrict_plane<T, G, K, true, false>(g, U(l), fg, Z, A.nz[l], zl, lam, l > 0, ln);
            else restrict_plane<T, G, K, true, true>(g, U(l), F(l), Z, A.nz[l], zl, lam, true, ln);
            if (act) store_row<T, K, true>(fc.at(Z), g, ln, sp);
        });
        __syncthreads();
    }
    if (tid < 32) {
        if (lt == L - 1) coarsest<T, G, K, false>(fg.p, ug, A.ny, A.coarse_iters, tab64, tid);
        else coarsest<T, G, K, true>(sm + A.sm_f[L - 1], sm + A.sm_u[L - 1], A.ny, A.coarse_iters, tab64, tid);
    }
    if (lt == L - 1) {
        // the lines past ny of a one-plane cycle: zero, as the transform expects
        for (int y = A.ny + tid; y < A.pitch; y += nt) ug[y] = T(0);
        return;
    }
    if (K6 * 32 > A.ny) {  // rows keep zeros past ny
        T *ul = sm + A.sm_u[L - 1];
        for (int y = A.ny + tid; y < sp; y += nt) ul[RowMap<T, K>::elem(y)] = T(0);
    }
    __syncthreads();
    for (int l = L - 2; l >= lt; --l) {
        const bool last = l == lt && A.npost == 0;
        const T *zl = zcs + (A.plane_base[l] - pb) * kCoefPerPlane;
        const int nzc = A.nz[l + 1];
        const Rows<T> u = U(l), uc = U(l + 1);
        if (A.npost > 0) build_tables<T, G, K>(tab, A, l, lam, tid, nt);
        for_planes<G>(A.nz[l], 0, 1, [&](int z, bool act) {
            T g[K], v[K];
            load_row<T, K, true>(g, u.at(z), ln, sp);
            if (z & 1) {
                load_row<T, K, true>(v, uc.at(z >> 1), ln, sp);
#pragma unroll
                for (int j = 0; j < K; ++j) g[j] += v[j];
            } else {
                const T wm = zl[z * kCoefPerPlane + 6], wp = zl[z * kCoefPerPlane + 7];
                if (z > 0) {
                    load_row<T, K, true>(v, uc.at(z / 2 - 1), ln, sp);
#pragma unroll
                    for (int j = 0; j < K; ++j) g[j] = fma(wm, v[j], g[j]);
                }
                if (z / 2 < nzc) {
                    load_row<T, K, true>(v, uc.at(z / 2), ln, sp);
#pragma unroll
                    for (int j = 0; j < K; ++j) g[j] = fma(wp, v[j], g[j]);
                }
            }
            if (act) {
                if (last) store_row<T, K, false>(ug + static_cast<long long>(z) * A.pitch, g, ln, A.pitch);
                else store_row<T, K, true>(u.at(z), g, ln, sp);
            }
        });
        if (!last) __syncthreads();
        for (int s = 0; s < A.npost; ++s) {
            relax(l, 1, 2);
            relax(l, 0, 2);
        }
    }
    if (A.npost > 0) {
        const Rows<T> u = U(lt);
        for_planes<G>(A.nz[lt], 0, 1, [&](int z, bool act) {
            T g[K];
            load_row<T, K, true>(g, u.at(z), ln, sp);
            if (act) store_row<T, K, false>(ug + static_cast<long long>(z) * A.pitch, g, ln, A.pitch);
        });
    }
}

template <class T, int G, int K>
__global__ void __launch_bounds__(modal_threads<T>(), 1) modal_tail_kernel(const ModalArgs<T> *__restrict__ args) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ ModalArgs<T> A;
    pdl_trigger();
    for (unsigned i = threadIdx.x; i < sizeof(ModalArgs<T>) / 4; i += blockDim.x)
        reinterpret_cast<unsigned *>(&A)[i] = reinterpret_cast<const unsigned *>(args)[i];
    __syncthreads();
    tail_body<T, G, K>(A, blockIdx.x, blockIdx.y, smem);
}

// ---- levels above the tail, over global memory ------------------------------------------------------

// The down-sweep of level l with one pre-relaxation (red, black, residual and restriction) for coarse
// planes Z0 .. Z1-1 of one mode in one CTA: the fine planes 2 Z0 - 2 .. 2 Z1 + 2 the result depends on
// are relaxed in shared memory (a few of them by two CTAs), so that f is read once from memory and
// u and the coarse f written once.
template <class T, int G, int K>
__global__ void __launch_bounds__(modal_threads<T>(), 1) modal_slab_kernel(const __grid_constant__ ModalArgs<T> A, int l, int nslab) {
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_trigger();
    T *sm = reinterpret_cast<T *>(smem);
    const int tid = threadIdx.x, nt = blockDim.x, ln = (tid & 31) % G;
    const int sp = A.sm_pitch, nz = A.nz[l], nzc = A.nz[l + 1], mode_idx = blockIdx.y;
    const int Z0 = static_cast<int>(static_cast<long long>(nzc) * blockIdx.x / nslab);
    const int Z1 = static_cast<int>(static_cast<long long>(nzc) * (blockIdx.x + 1) / nslab);
    const int za = max(0, 2 * Z0 - 2), zb = min(nz, 2 * Z1 + 3);
    const int own0 = 2 * Z0, own1 = (Z1 == nzc) ? nz : 2 * Z1;
    T *tab = sm;
    T *ur = sm + A.ncls[l] * Tab<G, K>::kElems;
    const double lam64 = A.lam[mode_idx];
    const T lam = static_cast<T>(lam64);
    build_tables<T, G, K>(tab, A, l, lam, tid, nt);
    pdl_wait();
    __syncthreads();
    const long long vec = static_cast<long long>(blockIdx.z) * A.nmode + mode_idx;
    const T *zl = A.zc + A.plane_base[l] * kCoefPerPlane;
    const unsigned char *cl = A.cls + A.plane_base[l];
    const Rows<T> f{const_cast<T *>(A.f[l]) + vec * nz * A.pitch, A.pitch, 0}, u{ur, sp, za};
    const Rows<T> ug{A.u[l] + vec * nz * A.pitch, A.pitch, 0};
    for (int colour = 0; colour < 2; ++colour) {
        const int first = za + ((za & 1) != colour), end = colour ? min(nz, 2 * Z1 + 2) : zb;
        const int n = end > first ? (end - first + 1) / 2 : 0;
        for_planes<G>(n, first, 2, [&](int z, bool act) {
            T g[K];
            relax_plane<T, G, K, true, false>(g, u, f, z, nz, zl + z * kCoefPerPlane, tab + cl[z] * Tab<G, K>::kElems, lam,
                                              colour, l > 0, ln);
            if (act) {
                store_row<T, K, true>(u.at(z), g, ln, sp);
                if (z >= own0 && z < own1) store_row<T, K, false>(ug.at(z), g, ln, A.pitch);
            }
        });
        __syncthreads();
    }
    const Rows<T> fc{A.fw[l + 1] + vec * nzc * A.pitch, A.pitch, 0};
    for_planes<G>(Z1 - Z0, Z0, 1, [&](int Z, bool act) {
        T g[K];
        restrict_plane<T, G, K, true, false>(g, u, f, Z, nz, zl, lam, l > 0, ln);
        if (act) store_row<T, K, false>(fc.at(Z), g, ln, A.pitch);
    });
}

// One colour of level l (blockIdx.x: a share of its planes; y: mode; z: right-hand side).
template <class T, int G, int K>
__global__ void __launch_bounds__(256, 1) modal_relax_kernel(const __grid_constant__ ModalArgs<T> A, int l, int colour, int mode) {
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_trigger();
    T *tab = reinterpret_cast<T *>(smem);
    const int tid = threadIdx.x, ln = (tid & 31) % G, nz = A.nz[l], mode_idx = blockIdx.y;
    const double lam64 = A.lam[mode_idx];
    const T lam = static_cast<T>(lam64);
    build_tables<T, G, K>(tab, A, l, lam, tid, blockDim.x);
    pdl_wait();
    __syncthreads();
    const long long vec = static_cast<long long>(blockIdx.z) * A.nmode + mode_idx;
    const T *zl = A.zc + A.plane_base[l] * kCoefPerPlane;
    const unsigned char *cl = A.cls + A.plane_base[l];
    const Rows<T> f{const_cast<T *>(A.f[l]) + vec * nz * A.pitch, A.pitch, 0}, u{A.u[l] + vec * nz * A.pitch, A.pitch, 0};
    const int n = colour ? nz / 2 : (nz + 1) / 2;
    const int p0 = static_cast<int>(static_cast<long long>(n) * blockIdx.x / gridDim.x);
    const int p1 = static_cast<int>(static_cast<long long>(n) * (blockIdx.x + 1) / gridDim.x);
    for_planes<G>(p1 - p0, colour + 2 * p0, 2, [&](int z, bool act) {
        T g[K];
        relax_plane<T, G, K, false, false>(g, u, f, z, nz, zl + z * kCoefPerPlane, tab + cl[z] * Tab<G, K>::kElems, lam, mode,
                                           l > 0, ln);
        if (act) store_row<T, K, false>(u.at(z), g, ln, A.pitch);
    });
}

template <class T, int G, int K>
__global__ void __launch_bounds__(256, 1) modal_restrict_kernel(const __grid_constant__ ModalArgs<T> A, int l) {
    pdl_trigger();
    pdl_wait();
    const int ln = (threadIdx.x & 31) % G, nz = A.nz[l], nzc = A.nz[l + 1], mode_idx = blockIdx.y;
    const T lam = static_cast<T>(A.lam[mode_idx]);
    const long long vec = static_cast<long long>(blockIdx.z) * A.nmode + mode_idx;
    const T *zl = A.zc + A.plane_base[l] * kCoefPerPlane;
    const Rows<T> f{const_cast<T *>(A.f[l]) + vec * nz * A.pitch, A.pitch, 0}, u{A.u[l] + vec * nz * A.pitch, A.pitch, 0};
    const Rows<T> fc{A.fw[l + 1] + vec * nzc * A.pitch, A.pitch, 0};
    const int p0 = static_cast<int>(static_cast<long long>(nzc) * blockIdx.x / gridDim.x);
    const int p1 = static_cast<int>(static_cast<long long>(nzc) * (blockIdx.x + 1) / gridDim.x);
    for_planes<G>(p1 - p0, p0, 1, [&](int Z, bool act) {
        T g[K];
        restrict_plane<T, G, K, false, false>(g, u, f, Z, nz, zl, lam, l > 0, ln);
        if (act) store_row<T, K, false>(fc.at(Z), g, ln, A.pitch);
    });
}

}  // namespace smg
