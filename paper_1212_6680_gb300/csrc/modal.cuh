// modal.cuh -- the SMG V-cycle (section "Preconditioning with SMG" of arXiv:1212.6680) in the sine
// eigenvectors of the x-lines.
//
// Every x-line matrix of the cycle is S Lx + T I with one and the same Lx = tridiag(-1, 2, -1), and
// every coupling between lines and planes is of that form too.  In the orthonormal sine basis of the
// x-direction (Lx v_k = lambda_k v_k) an exact line solve is a division by S lambda_k + T, a coupling
// a multiplication, and the modes k do not couple at all: the V-cycle is nx independent 2D (y, z)
// cycles between two dense transforms of the x-lines (sine.cu, FP64: modal.cu).  The same linear operator as the
// plane kernels' in exact arithmetic, step by step the same relaxations.  What it removes is the
// serial chain of a line solve (elimination, five rounds of cyclic reduction, back substitution) in
// each of a plane's 4P - 3 dependent steps, and the CTA barrier between them.  One application at
// 128^3: 672 -> 75 us (FP32), 2352 -> 969 us (FP64); 256^3 FP32 2154 -> 645 us; 1280x80x80 FP32
// 3802 -> 704 us; 24x20x16 FP32 135 -> 24 us.
//
// One CTA runs the whole cycle of one mode in shared memory (modal_tail); levels whose planes do
// not fit there run as launches over global memory first (modal_slab, or the single steps).
//
// One plane of one mode is a vector of ny values.  G lanes hold K consecutive lines each
// (G K >= ny, both powers of two), and the plane's y-cycle runs in registers:
//   * coarse line i of level m+1 is line 2i+1 of level m, so a lane's K lines hold K/2 lines of the
//     next level, and so on: the first log2 K levels need shuffles only at the lane borders;
//   * from level log2 K on (one line per lane) the rest of the y-cycle is a linear map of G values
//     that depends on the mode and the plane's class only: one G x G product with a matrix formed at
//     set-up (log2 G levels of dependent shuffles before: 510 of 1190 cycles of a plane's latency);
//   * right-hand sides are kept divided by the line's diagonal (gi = g / (S lambda + T)), which
//     turns each relaxation into two FMAs a line and makes the first even sweep the identity;
//   * the lines' multipliers come from a table in shared memory, laid out so that a group's lanes
//     read consecutive words.  It is spread there at each z-level from the few line types that
//     differ (ModalArgs), fetched by cp.async while the level before is relaxed: formed in the
//     kernel with its divisions it took 5300 of about 14000 cycles a level.
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
// per even line {a-, a+, wm, wp}, per odd line {a-, a+, ca, cc} and cb.  a-, a+: couplings over the
// diagonal; wm, wp: interpolation weights; ca, cb, cc: the restriction from lines 2j-1, 2j+1, 2j+3 to
// coarse line j, over the coarse line's diagonal.  Then the G x G matrix D of the levels from log2 K
// on (D[k][lane], four k together) and the reciprocal diagonals of level 0.
template <int G, int K>
struct Tab {
    static constexpr int M0 = ilog2(K);
    static constexpr int quad(int m) { return 2 * G * (K - (K >> m)); }
    static constexpr int even(int m) { return 4 * quad(m); }
    static constexpr int odd(int m) { return 4 * (quad(m) + (K >> m) / 2 * G); }
    static constexpr int kScal = 4 * quad(M0);
    static constexpr int scal(int m) { return kScal + G * (K - (K >> m)); }
    static constexpr int kDense = scal(M0) + (G * (K - 1)) % 4;  // a multiple of 4
    static constexpr int kInv = kDense + G * G;
    static constexpr int kElems = kInv + K * G;
    static constexpr int kEntries = quad(M0);  // lines of the in-register levels
    __host__ __device__ static constexpr int dense(int k, int lane) { return kDense + ((k / 4) * G + lane) * 4 + (k & 3); }
    __host__ __device__ static constexpr int inv(int lane, int j) {  // four lines of a lane together
        return kInv + (K >= 4 ? ((j / 4) * G + lane) * 4 + (j & 3) : j * G + lane);
    }
};
// values of one class in global memory: the line types' rows, then D row by row of four k (Tab::dense)
template <int G> constexpr int class_values(int ntype) { return ntype * kRow + G * G; }

// Spread the rows of ncls classes (class c's values at src + c blk, in shared or global memory) over their
// tables.  Entry e of a class: level m, lane, and the lane's line j of that level (line y of the level).
template <class T, int G, int K>
__device__ __forceinline__ void spread_tables(T *tab, const T *src, int ncls, int blk, const unsigned short *ltype, const int *ny_m,
                                              const int *line_base, int P, int ntype, int tid, int nt) {
    using L = Tab<G, K>;
    constexpr int kLines = K == 1 ? G : L::kEntries, kItems = kLines + G * G / 4;
    for (int it = tid; it < ncls * kItems; it += nt) {
        const int c = it / kItems, e = it - c * kItems;
        T *t = tab + c * L::kElems;
        const T *s = src + c * blk;
        if (e >= kLines) {
            const int i = 4 * (e - kLines);
            const V4<T> v = ld4(s + ntype * kRow + i);
            st4(t + L::kDense + i, v.x, v.y, v.z, v.w);
            continue;
        }
        int m = 0, y = e;
#pragma unroll
        for (int q = 0; q + 1 < L::M0; ++q)
            if (m == q && y >= (K >> q) * G) y -= (K >> q) * G, m = q + 1;
        const int lg = L::M0 - m, lane = y >> lg, j = y & ((1 << lg) - 1), i = j >> 1;
        V4<T> v{T(0), T(0), T(0), T(0)};
        T inv = T(0), cb = T(0);
        if (m < P && y < ny_m[m]) {
            const T *r = s + ltype[line_base[m] + y] * kRow;
            v = ld4(r);
            inv = r[4];
            cb = r[5];
        }
        if constexpr (K > 1) {
            st4(t + 4 * (2 * G * (K - (1 << lg)) + ((j & 1) ? (G << lg) / 2 : 0) + i * G + lane), v.x, v.y, v.z, v.w);
            if (j & 1) t[L::kScal + G * (K - (1 << lg)) + i * G + lane] = cb;
        }
        if (m == 0) t[L::inv(lane, j)] = inv;
    }
}

// Shuffles within a group of G lanes; at the group's ends they return the lane's own value, which the
// zero multiplier of the missing neighbour removes.
template <class T, int G>
__device__ __forceinline__ T up(T v, int s) { return __shfl_up_sync(0xffffffffu, v, s, G); }
template <class T, int G>
__device__ __forceinline__ T dn(T v, int s) { return __shfl_down_sync(0xffffffffu, v, s, G); }

// The y-cycle from level log2 K on: gi in, the correction out.
template <class T, int G, int K>
__device__ __forceinline__ T ycycle_dense(T gi, const T *tab, int ln) {
    T a = T(0), b = T(0);
#pragma unroll
    for (int k = 0; k < G; k += 4) {
        const V4<T> d = ld4(tab + Tab<G, K>::dense(k, ln));
        a = fma(d.x, __shfl_sync(0xffffffffu, gi, k, G), a);
        b = fma(d.y, __shfl_sync(0xffffffffu, gi, k + 1, G), b);
        a = fma(d.z, __shfl_sync(0xffffffffu, gi, k + 2, G), a);
        b = fma(d.w, __shfl_sync(0xffffffffu, gi, k + 3, G), b);
    }
    return a + b;
}

// The y-cycle from in-register level M on: g (right-hand sides over the diagonals) in, the
// correction out.  Down: even lines (zero neighbours), odd lines, restriction (the residual is zero on
// odd lines); up: odd lines against the corrected even ones, then even lines.
template <class T, int G, int K, int M>
__device__ __forceinline__ void ycycle(T (&g)[(K >> M)], const T *tab, int ln) {
    using L = Tab<G, K>;
    constexpr int N = K >> M;
    if constexpr (N == 1) {
        g[0] = ycycle_dense<T, G, K>(g[0], tab, ln);
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
// The same from either place: shared rows are swizzled, global ones are not.
template <class T, int K>
__device__ __forceinline__ void load_row_at(T (&v)[K], const T *row, bool shared, int ln, int pitch) {
    if (shared) load_row<T, K, true>(v, row, ln, pitch);
    else load_row<T, K, false>(v, row, ln, pitch);
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
    bool shared;
    __device__ __forceinline__ T *at(int z) const { return p + static_cast<long long>(z - z0) * pitch; }
};

// One plane's part of f - sum (M (lambda + Ly) + Kc) u, on a row u (M = Kc = 0 where the plane is absent).
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
// Relaxation of plane z: u_z = C_z (f - A u)_z (modes 0 and 1: the own plane is zero, mode 0: all
// planes are) or u_z += (mode 2).  cross: the couplings between planes have an in-plane part (all
// levels but the finest).  f's row comes in g; the result stays there.
template <class T, int G, int K, bool SMU>
__device__ __forceinline__ void relax_plane(T (&g)[K], const Rows<T> &u, int z, int nz, const T *zc, const T *tab, T lam, int mode,
                                            bool cross, int ln) {
    if (mode > 0) {
        // a plane at the end couples to its one neighbour; the other's coefficients are zero
        T v[K], w[K];
        load_row<T, K, SMU>(v, u.at(z > 0 ? z - 1 : z + 1), ln, u.pitch);
        load_row<T, K, SMU>(w, u.at(z + 1 < nz ? z + 1 : z - 1), ln, u.pitch);
        couple<T, G, K>(g, v, zc[0], zc[3], lam, cross, ln);
        couple<T, G, K>(g, w, zc[2], zc[5], lam, cross, ln);
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

// Sixteen bytes of a row at chunk c (shared rows are swizzled, global ones are not), and one value.
template <class T, int K>
struct Chunk {
    static constexpr int CH = RowMap<T, K>::CH;
    union {
        T t[CH];
        uint4 q;
    };
    __device__ __forceinline__ void load(const Rows<T> &r, int z, int c) {
        q = reinterpret_cast<const uint4 *>(r.at(z))[r.shared ? RowMap<T, K>::chunk(c) : c];
    }
    __device__ __forceinline__ void store(const Rows<T> &r, int z, int c) const {
        reinterpret_cast<uint4 *>(r.at(z))[r.shared ? RowMap<T, K>::chunk(c) : c] = q;
    }
};

// Runs body(plane, chunk) for planes 0 .. count-1 and chunks 0 .. nch-1 of each, the chunks of a plane on
// neighbouring lanes.
template <class F>
__device__ __forceinline__ void for_chunks(int count, int nch, F body) {
    const int lg = nch >= 17 ? 5 : nch >= 9 ? 4 : nch >= 5 ? 3 : 2;  // lanes of a plane: 2^lg
    for (int c = threadIdx.x & ((1 << lg) - 1); c < nch; c += 1 << lg)
        for (int z = threadIdx.x >> lg; z < count; z += blockDim.x >> lg) body(z, c);
}

// A row's chunk with the lines before and after it.
template <class T, int K>
struct Window {
    Chunk<T, K> v;
    T l, r;
    __device__ __forceinline__ void load(const Rows<T> &u, int z, int c, int nch, bool ends) {
        constexpr int CH = Chunk<T, K>::CH;
        v.load(u, z, c);
        l = r = T(0);
        if (!ends) return;
        const T *row = u.at(z);
        const int yl = max(c * CH - 1, 0), yr = min(c + 1, nch - 1) * CH;
        l = row[u.shared ? RowMap<T, K>::elem(yl) : yl];
        r = row[u.shared ? RowMap<T, K>::elem(yr) : yr];
        if (c == 0) l = T(0);
        if (c + 1 == nch) r = T(0);
    }
    // couple() for this chunk
    __device__ __forceinline__ void couple(Chunk<T, K> &g, T M, T Kc, T lam, bool in_plane) const {
        constexpr int CH = Chunk<T, K>::CH;
#pragma unroll
        for (int j = 0; j < CH; ++j) g.t[j] = fma(-Kc, v.t[j], g.t[j]);
        if (!in_plane) return;
#pragma unroll
        for (int j = 0; j < CH; ++j) {
            const T d = (v.t[j] - (j > 0 ? v.t[(j + CH - 1) % CH] : l)) + (v.t[j] - (j + 1 < CH ? v.t[(j + 1) % CH] : r));
            g.t[j] = fma(-M, fma(lam, v.t[j], d), g.t[j]);
        }
    }
};

// Coarse plane Z's right-hand side P^T (f - A u) at chunk c: the residuals of planes 2Z, 2Z+1 and 2Z+2 with
// the weights of P, as one combination of five planes of u and three of f.  row(z): plane z's coefficients.
// Planes past the ends are replaced by the last one: their weights and couplings are zero (an odd
// plane's weights are).  All loads are issued before the arithmetic.
template <class T, int K>
struct RestrictF {
    Chunk<T, K> f0, g, f1;   // planes 2Z, 2Z+1, 2Z+2 of f
    __device__ __forceinline__ void load(const Rows<T> &f, int Z, int nz, int c) {
        f0.load(f, 2 * Z, c);
        g.load(f, 2 * Z + 1, c);
        f1.load(f, min(2 * Z + 2, nz - 1), c);
    }
};
template <class T, int K, class F>
__device__ __forceinline__ void restrict_chunk(RestrictF<T, K> &r, const Rows<T> &u, int Z, int nz, F row, T lam, bool cross, int c,
                                               int nch) {
    constexpr int CH = Chunk<T, K>::CH;
    Chunk<T, K> &g = r.g;
    const int o = 2 * Z + 1, e1 = min(o + 1, nz - 1);
    const T *zo = row(o), *z0 = row(o - 1), *z1 = row(e1);
    Window<T, K> v0, v1, v2, v3, v4;
    v0.load(u, max(o - 2, 0), c, nch, cross);
    v1.load(u, o - 1, c, nch, true);
    v2.load(u, o, c, nch, true);
    v3.load(u, e1, c, nch, true);
    v4.load(u, min(o + 2, nz - 1), c, nch, cross);
    const T w0 = z0[7], w1 = z1[6];
#pragma unroll
    for (int j = 0; j < CH; ++j) g.t[j] = fma(w1, r.f1.t[j], fma(w0, r.f0.t[j], g.t[j]));
    v0.couple(g, w0 * z0[0], w0 * z0[3], lam, cross);
    v1.couple(g, fma(w0, z0[1], zo[0]), fma(w0, z0[4], zo[3]), lam, true);
    v2.couple(g, fma(w1, z1[0], fma(w0, z0[2], zo[1])), fma(w1, z1[3], fma(w0, z0[5], zo[4])), lam, true);
    v3.couple(g, fma(w1, z1[1], zo[2]), fma(w1, z1[4], zo[5]), lam, true);
    v4.couple(g, w1 * z1[2], w1 * z1[5], lam, cross);
}

// The restriction of coarse planes Z0 .. Z0 + count - 1, chunks 0 .. nchw - 1 (those from nch on are past
// the rows: zero), f's chunks one plane ahead; store(Z, chunk, value).
template <class T, int K, class F, class S>
__device__ __forceinline__ void restrict_planes(int Z0, int count, int nch, int nchw, const Rows<T> &u, const Rows<T> &f, int nz, F row,
                                                T lam, bool cross, S store) {
    const int lg = nchw >= 17 ? 5 : nchw >= 9 ? 4 : nchw >= 5 ? 3 : 2, dz = blockDim.x >> lg, z0 = threadIdx.x >> lg;
    if (z0 >= count) return;
    for (int c = threadIdx.x & ((1 << lg) - 1); c < nchw; c += 1 << lg) {
        if (c >= nch) {
            Chunk<T, K> zero;
            zero.q = make_uint4(0u, 0u, 0u, 0u);
            for (int z = z0; z < count; z += dz) store(Z0 + z, c, zero);
            continue;
        }
        RestrictF<T, K> next;
        next.load(f, Z0 + z0, nz, c);
        for (int z = z0; z < count; z += dz) {
            RestrictF<T, K> r = next;
            if (z + dz < count) next.load(f, Z0 + z + dz, nz, c);
            restrict_chunk<T, K>(r, u, Z0 + z, nz, row, lam, cross, c, nch);
            store(Z0 + z, c, r.g);
        }
    }
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
                const double *k = tab + (K6 == 1 ? L::kElems + 2 * lane
                                                 : ((j & 1) ? L::odd(0) : L::even(0)) + 4 * ((j >> 1) * 32 + lane));
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
// its table: with one line a lane the couplings of level 0 (needed beyond the first step) follow it
template <int G, int K> constexpr int tab64_elems() { return Tab<32, G * K / 32>::kElems + (G * K == 32 ? 64 : 0); }

// Runs body(plane, active, f row) for the planes first, first + step, ... (count of them), one per group
// of G lanes; every lane of a warp takes the same number of trips (groups past the end repeat the last
// plane with active = false).  The next plane's f row is on its way while one is relaxed: from global
// memory its latency is as long as the relaxation.
template <class T, int G, int K, class F>
__device__ __forceinline__ void for_planes(int count, int first, int step, const Rows<T> &f, F body) {
    constexpr int GPW = 32 / G;
    const int p0 = (threadIdx.x >> 5) * GPW, dp = (blockDim.x >> 5) * GPW, sub = (threadIdx.x & 31) / G, ln = (threadIdx.x & 31) % G;
    if (p0 >= count) return;
    auto plane = [&](int p) { return first + step * min(p, count - 1); };
    T next[K];
    load_row_at<T, K>(next, f.at(plane(p0 + sub)), f.shared, ln, f.pitch);
    for (int p = p0; p < count; p += dp) {
        T g[K];
#pragma unroll
        for (int j = 0; j < K; ++j) g[j] = next[j];
        if (p + dp < count) load_row_at<T, K>(next, f.at(plane(p + dp + sub)), f.shared, ln, f.pitch);
        body(plane(p + sub), p + sub < count, g);
    }
}

// ---- set-up: the multipliers and matrices of every mode and class ------------------------------------

// The y-cycle below the in-register levels on the unit vectors: thread k of a warp runs level m0 with
// right-hand side (over the diagonals) e_k.  rows: this class's line types in FP64.
template <int G>
__device__ void dense_column(double *col, int k, const double *rows, const unsigned short *ltype, const int *ny_m,
                             const int *line_base, int P, int m0) {
    double gi[2 * G], c[G];
    const int n0 = m0 < P ? ny_m[m0] : 0;
    for (int i = 0; i < G; ++i) gi[i] = 0.0, col[i] = 0.0;
    if (k >= n0) return;
    gi[k] = 1.0;
    int m = m0, base = 0;  // level m's right-hand sides start at base
    auto row = [&](int mm, int y) { return rows + ltype[line_base[mm] + y] * kRow; };
    for (; m + 1 < P; ++m) {
        const int n = ny_m[m];
        double *g = gi + base, *gc = g + n;
        double prev = 0.0, here = 0.0;
        auto odd = [&](int y) {
            const double *r = row(m, y);
            return g[y] - r[0] * g[y - 1] - (y + 1 < n ? r[1] * g[y + 1] : 0.0);
        };
        here = n > 1 ? odd(1) : 0.0;
        for (int j = 0; j < n / 2; ++j) {
            const double next = 2 * j + 3 < n ? odd(2 * j + 3) : 0.0;
            const double *r = row(m, 2 * j + 1);
            gc[j] = r[2] * prev + r[5] * here + r[3] * next;
            prev = here;
            here = next;
        }
        base += n;
    }
    c[0] = gi[base];
    for (--m; m >= m0; --m) {
        const int n = ny_m[m], nc = n / 2;
        base -= n;
        double *g = gi + base, v[G];
        for (int y = 0; y < n; y += 2) {
            const double *r = row(m, y);
            v[y] = g[y] + (y > 0 ? r[2] * c[y / 2 - 1] : 0.0) + (y / 2 < nc ? r[3] * c[y / 2] : 0.0);
        }
        for (int y = 1; y < n; y += 2) {
            const double *r = row(m, y);
            v[y] = g[y] - r[0] * v[y - 1] - (y + 1 < n ? r[1] * v[y + 1] : 0.0);
        }
        for (int y = 0; y < n; y += 2) {
            const double *r = row(m, y);
            c[y] = g[y] - (y > 0 ? r[0] * v[y - 1] : 0.0) - (y + 1 < n ? r[1] * v[y + 1] : 0.0);
        }
        for (int y = 1; y < n; y += 2) c[y] = v[y];
    }
    for (int i = 0; i < n0; ++i) col[i] = c[i];
}

// rows of one class from its raw coefficients (s, t): s lambda + t
__device__ __forceinline__ void type_row(double *r, const double *__restrict__ raw, double lam) {
    auto at = [&](int i) { return fma(raw[i], lam, raw[i + 1]); };
    const double inv = 1.0 / at(0);
    r[0] = at(2) * inv;
    r[1] = at(4) * inv;
    r[4] = inv;
    r[5] = r[6] = r[7] = 0.0;
    if (raw[12] == 0.0) {  // an even line: its weights
        r[2] = raw[6];
        r[3] = raw[7];
    } else {
        const double ic = 1.0 / at(12);
        r[2] = at(6) * ic;
        r[3] = at(10) * ic;
        r[5] = at(8) * ic;
    }
}

// One warp per (mode, class): rows and matrix in FP64, rounded to T; the last class's (the coarsest
// level's) also in FP64 for the 32 lanes of coarsest().  FP64-pipe bound; once per set-up.
template <class T, int G, int K>
__global__ void __launch_bounds__(128) modal_setup_kernel(const __grid_constant__ ModalArgs<T> A, T *coef, double *coef64) {
    extern __shared__ double rows_all[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    double *rows = rows_all + warp * A.ntype * kRow;
    const long long job = static_cast<long long>(blockIdx.x) * nw + warp;
    if (job >= static_cast<long long>(A.nmode) * A.ncls_all) return;
    const int mode_idx = static_cast<int>(job / A.ncls_all), c = static_cast<int>(job - static_cast<long long>(mode_idx) * A.ncls_all);
    const double lam = A.lam[mode_idx];
    T *out = coef + job * A.blk;
    for (int t = lane; t < A.ntype; t += 32) {
        double r[kRow];
        type_row(r, A.raw + (static_cast<long long>(c) * A.ntype + t) * kRawPerLine, lam);
        for (int i = 0; i < kRow; ++i) {
            rows[t * kRow + i] = r[i];
            out[t * kRow + i] = static_cast<T>(r[i]);
        }
    }
    __syncwarp();
    double col[32];
    if (lane < G) {
        dense_column<G>(col, lane, rows, A.ltype, A.ny_m, A.line_base, A.P, ilog2(K));
        for (int i = 0; i < G; ++i) out[A.ntype * kRow + ((lane / 4) * G + i) * 4 + (lane & 3)] = static_cast<T>(col[i]);
    }
    if (c == A.ncls_all - 1) {
        constexpr int K6 = G * K / 32;
        double *o = coef64 + static_cast<long long>(mode_idx) * class_values<32>(A.ntype);
        for (int t = lane; t < A.ntype * kRow; t += 32) o[t] = rows[t];
        dense_column<32>(col, lane, rows, A.ltype, A.ny_m, A.line_base, A.P, ilog2(K6));
        for (int i = 0; i < 32; ++i) o[A.ntype * kRow + ((lane / 4) * 32 + i) * 4 + (lane & 3)] = col[i];
    }
}

// ---- the tail ---------------------------------------------------------------------------------------

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(dst))), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <class T>
constexpr int modal_threads() { return sizeof(T) == 8 ? 256 : 512; }

// The cycle of one mode and right-hand side on the tail levels, as one loop over planned steps, a CTA
// barrier after each: every kind of step is compiled once (inlined at each place of the cycle it
// appears, the kernel would not fit the instruction cache).
template <class T, int G, int K>
__device__ __forceinline__ void tail_body(const ModalArgs<T> &A, int mode_idx, int rhs, int coarse_iters, unsigned char *smem) {
    __shared__ TailOp ring[2];  // the step that runs and the next
    T *sm = reinterpret_cast<T *>(smem);
    const int tid = threadIdx.x, nt = blockDim.x, ln = (tid & 31) % G;
    const int L = A.L, lt = A.lt, sp = A.sm_pitch;
    T *tab = sm + A.sm_tab, *stage = sm + A.sm_stage, *zt = sm + A.sm_zt;
    double *tab64 = reinterpret_cast<double *>(smem + A.sm_tab64);
    unsigned short *ltype = reinterpret_cast<unsigned short *>(smem + A.sm_ltype), *ptype = reinterpret_cast<unsigned short *>(smem + A.sm_ptype),
                   *pcls = reinterpret_cast<unsigned short *>(smem + A.sm_pcls);
    const T lam = static_cast<T>(A.lam[mode_idx]);
    const int pb = A.plane_base[lt], np = A.plane_base[L - 1] + 1 - pb;
    constexpr int K6 = G * K / 32, CH = Chunk<T, K>::CH;
    const long long vec = static_cast<long long>(rhs) * A.nmode + mode_idx;
    const Rows<T> fg{const_cast<T *>(A.f[lt]) + vec * A.nz[lt] * A.pitch, A.pitch, 0, false};
    const Rows<T> ug{A.u[lt] + vec * A.nz[lt] * A.pitch, A.pitch, 0, false};
    const T *coef = A.coef + static_cast<long long>(mode_idx) * A.ncls_all * A.blk;
    auto fetch_classes = [&](int at, int n) {
        for (int i = tid; i < n / CH; i += nt) cp_async16(stage + i * CH, coef + at + i * CH);
    };
    auto fetch_op = [&](int i) {
        if (tid < 4) cp_async16(reinterpret_cast<int4 *>(&ring[i & 1]) + tid, reinterpret_cast<const int4 *>(A.ops + i) + tid);
    };
    // what does not depend on the right-hand side
    fetch_op(0);
    if (lt < L - 1) fetch_classes(A.cls_base[lt] * A.blk, A.ncls[lt] * A.blk);
    for (int i = tid; i < A.nptype * kCoefPerPlane; i += nt) zt[i] = A.zt[i];
    for (int i = tid; i < A.nptype; i += nt) pcls[i] = A.pcls[i];
    for (int i = tid; i < np; i += nt) ptype[i] = A.ptype[pb + i];
    for (int i = tid; i < A.sum_ny; i += nt) ltype[i] = A.ltype[i];
    cp_async_wait();
    __syncthreads();
    for (int step = 0;; ++step) {
        const TailOp &o = ring[step & 1];
        const int kind = o.kind;
        if (kind == OP_END) break;
        fetch_op(step + 1);
        if (o.fetch_n > 0) fetch_classes(o.fetch, o.fetch_n);  // of the level relaxed after this one
        // spread the line tables of the next level to be relaxed (nothing reads the present ones now), from
        // the last thread on: the first ones have the restriction's planes
        if (o.spread > 0)
            spread_tables<T, G, K>(tab, stage, o.spread, A.blk, ltype, A.ny_m, A.line_base, A.P, A.ntype, nt - 1 - tid, nt);
        const unsigned short *pt = ptype + o.ptype;
        auto row = [&](int z) -> const T * { return zt + pt[z] * kCoefPerPlane; };
        const Rows<T> u{sm + o.u, sp, 0, true}, f = o.f < 0 ? fg : Rows<T>{sm + o.f, sp, 0, true};
        const bool lower = o.level > 0;
        const int nz = o.nz;
        if (kind == OP_RELAX) {
            const int mode = o.mode;
            for_planes<T, G, K>(o.n, o.colour, 2, f, [&](int z, bool act, T (&g)[K]) {
                relax_plane<T, G, K, true>(g, u, z, nz, row(z), tab + pcls[pt[z]] * Tab<G, K>::kElems, lam, mode, lower, ln);
                if (act) store_row<T, K, true>(u.at(z), g, ln, sp);
            });
        } else if (kind == OP_RESTRICT) {
            const Rows<T> fc{sm + o.fc, sp, 0, true};
            restrict_planes<T, K>(0, o.nzc, A.pitch / CH, sp / CH, u, f, nz, row, lam, lower,
                                  [&](int Z, int c, const Chunk<T, K> &g) { g.store(fc, Z, c); });
        } else if (kind == OP_COARSEST) {
            if (lt == L - 1) {  // the only level: straight to global memory
                if (tid < 32) coarsest<T, G, K, false>(fg.p, ug.p, A.ny, coarse_iters, tab64, tid);
                for (int y = A.ny + tid; y < A.pitch; y += nt) ug.p[y] = T(0);
            } else {
                if (tid < 32) coarsest<T, G, K, true>(f.p, u.p, A.ny, coarse_iters, tab64, tid);
                for (int y = A.ny + tid; y < sp; y += nt) u.p[RowMap<T, K>::elem(y)] = T(0);
            }
        } else if (kind == OP_PROLONG || kind == OP_STORE) {
            // u_l += P u_{l+1}; on the last level, with no sweep to follow, straight to global memory
            const bool add = kind == OP_PROLONG, out = o.out != 0;
            const int nzc = add ? o.nzc : 1;
            const Rows<T> uc{sm + o.uc, sp, 0, true};
            for_chunks(nz, (out ? A.pitch : sp) / CH, [&](int z, int c) {
                Chunk<T, K> g, v, w;
                g.load(u, z, c);
                if (add) {
                    // coarse planes z/2 - 1 and z/2 of an even z (weights zero past the ends); z/2 alone of an odd z
                    const T *zr = row(z);
                    v.load(uc, max(z / 2 - 1, 0), c);
                    w.load(uc, min(z / 2, nzc - 1), c);
                    const T wm = zr[6], wp = (z & 1) ? T(1) : zr[7];
#pragma unroll
                    for (int j = 0; j < CH; ++j) g.t[j] = fma(wp, w.t[j], fma(wm, v.t[j], g.t[j]));
                }
                g.store(out ? ug : u, z, c);
            });
        } else {  // OP_TABLES
            // the coarsest plane's table is spread over 32 lanes, from global memory
            const double *src = A.coef64 + static_cast<long long>(mode_idx) * class_values<32>(A.ntype);
            spread_tables<double, 32, K6>(tab64, src, 1, 0, ltype, A.ny_m, A.line_base, A.P, A.ntype, tid, nt);
            if (K6 == 1)
                for (int i = tid; i < 32; i += nt) {
                    tab64[Tab<32, K6>::kElems + 2 * i] = i < A.ny ? src[ltype[i] * kRow] : 0.0;
                    tab64[Tab<32, K6>::kElems + 2 * i + 1] = i < A.ny ? src[ltype[i] * kRow + 1] : 0.0;
                }
            pdl_wait();
        }
        cp_async_wait();
        __syncthreads();
    }
}

template <class T, int G, int K>
__global__ void __launch_bounds__(modal_threads<T>(), 1) modal_tail_kernel(const ModalArgs<T> *__restrict__ args, int coarse_iters) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ ModalArgs<T> A;
    pdl_trigger();
    for (unsigned i = threadIdx.x; i < sizeof(ModalArgs<T>) / 4; i += blockDim.x)
        reinterpret_cast<unsigned *>(&A)[i] = reinterpret_cast<const unsigned *>(args)[i];
    __syncthreads();
    tail_body<T, G, K>(A, blockIdx.x, blockIdx.y, coarse_iters, smem);
}

// One (system, mode) of a list per CTA; systems that are not being iterated are skipped.
template <class T, int G, int K>
__global__ void __launch_bounds__(modal_threads<T>(), 1) modal_tail_batch_kernel(const ModalArgs<T> *__restrict__ args,
                                                                              const ModalTask *__restrict__ tasks, const int *active) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ ModalArgs<T> A;
    const ModalTask t = tasks[blockIdx.x];
    if (active[t.sys] != 1) return;
    for (unsigned i = threadIdx.x; i < sizeof(ModalArgs<T>) / 4; i += blockDim.x)
        reinterpret_cast<unsigned *>(&A)[i] = reinterpret_cast<const unsigned *>(args + t.sys)[i];
    __syncthreads();
    tail_body<T, G, K>(A, t.mode, 0, 1, smem);
}

// ---- levels above the tail, over global memory ------------------------------------------------------

// The line tables of level l for one mode, from global memory.
template <class T, int G, int K>
__device__ __forceinline__ void level_tables(T *tab, const ModalArgs<T> &A, int l, int mode_idx) {
    spread_tables<T, G, K>(tab, A.coef + (static_cast<long long>(mode_idx) * A.ncls_all + A.cls_base[l]) * A.blk, A.ncls[l], A.blk,
                           A.ltype, A.ny_m, A.line_base, A.P, A.ntype, threadIdx.x, blockDim.x);
}

// The down-sweep of level l with one pre-relaxation (red, black, residual and restriction) for coarse
// planes Z0 .. Z1-1 of one mode in one CTA: the fine planes 2 Z0 - 2 .. 2 Z1 + 2 the result depends on
// are relaxed in shared memory (a few of them by two CTAs), so that f is read once from memory and
// u and the coarse f written once.
template <class T, int G, int K>
__global__ void __launch_bounds__(modal_threads<T>(), 1) modal_slab_kernel(const __grid_constant__ ModalArgs<T> A, int l, int nslab) {
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_trigger();
    constexpr int CH = Chunk<T, K>::CH;
    const int ln = (threadIdx.x & 31) % G;
    const int sp = A.sm_pitch, nz = A.nz[l], nzc = A.nz[l + 1], mode_idx = blockIdx.y;
    const int Z0 = static_cast<int>(static_cast<long long>(nzc) * blockIdx.x / nslab);
    const int Z1 = static_cast<int>(static_cast<long long>(nzc) * (blockIdx.x + 1) / nslab);
    const int za = max(0, 2 * Z0 - 2), zb = min(nz, 2 * Z1 + 3);
    const int own0 = 2 * Z0, own1 = (Z1 == nzc) ? nz : 2 * Z1;
    T *tab = reinterpret_cast<T *>(smem);
    T *ur = tab + A.ncls[l] * Tab<G, K>::kElems;
    const T lam = static_cast<T>(A.lam[mode_idx]);
    level_tables<T, G, K>(tab, A, l, mode_idx);
    pdl_wait();
    __syncthreads();
    const long long vec = static_cast<long long>(blockIdx.z) * A.nmode + mode_idx;
    const unsigned short *pt = A.ptype + A.plane_base[l];
    auto row = [&](int z) -> const T * { return A.zt + pt[z] * kCoefPerPlane; };
    const Rows<T> f{const_cast<T *>(A.f[l]) + vec * nz * A.pitch, A.pitch, 0, false}, u{ur, sp, za, true};
    const Rows<T> ug{A.u[l] + vec * nz * A.pitch, A.pitch, 0, false};
    for (int colour = 0; colour < 2; ++colour) {
        const int first = za + ((za & 1) != colour), end = colour ? min(nz, 2 * Z1 + 2) : zb;
        const int n = end > first ? (end - first + 1) / 2 : 0;
        for_planes<T, G, K>(n, first, 2, f, [&](int z, bool act, T (&g)[K]) {
            relax_plane<T, G, K, true>(g, u, z, nz, row(z), tab + A.pcls[pt[z]] * Tab<G, K>::kElems, lam, colour, l > 0, ln);
            if (act) {
                store_row<T, K, true>(u.at(z), g, ln, sp);
                if (z >= own0 && z < own1) store_row<T, K, false>(ug.at(z), g, ln, A.pitch);
            }
        });
        __syncthreads();
    }
    const Rows<T> fc{A.fw[l + 1] + vec * nzc * A.pitch, A.pitch, 0, false};
    const int nch = A.pitch / CH;
    restrict_planes<T, K>(Z0, Z1 - Z0, nch, nch, u, f, nz, row, lam, l > 0,
                          [&](int Z, int c, const Chunk<T, K> &g) { g.store(fc, Z, c); });
}

// One colour of level l (blockIdx.x: a share of its planes; y: mode; z: right-hand side).
template <class T, int G, int K>
__global__ void __launch_bounds__(256, 1) modal_relax_kernel(const __grid_constant__ ModalArgs<T> A, int l, int colour, int mode) {
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_trigger();
    T *tab = reinterpret_cast<T *>(smem);
    const int ln = (threadIdx.x & 31) % G, nz = A.nz[l], mode_idx = blockIdx.y;
    const T lam = static_cast<T>(A.lam[mode_idx]);
    level_tables<T, G, K>(tab, A, l, mode_idx);
    pdl_wait();
    __syncthreads();
    const long long vec = static_cast<long long>(blockIdx.z) * A.nmode + mode_idx;
    const unsigned short *pt = A.ptype + A.plane_base[l];
    const Rows<T> f{const_cast<T *>(A.f[l]) + vec * nz * A.pitch, A.pitch, 0, false};
    const Rows<T> u{A.u[l] + vec * nz * A.pitch, A.pitch, 0, false};
    const int n = colour ? nz / 2 : (nz + 1) / 2;
    const int p0 = static_cast<int>(static_cast<long long>(n) * blockIdx.x / gridDim.x);
    const int p1 = static_cast<int>(static_cast<long long>(n) * (blockIdx.x + 1) / gridDim.x);
    for_planes<T, G, K>(p1 - p0, colour + 2 * p0, 2, f, [&](int z, bool act, T (&g)[K]) {
        relax_plane<T, G, K, false>(g, u, z, nz, A.zt + pt[z] * kCoefPerPlane, tab + A.pcls[pt[z]] * Tab<G, K>::kElems, lam, mode,
                                    l > 0, ln);
        if (act) store_row<T, K, false>(u.at(z), g, ln, A.pitch);
    });
}

template <class T, int G, int K>
__global__ void __launch_bounds__(256, 1) modal_restrict_kernel(const __grid_constant__ ModalArgs<T> A, int l) {
    pdl_trigger();
    pdl_wait();
    const int nz = A.nz[l], nzc = A.nz[l + 1], mode_idx = blockIdx.y;
    const T lam = static_cast<T>(A.lam[mode_idx]);
    const long long vec = static_cast<long long>(blockIdx.z) * A.nmode + mode_idx;
    const unsigned short *pt = A.ptype + A.plane_base[l];
    auto row = [&](int z) -> const T * { return A.zt + pt[z] * kCoefPerPlane; };
    const Rows<T> f{const_cast<T *>(A.f[l]) + vec * nz * A.pitch, A.pitch, 0, false};
    const Rows<T> u{A.u[l] + vec * nz * A.pitch, A.pitch, 0, false};
    const Rows<T> fc{A.fw[l + 1] + vec * nzc * A.pitch, A.pitch, 0, false};
    const int p0 = static_cast<int>(static_cast<long long>(nzc) * blockIdx.x / gridDim.x);
    const int p1 = static_cast<int>(static_cast<long long>(nzc) * (blockIdx.x + 1) / gridDim.x);
    const int nch = A.pitch / Chunk<T, K>::CH;
    restrict_planes<T, K>(p0, p1 - p0, nch, nch, u, f, nz, row, lam, l > 0,
                          [&](int Z, int c, const Chunk<T, K> &g) { g.store(fc, Z, c); });
}

}  // namespace smg
