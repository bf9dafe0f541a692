// sine.cu -- the FP32 transforms of the x-lines into their sine eigenvectors and back (modal.cuh).
//
// The orthonormal eigenvectors of tridiag(-1, 2, -1) of order n are s_k(x) = sqrt(2 / (n + 1))
// sin(pi k x / (n + 1)), x, k = 1 .. n.  s_k is symmetric about the middle for odd k and antisymmetric
// for even k, so a line is folded first (x with n + 1 - x: sum and difference) and each parity is a
// product of half the order: n / 2 multiply-adds a point and transform, as two dense products over all
// lines.  No fast sine transform: n + 1 is 129, 257 or 1281 for the sizes in use (few small factors), and
// at n <= 256 the product costs less than the passes over memory of a factored transform.
//
// Both directions are C[col][line] += B[k][col] A[k][line] for two parities.  A CTA of 128 threads forms
// 16 LT lines by 32 columns of each parity, a thread LT lines by 4 columns of each, in packed pairs of
// lines (fma.rn.f32x2, two cycles of the FMA pipe each: at LT = 8 32 of them a step, against 6
// shared-memory reads of 16 bytes and 8 moves that duplicate B's values).  LT = 8 while that gives every SM
// its CTAs, LT = 4 for smaller problems.  Operands come by cp.async three stages
// ahead.  Each stage's sum (16 terms) is formed apart and added once, which keeps the rounding error
// of a long line that of a short sum (128 points: 0.94e-7 of the result's norm instead of 1.5e-7, 1280:
// 1.5e-7).
//
// Forward, lines of up to 256 points (FP64 input: 128) are folded on their way into shared memory; longer
// ones by a pass of their own (folds_on_the_way).
#include "modal.cuh"

namespace smg {
namespace {

constexpr int kBK = 16;      // terms per stage
constexpr int kBN = 32;      // columns of a parity per CTA
constexpr int kNT = 128;     // threads: 16 groups of lines by 8 of columns
constexpr int kStages = 3;

using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 dup2(float v) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
    return d;
}
__device__ __forceinline__ void unpack2(float &x, float &y, f32x2 v) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }

template <int LT>
struct Smem {
    static constexpr int BM = 16 * LT, LD = BM + 4;
    float a[kStages][2][kBK * LD];   // [stage][parity]
    float b[kStages][2][kBK * kBN];
    long long off[BM];               // first element of each line in the physical vector, -1: none
};

__device__ __forceinline__ void cp_async16_zfill(void *dst, const void *src, bool in) {
    const int n = in ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(dst))), "l"(src),
                 "r"(n)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int LT>
__device__ __forceinline__ void line_offsets(Smem<LT> &s, const SineArgs &g, long long p0) {
    for (int i = threadIdx.x; i < Smem<LT>::BM; i += kNT) {
        const long long p = p0 + i;
        const unsigned z = static_cast<unsigned>(p / g.pitch), y = static_cast<unsigned>(p - static_cast<long long>(z) * g.pitch);
        s.off[i] = (p < static_cast<long long>(g.nz) * g.pitch && y < static_cast<unsigned>(g.ny))
                       ? (static_cast<long long>(z) * g.ny + y) * g.nx : -1;
    }
}

// Terms k0 .. k0+15 of both parities' matrices, columns c0 .. c0+31 (the matrices are padded).
template <int LT>
__device__ __forceinline__ void fetch_b(Smem<LT> &s, int st, const float *m, int hp, int k0, int c0) {
#pragma unroll
    for (int i = 0; i < 2 * kBK * kBN / 4 / kNT; ++i) {
        const int e = threadIdx.x + i * kNT, par = e / (kBK * kBN / 4), q = e % (kBK * kBN / 4), r = q / (kBN / 4), c = q % (kBN / 4) * 4;
        cp_async16_zfill(&s.b[st][par][r * kBN + c], m + static_cast<long long>(par) * hp * hp + static_cast<long long>(k0 + r) * hp + c0 + c, true);
    }
}
// The same terms of A, from [k][line] in global memory: parity 0 has n0 of them, parity 1, which follows, n1.
template <int LT>
__device__ __forceinline__ void fetch_a(Smem<LT> &s, int st, const float *a, int n0, int n1, long long lines, int k0, long long p0) {
    constexpr int W = Smem<LT>::BM / 4;
#pragma unroll
    for (int i = 0; i < 2 * kBK * W / kNT; ++i) {
        const int e = threadIdx.x + i * kNT, par = e / (kBK * W), q = e % (kBK * W), r = q / W, c = q % W * 4;
        const bool in = k0 + r < (par ? n1 : n0) && p0 + c < lines;
        cp_async16_zfill(&s.a[st][par][r * Smem<LT>::LD + c], in ? a + static_cast<long long>((par ? n0 : 0) + k0 + r) * lines + p0 + c : a, in);
    }
}

__device__ __forceinline__ void thread_tile(int &ty, int &tx) {
    tx = threadIdx.x & 7;   // a warp: 8 groups of columns by 4 of lines (one wavefront a read)
    ty = threadIdx.x >> 3;
}

template <int LT>
using Acc = f32x2[2][4][LT / 2];   // [parity][column][pair of lines]

// acc += this stage's sum
template <int LT>
__device__ __forceinline__ void stage_sum(Acc<LT> &acc, const Smem<LT> &s, int st, int ty, int tx) {
    constexpr int LD = Smem<LT>::LD;
    Acc<LT> part;
    // LT = 8, two CTAs an SM: the next term's operands are read while one is multiplied (at three CTAs, 168
    // registers a thread, the compiler reads them when they are needed: 270 instead of 235 us at 1280 points)
    constexpr bool kAhead = LT == 8;
    f32x2 av[2][2][LT / 2];
    float4 bq[2][2];
    auto read = [&](int k, int to) {
#pragma unroll
        for (int par = 0; par < 2; ++par) {
#pragma unroll
            for (int h = 0; h < LT / 4; ++h) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&s.a[st][par][k * LD + ty * LT + 4 * h]);
                av[to][par][2 * h] = v.x;
                av[to][par][2 * h + 1] = v.y;
            }
            bq[to][par] = *reinterpret_cast<const float4 *>(&s.b[st][par][k * kBN + tx * 4]);
        }
    };
    if (kAhead) read(0, 0);
#pragma unroll
    for (int k = 0; k < kBK; ++k) {
        const int c = kAhead ? k & 1 : 0;
        if (!kAhead) read(k, 0);
        else if (k + 1 < kBK) read(k + 1, c ^ 1);
#pragma unroll
        for (int par = 0; par < 2; ++par) {
            const float4 b = bq[c][par];
            const f32x2 bv[4] = {dup2(b.x), dup2(b.y), dup2(b.z), dup2(b.w)};
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < LT / 2; ++i) part[par][j][i] = k == 0 ? mul2(av[c][par][i], bv[j]) : fma2(av[c][par][i], bv[j], part[par][j][i]);
        }
    }
#pragma unroll
    for (int par = 0; par < 2; ++par)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < LT / 2; ++i) acc[par][j][i] = add2(acc[par][j][i], part[par][j][i]);
}

template <int LT>
__device__ __forceinline__ void clear(Acc<LT> &acc) {
#pragma unroll
    for (int par = 0; par < 2; ++par)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < LT / 2; ++i) acc[par][j][i] = 0ull;
}

// The product over all terms with A in global memory, three stages in flight.
template <int LT>
__device__ __forceinline__ void product(Acc<LT> &acc, Smem<LT> &s, const float *a, int n0, int n1, long long lines, const float *m,
                                        int hp, long long p0, int c0, int ty, int tx) {
    const int nk = (n0 + kBK - 1) / kBK;
    for (int q = 0; q < kStages - 1; ++q) {
        if (q < nk) {
            fetch_a<LT>(s, q, a, n0, n1, lines, q * kBK, p0);
            fetch_b<LT>(s, q, m, hp, q * kBK, c0);
        }
        cp_async_commit();
    }
    for (int kt = 0; kt < nk; ++kt) {
        cp_async_wait_group<kStages - 2>();
        __syncthreads();  // stage kt is there, and everybody is done with the one refilled next
        const int n = kt + kStages - 1;
        if (n < nk) {
            fetch_a<LT>(s, n % kStages, a, n0, n1, lines, n * kBK, p0);
            fetch_b<LT>(s, n % kStages, m, hp, n * kBK, c0);
        }
        cp_async_commit();
        stage_sum<LT>(acc, s, kt % kStages, ty, tx);
    }
}

// Columns of the forward product: mode rows of the result, LT lines a thread.
template <int LT>
__device__ __forceinline__ void store_modes(const Acc<LT> &acc, float *o, const SineArgs &g, long long lines, long long p0, int c0, int ty,
                                            int tx) {
    const int ne = g.nx / 2;
#pragma unroll
    for (int par = 0; par < 2; ++par)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = c0 + tx * 4 + j;
            if (c >= (par ? ne : g.nh)) continue;
            float *row = o + static_cast<long long>(par ? g.nh + c : c) * lines + p0 + ty * LT;
#pragma unroll
            for (int h = 0; h < LT / 4; ++h)
                if (p0 + ty * LT + 4 * h < lines) {  // lines is a multiple of 4
                    const ulonglong2 v{acc[par][j][2 * h], acc[par][j][2 * h + 1]};
                    *reinterpret_cast<ulonglong2 *>(row + 4 * h) = v;
                }
        }
}

template <class S> __device__ __forceinline__ float in_val(S v);
template <> __device__ __forceinline__ float in_val<float>(float v) { return v; }
template <> __device__ __forceinline__ float in_val<double>(double v) { return narrow_f64(v); }

// fhat[mode][line] = sum_x s_mode(x) f[line][x], modes in the order odd, even, folded on the way in: a
// thread takes one pair of points of every 8th line of a stage.
template <int LT, class S>
__device__ __forceinline__ void in_fold_body(const SineArgs &g, const S *__restrict__ f, float *__restrict__ o, int line_tile, int mode_tile,
                                             unsigned char *smem_raw) {
    Smem<LT> &s = *reinterpret_cast<Smem<LT> *>(smem_raw);
    constexpr int BM = Smem<LT>::BM, LD = Smem<LT>::LD, NL = BM * kBK / kNT;
    const long long lines = static_cast<long long>(g.nz) * g.pitch, p0 = static_cast<long long>(line_tile) * Smem<LT>::BM;
    const int c0 = mode_tile * kBN, ne = g.nx / 2, nk = (g.nh + kBK - 1) / kBK;
    const float *m = static_cast<const float *>(g.mat);
    int ty, tx;
    thread_tile(ty, tx);
    line_offsets<LT>(s, g, p0);
    fetch_b<LT>(s, 0, m, g.hp, 0, c0);
    pdl_wait();
    __syncthreads();
    const int lx = threadIdx.x % kBK, ll = threadIdx.x / kBK;
    S ra[NL], rb[NL];
    auto fetch = [&](int k0) {
        const int x = k0 + lx, xm = g.nx - 1 - x;
        const bool in = x < g.nh, two = in && xm != x;
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const long long q = s.off[ll + i * (kNT / kBK)];
            ra[i] = (in && q >= 0) ? f[q + x] : S(0);
            rb[i] = (two && q >= 0) ? f[q + xm] : S(0);
        }
    };
    auto fold = [&](int st, int k0) {
        const bool two = k0 + lx < ne;  // the middle point of an odd line has no partner: odd modes only
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const float u = in_val<S>(ra[i]), v = in_val<S>(rb[i]);
            s.a[st][0][lx * LD + ll + i * (kNT / kBK)] = u + v;
            s.a[st][1][lx * LD + ll + i * (kNT / kBK)] = two ? u - v : 0.0f;
        }
    };
    Acc<LT> acc;
    clear<LT>(acc);
    fetch(0);
    fold(0, 0);
    cp_async_wait();
    __syncthreads();
    for (int kt = 0; kt < nk; ++kt) {
        const int cur = kt & 1;
        const bool more = kt + 1 < nk;
        if (more) {
            fetch((kt + 1) * kBK);
            fetch_b<LT>(s, cur ^ 1, m, g.hp, (kt + 1) * kBK, c0);
        }
        stage_sum<LT>(acc, s, cur, ty, tx);
        if (more) fold(cur ^ 1, (kt + 1) * kBK);
        cp_async_wait();
        __syncthreads();
    }
    store_modes<LT>(acc, o, g, lines, p0, c0, ty, tx);
}

template <int LT, class S>
__global__ void __launch_bounds__(kNT) in_fold_kernel(const __grid_constant__ SineArgs g, const S *__restrict__ f, float *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_trigger();
    const long long rhs = blockIdx.z;
    in_fold_body<LT, S>(g, f + rhs * g.nx * g.ny * g.nz, out + rhs * g.nx * g.nz * g.pitch, blockIdx.x, blockIdx.y, smem_raw);
}
__global__ void __launch_bounds__(kNT) in_batch_kernel(const SineJob *__restrict__ jobs, const SineTile *__restrict__ tiles, const int *active) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SineTile t = tiles[blockIdx.x];
    if (active[t.sys] != 1) return;
    const SineJob j = jobs[t.sys];
    in_fold_body<8, float>(j.g, j.in, j.fh, t.line_tile, t.mode_tile, smem_raw);
}

// The fold of long lines alone: e[x][line] = f(x) + f(mirror), then o[x][line] = f(x) - f(mirror), 32 pairs by 64
// lines a CTA through shared memory (both sides in whole sectors).  HBM: reads each point once, writes 4 bytes.
template <class S>
__global__ void __launch_bounds__(256) fold_kernel(const __grid_constant__ SineArgs g, const S *__restrict__ f, float *__restrict__ out) {
    __shared__ float e[32][65], o[32][65];
    pdl_trigger();
    const long long rhs = blockIdx.z, lines = static_cast<long long>(g.nz) * g.pitch, p0 = static_cast<long long>(blockIdx.x) * 64;
    const int x0 = blockIdx.y * 32, lane = threadIdx.x & 31, w = threadIdx.x >> 5, ne = g.nx / 2;
    f += rhs * g.nx * g.ny * g.nz;
    out += rhs * g.nx * lines;
    pdl_wait();
    const int x = x0 + lane, xm = g.nx - 1 - x;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const long long p = p0 + w + 8 * i, z = p / g.pitch, y = p - z * g.pitch;
        const bool in = p < lines && y < g.ny && x < g.nh;
        const S *r = f + (z * g.ny + y) * g.nx;
        const float u = in ? in_val<S>(r[x]) : 0.0f, v = in && xm != x ? in_val<S>(r[xm]) : 0.0f;
        e[lane][w + 8 * i] = u + v;
        o[lane][w + 8 * i] = u - v;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < 32 * 64; q += 256) {
        const int r = q >> 6, c = q & 63;
        if (p0 + c >= lines) continue;
        if (x0 + r < g.nh) out[static_cast<long long>(x0 + r) * lines + p0 + c] = e[r][c];
        if (x0 + r < ne) out[static_cast<long long>(g.nh + x0 + r) * lines + p0 + c] = o[r][c];
    }
}

template <int LT>
__global__ void __launch_bounds__(kNT, LT == 8 ? 2 : 4) in_kernel(const __grid_constant__ SineArgs g, const float *__restrict__ a, float *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_trigger();
    pdl_wait();
    Smem<LT> &s = *reinterpret_cast<Smem<LT> *>(smem_raw);
    const long long lines = static_cast<long long>(g.nz) * g.pitch, p0 = static_cast<long long>(blockIdx.x) * Smem<LT>::BM, rhs = blockIdx.z;
    const int c0 = blockIdx.y * kBN;
    int ty, tx;
    thread_tile(ty, tx);
    Acc<LT> acc;
    clear<LT>(acc);
    product<LT>(acc, s, a + rhs * g.nx * lines, g.nh, g.nx / 2, lines, static_cast<const float *>(g.mat), g.hp, p0, c0, ty, tx);
    store_modes<LT>(acc, out + rhs * g.nx * lines, g, lines, p0, c0, ty, tx);
}

template <class S> __device__ __forceinline__ S out_val(float v);
template <> __device__ __forceinline__ float out_val<float>(float v) { return v; }
template <> __device__ __forceinline__ double out_val<double>(float v) { return widen_f32(v); }
template <> __device__ __forceinline__ __nv_bfloat16 out_val<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
// A BF16 result handed out in FP64: rounded to bfloat16, then widened exactly.
struct Bf16AsF64 {
    double v;
};
template <> __device__ __forceinline__ Bf16AsF64 out_val<Bf16AsF64>(float v) {
    return Bf16AsF64{widen_f32(__bfloat162float(__float2bfloat16_rn(v)))};
}

// u[line][x] = sum_mode s_mode(x) uhat[mode][line]: both parities' sums for BN points and their mirror images,
// sum and difference staged in shared memory so that lines are written whole words in x order.
template <int LT, class S>
__device__ __forceinline__ void out_body(const SineArgs &g, const float *__restrict__ a, S *__restrict__ u, int line_tile, int mode_tile,
                                         unsigned char *smem_raw) {
    Smem<LT> &s = *reinterpret_cast<Smem<LT> *>(smem_raw);
    const long long lines = static_cast<long long>(g.nz) * g.pitch, p0 = static_cast<long long>(line_tile) * Smem<LT>::BM;
    const int c0 = mode_tile * kBN, ne = g.nx / 2;
    const float *m = static_cast<const float *>(g.mat) + 2 * static_cast<long long>(g.hp) * g.hp;
    int ty, tx;
    thread_tile(ty, tx);
    line_offsets<LT>(s, g, p0);
    pdl_wait();
    Acc<LT> acc;
    clear<LT>(acc);
    product<LT>(acc, s, a, g.nh, ne, lines, m, g.hp, p0, c0, ty, tx);
    // [line][x and mirror image] over the operand stages
    constexpr int LS = 2 * kBN + 1, BM = Smem<LT>::BM;
    static_assert(sizeof(float) * BM * LS <= sizeof(s.a), "the result tile fits over the operand stages");
    float *w = &s.a[0][0][0];
    cp_async_wait();
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < LT / 2; ++i) {
            float e0, e1, o0, o1;
            unpack2(e0, e1, acc[0][j][i]);
            unpack2(o0, o1, acc[1][j][i]);
            float *r = w + (ty * LT + 2 * i) * LS + tx * 4 + j;
            r[0] = e0 + o0;
            r[kBN] = e0 - o0;
            r[LS] = e1 + o1;
            r[LS + kBN] = e1 - o1;
        }
    __syncthreads();
    const int lane = threadIdx.x & 31, x = c0 + lane;
#pragma unroll 4
    for (int i = threadIdx.x >> 5; i < BM; i += kNT / 32) {
        const long long q = s.off[i];
        if (q < 0) continue;
        if (x < g.nh) u[q + x] = out_val<S>(w[i * LS + lane]);
        if (x < ne) u[q + g.nx - 1 - x] = out_val<S>(w[i * LS + kBN + lane]);
    }
}
template <int LT, class S>
__global__ void __launch_bounds__(kNT, LT == 8 ? 2 : 4) out_kernel(const __grid_constant__ SineArgs g, const float *__restrict__ a,
                                                            S *__restrict__ u) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_trigger();
    const long long rhs = blockIdx.z;
    out_body<LT, S>(g, a + rhs * g.nx * g.nz * g.pitch, u + rhs * g.nx * g.ny * g.nz, blockIdx.x, blockIdx.y, smem_raw);
}
__global__ void __launch_bounds__(kNT, 2) out_batch_kernel(const SineJob *__restrict__ jobs, const SineTile *__restrict__ tiles, const int *active) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SineTile t = tiles[blockIdx.x];
    if (active[t.sys] != 1) return;
    const SineJob j = jobs[t.sys];
    out_body<8, float>(j.g, j.uh, j.out, t.line_tile, t.mode_tile, smem_raw);
}

// ---- host -------------------------------------------------------------------------------------------

template <int LT>
dim3 grid_of(const SineArgs &g, int nb) {
    const long long lines = static_cast<long long>(g.nz) * g.pitch;
    return dim3(static_cast<unsigned>((lines + 16 * LT - 1) / (16 * LT)), (g.nh + kBN - 1) / kBN, nb);
}
// Whether 128-line tiles give every SM three CTAs (two run at once; a third evens out the last wave).  Applications with
// 64-line tiles / 128-line tiles, us: below the line 24x20x16 23 / 29, 101x75x53 55 / 63, 128^3 74 / 80; above it 200x128x128
// 166 / 170, 8 vectors at 96^3 305 / 322, 512x512x64 964 / 943, 384^3 2550 / 2496, 1280x80x80 757 / 703.
bool wide_tiles(const SineArgs &g, int nb) {
    const dim3 d = grid_of<8>(g, nb);
    return static_cast<long long>(d.x) * d.y * d.z >= 3 * 152;
}

template <class K, class... Args>
cudaError_t launch(K kernel, dim3 grid, size_t smem, cudaStream_t st, Args... args) {
    const cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(kernel), smem);
    return e != cudaSuccess ? e : launch_pdl(kernel, grid, dim3(kNT), smem, st, args...);
}

// Whether lines are folded on their way into shared memory, once for every column tile, or by a pass of their
// own first, whose result (4 bytes a point) the tiles then read: by the traffic, 4 tiles of FP32 (16 bytes a
// point against 24; 256^3 solve: 13.46 -> 13.31 ms) but 2 of FP64 (4 tiles: 366 us for both transforms at 256^3
// against 303).
template <class S>
bool folds_on_the_way(int nh) {
    return nh <= (sizeof(S) == 4 ? 4 : 2) * kBN;
}

template <int LT, class S>
cudaError_t in_any(const SineArgs &g, int nb, const S *f, float *out, float *scratch, cudaStream_t st, long long &launches) {
    launches += 1;
    if (folds_on_the_way<S>(g.nh)) return launch(in_fold_kernel<LT, S>, grid_of<LT>(g, nb), sizeof(Smem<LT>), st, g, f, out);
    launches += 1;
    const long long lines = static_cast<long long>(g.nz) * g.pitch;
    const cudaError_t e =
        launch_pdl(fold_kernel<S>, dim3(static_cast<unsigned>((lines + 63) / 64), (g.nh + 31) / 32, nb), dim3(256), 0, st, g, f, scratch);
    return e != cudaSuccess ? e : launch(in_kernel<LT>, grid_of<LT>(g, nb), sizeof(Smem<LT>), st, g, static_cast<const float *>(scratch), out);
}
template <class S>
cudaError_t in_of(const SineArgs &g, int nb, const void *f, float *out, float *scratch, cudaStream_t st, long long &launches) {
    const S *p = static_cast<const S *>(f);
    return wide_tiles(g, nb) ? in_any<8, S>(g, nb, p, out, scratch, st, launches) : in_any<4, S>(g, nb, p, out, scratch, st, launches);
}
template <class S>
cudaError_t out_of(const SineArgs &g, int nb, const float *a, void *u, cudaStream_t st) {
    S *p = static_cast<S *>(u);
    return wide_tiles(g, nb) ? launch(out_kernel<8, S>, grid_of<8>(g, nb), sizeof(Smem<8>), st, g, a, p)
                             : launch(out_kernel<4, S>, grid_of<4>(g, nb), sizeof(Smem<4>), st, g, a, p);
}

}  // namespace

cudaError_t sine_in_f32(const SineArgs &g, int nb, Prec type, const void *f, float *out, float *scratch, cudaStream_t st, long long &launches) {
    return type == Prec::F32 ? in_of<float>(g, nb, f, out, scratch, st, launches) : in_of<double>(g, nb, f, out, scratch, st, launches);
}
cudaError_t sine_out_f32(const SineArgs &g, int nb, const float *a, Prec value, Prec type, void *u, cudaStream_t st, long long &launches) {
    launches += 1;
    if (type == Prec::F64) return value == Prec::BF16 ? out_of<Bf16AsF64>(g, nb, a, u, st) : out_of<double>(g, nb, a, u, st);
    return type == Prec::BF16 ? out_of<__nv_bfloat16>(g, nb, a, u, st) : out_of<float>(g, nb, a, u, st);
}

int sine_line_tiles(const SineArgs &g) { return static_cast<int>(grid_of<8>(g, 1).x); }
int sine_mode_tiles(const SineArgs &g) { return static_cast<int>(grid_of<8>(g, 1).y); }

cudaError_t launch_sine_in_batch(const SineJob *jobs, const SineTile *tiles, int ntiles, const int *active, cudaStream_t st) {
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&in_batch_kernel), sizeof(Smem<8>));
    if (e != cudaSuccess) return e;
    in_batch_kernel<<<ntiles, kNT, sizeof(Smem<8>), st>>>(jobs, tiles, active);
    return cudaGetLastError();
}
cudaError_t launch_sine_out_batch(const SineJob *jobs, const SineTile *tiles, int ntiles, const int *active, cudaStream_t st) {
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&out_batch_kernel), sizeof(Smem<8>));
    if (e != cudaSuccess) return e;
    out_batch_kernel<<<ntiles, kNT, sizeof(Smem<8>), st>>>(jobs, tiles, active);
    return cudaGetLastError();
}

}  // namespace smg
