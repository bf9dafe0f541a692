// reduce.cuh -- sums for the FP64 Krylov kernels (krylov_kernels.cu, batched.cu) and division by an
// invariant.
#pragma once

#include <cuda_runtime.h>

namespace smg {

struct DSum {
    double s, c;
};

__device__ __forceinline__ void two_sum_acc(DSum &a, double b) {
    const double t = a.s + b;
    const double bp = t - a.s;
    const double err = (a.s - (t - bp)) + (b - bp);
    a.s = t;
    a.c += err;
}
__device__ __forceinline__ DSum dsum_combine(DSum a, const DSum &b) {
    two_sum_acc(a, b.s);
    a.c += b.c;
    return a;
}
__device__ __forceinline__ DSum shfl_down_dsum(const DSum &v, int o) {
    return DSum{__shfl_down_sync(0xffffffffu, v.s, o), __shfl_down_sync(0xffffffffu, v.c, o)};
}

// Inner products: every thread accumulates its (about 2N / (threads in the grid)) products with
// FMA, the block adds the thread partials through shared memory, and the last block to finish
// combines the block partials exactly (warp_sum_exact).  FP64 work per
// element stays at one FMA, which matters on GB300 where a warp's FP64 instruction holds its
// sub-partition's unit for about 64 cycles however few lanes it serves.  That prices the reductions
// themselves: a shuffle tree in every warp is 5 instructions a warp and value, a compensated sum
// 6 a term.  So the grid is one CTA of up to 1024 threads per SM (152 partials instead of 608), a
// block folds its partials four to one on full warps (36 instructions a value instead of 165), and
// one warp per value adds the block partials as integers.
constexpr int kMaxThreads = 1024;

template <int NV>
__device__ __forceinline__ void block_reduce_plain(double (&v)[NV]) {
    __shared__ double sh[NV][kMaxThreads];
    const int t = threadIdx.x;
    int n = blockDim.x;
    while (n > 32) {
        const int f = (n % 4 == 0 && n / 4 >= 32) ? 4 : 2, m = n / f;  // blockDim.x is a multiple of 64, or 32
        if (t < n)
#pragma unroll
            for (int k = 0; k < NV; ++k) sh[k][t] = v[k];
        __syncthreads();
        if (t < m)
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                double a = v[k] + sh[k][t + m];
                if (f == 4) a += sh[k][t + 2 * m] + sh[k][t + 3 * m];
                v[k] = a;
            }
        n = m;
        __syncthreads();
    }
    if (t < 32)
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const double w = __shfl_down_sync(0xffffffffu, v[k], o);
                v[k] += (t + o < n) ? w : 0.0;
            }
}

// The sum of one warp's values (kPer a lane), rounded once: integers in place of error-free FP64
// additions, of which 70 would follow one another here (a dependent FP64 instruction takes about as long
// as 15 integer ones).  Every value is aligned to the largest exponent in 128 bits -- 53 bits of mantissa
// above 56 further bits, 18 bits of headroom for the count -- so only bits below 2^-108 of the largest
// value are lost.  Sums with infinities, NaNs or exponents near the ends of the range go through
// compensated FP64 additions.  The result is lane 0's.
template <int kPer>
__device__ __forceinline__ double warp_sum_exact(const double (&p)[kPer]) {
    unsigned emax = 1u;
#pragma unroll
    for (int i = 0; i < kPer; ++i) emax = max(emax, static_cast<unsigned>(__double2hiint(p[i]) >> 20) & 0x7ffu);
    emax = __reduce_max_sync(0xffffffffu, emax);
    if (emax < 128u || emax > 2000u) {
        DSum a{p[0], 0.0};
#pragma unroll
        for (int i = 1; i < kPer; ++i) two_sum_acc(a, p[i]);
        for (int o = 16; o > 0; o >>= 1) a = dsum_combine(a, shfl_down_dsum(a, o));
        return isfinite(a.s) ? a.s + a.c : a.s;  // the correction of an infinite sum is NaN
    }
    unsigned __int128 t = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(p[i]));
        const unsigned e = static_cast<unsigned>(b >> 52) & 0x7ffu, s = emax - max(e, 1u);
        const unsigned long long m = (b & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0ull);
        const unsigned __int128 v = s <= 56u ? static_cast<unsigned __int128>(m) << (56u - s)
                                             : static_cast<unsigned __int128>(s < 120u ? m >> (s - 56u) : 0ull);
        t = (b >> 63) ? t - v : t + v;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long lo = __shfl_down_sync(0xffffffffu, static_cast<unsigned long long>(t), o);
        const unsigned long long hi = __shfl_down_sync(0xffffffffu, static_cast<unsigned long long>(t >> 64), o);
        t += (static_cast<unsigned __int128>(hi) << 64) | lo;
    }
    const unsigned long long sign = static_cast<unsigned long long>(t >> 127) << 63;
    if (sign) t = -t;
    unsigned long long hi = static_cast<unsigned long long>(t >> 64), lo = static_cast<unsigned long long>(t);
    if ((hi | lo) == 0ull) return 0.0;
    const int z = hi ? __clzll(static_cast<long long>(hi)) : 64 + __clzll(static_cast<long long>(lo));
    t <<= z;  // the leading bit to bit 127
    hi = static_cast<unsigned long long>(t >> 64);
    lo = static_cast<unsigned long long>(t);
    unsigned long long mant = hi >> 11;  // 53 bits, then round to nearest, ties to even
    const unsigned long long rest = hi & 0x7ffull;
    if (rest > 0x400ull || (rest == 0x400ull && (lo != 0ull || (mant & 1ull)))) mant += 1ull;
    // bit 108 of the sum has the value 2^(emax - 1023); a carry out of the mantissa raises the exponent
    const unsigned long long e = static_cast<unsigned long long>(static_cast<int>(emax) + 19 - z);
    return __longlong_as_double(static_cast<long long>(sign | ((e << 52) + (mant - 0x10000000000000ull))));
}

// n / d for 0 <= n < 2^31 by a multiplication (Granlund and Montgomery's invariant division).
struct FastDiv {
    unsigned mul, shift, d;
};
inline FastDiv fast_div(int d) {
    unsigned s = 0;
    while ((1ull << s) < static_cast<unsigned long long>(d)) ++s;
    return FastDiv{static_cast<unsigned>(((1ull << 32) * ((1ull << s) - d)) / d + 1), s, static_cast<unsigned>(d)};
}
__device__ __forceinline__ int div_by(int n, const FastDiv &f) {
    return static_cast<int>((__umulhi(static_cast<unsigned>(n), f.mul) + static_cast<unsigned>(n)) >> f.shift);
}
// The same for 0 <= n < 2^32 (the sum may need a 33rd bit).
__device__ __forceinline__ int div_by_wide(unsigned n, const FastDiv &f) {
    return static_cast<int>((static_cast<unsigned long long>(__umulhi(n, f.mul)) + n) >> f.shift);
}

}  // namespace smg
