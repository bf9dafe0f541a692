// form.cpp -- which form of the FP64 V-cycle is faster for a size: mode space (modal.cuh) or the plane kernels
// (plane_relax.cuh, plane_lean.cuh, plane_wide.cu).
//
// Mode space pays for two transforms, FP64 products of order nx / 2 over all lines in tiles of 64 lines, and then
// relaxes every plane of every mode in few steps; the plane kernels pay for a chain of 4P - 3 dependent line solves
// in each relaxation, whatever the number of lines, and for FP64 issue in the SMs that the planes fill.  So the planes
// win where there are few lines (one or two planes, planes of a line or two) and where long lines fill the chip, and
// mode space in between.  (1,0) applications in us, planes / mode space: 2048x1x1 14 / 2350, 100x1x1 4 / 152, 128x64x1
// 77 / 153, 2048x24x16 3394 / 4584, 1280x80x80 11103 / 20411, 512^3 64100 / 137819; 24x20x16 321 / 82, 128^3 2349 / 971,
// 768x48x48 4815 / 2983, 320^3 34601 / 25498.  No single product of the sizes draws that line: the two estimates
// below do, sums of each form's launches, steps and waves on 152 SMs, fitted to 8477 applications timed in
// both forms (1 to 2048 by 1 to 512 by 1 to 1024 points, 1 to 64 vectors, (1,0) to (2,1) cycles; microseconds).  They meet
// the times within 10 %, and of these the form picked is more than 5 % slower than the other one in 1.2 %.
#include <algorithm>

#include "modal.h"
#include "smg_internal.h"

namespace smg {

namespace {

constexpr int kSMs = 152;

long long div_up(long long a, long long b) { return (a + b - 1) / b; }
int levels_of(int n) { return n <= 1 ? 1 : 1 + levels_of(n / 2); }

// Dependent line solves of one 2D cycle on R CTAs of `teams` teams each: per 2D level two solves of the even lines
// and two of the odd ones, then the last line.
long long solve_rounds(int ny, int R, int teams) {
    long long s = 1;
    for (int n = ny; n > 1; n /= 2) s += 2 * (div_up(div_up((n + 1) / 2, R), teams) + div_up(div_up(n / 2, R), teams));
    return s;
}

double planes_us(int nx, int ny, int nz, int nb, int npre, int npost) {
    // rows a lane K, warps a line W, and the time of one dependent line solve: K = 1, 2, 3, 4, 6, 8; two warps of 8; two to
    // four warps of 16
    constexpr double kStep[10] = {1.72, 2.15, 2.53, 3.08, 4.42, 5.64, 7.5, 14.0, 15.4, 15.9};
    constexpr int kRows[10] = {1, 2, 3, 4, 6, 8, 8, 16, 16, 16};
    constexpr int kClusters[5] = {kSMs, 76, 36, 15, 7};  // clusters of 1, 2, 4, 8 and 16 CTAs that run at once
    const int q = static_cast<int>(div_up(nx, 32));
    const int c = nx > 512 ? 7 + static_cast<int>(div_up(nx, 512)) - 2 : nx > 256 ? 6 : q <= 4 ? q - 1 : q <= 6 ? 4 : 5;
    const int W = nx > 512 ? static_cast<int>(div_up(nx, 512)) : nx > 256 ? 2 : 1, K = kRows[c], teams = 16 / W;
    const double line = W == 1 ? 0.79 + 3.65 * K : 4.58 * K;  // FP64 issue of a line's two solves a sweep
    auto relax = [&](int planes, int most) {
        if (planes == 0) return 0.0;
        const long long p = static_cast<long long>(planes) * nb;
        int R = 1, lr = 0;
        while (2 * R <= most && p * 2 * R <= kSMs) R *= 2, ++lr;
        return 2.27 + div_up(p, kClusters[lr]) * (solve_rounds(ny, R, teams) * kStep[c] + 2.0 * ny / R / teams * line);
    };
    double t = relax(1, 16);
    for (int n = nz; n > 1; n /= 2) t += (npre + npost) * (relax((n + 1) / 2, 8) + relax(n / 2, 8)) + 8.66;
    return t;
}

double modes_us(int nx, int ny, int nz, int nb, int npre, int npost) {
    constexpr double kPass[5] = {4.9, 9.19, 9.33, 10.2, 18.5};     // one plane on each group of lanes
    constexpr int kTables[5] = {6000, 9000, 18000, 28000, 90000};      // shared memory beside the vectors, about
    const ModalConfig cfg = modal_config(ny, true);
    const int ci = ny <= 32 ? 0 : ny <= 64 ? 1 : ny <= 128 ? 2 : ny <= 256 ? 3 : 4;
    const int L = levels_of(nz), nh = (nx + 1) / 2, sweeps = npre + npost;
    const long long stages = div_up(nh, 16);
    const long long tiles = div_up(static_cast<long long>(nz) * ((ny + 3) / 4 * 4), 64) * div_up(nh, 32) * nb;
    double t = 35.1 * div_up(tiles, kSMs) * stages + 55.2e-6 * nx * ny * nz * nb;
    // the tail: first level whose vectors fit, CTAs an SM, and a CTA's passes over its planes
    const double row = static_cast<double>(div_up(ny, cfg.K)) * cfg.K * 8, most = 225.0 * 1024;
    int lt = 0;
    double smem = 0;
    for (; lt < L; ++lt) {
        smem = kTables[ci];
        for (int l = lt; l < L; ++l) smem += (l == lt ? 1 : 2) * row * (nz >> l);
        if (smem < most) break;
    }
    const double ctas = static_cast<double>(nx) * nb;
    const int per_sm = ctas <= kSMs ? 1 : 4 * (smem + 2048) <= most ? 4 : 2 * (smem + 2048) <= most ? 2 : 1;
    const double waves = static_cast<double>(div_up(static_cast<long long>(nx) * nb, static_cast<long long>(kSMs) * per_sm));
    const int groups = (per_sm <= 2 ? 256 : 128) / cfg.G;
    t += 61.2 * lt + 8.2 * waves;
    for (int l = lt; l + 1 < L; ++l) {
        const int n = nz >> l;
        t += sweeps * (waves * kPass[ci] * (div_up((n + 1) / 2, groups) + div_up(n / 2, groups)) + 8.74 * ctas / kSMs * n / groups * cfg.G / 32);
    }
    for (int l = 0; l < lt; ++l) t += 47.4e-6 * ctas * cfg.G * cfg.K * (nz >> l) * sweeps;
    return t;
}

}  // namespace

bool mode_space_faster(int nx, int ny, int nz, int nb, int npre, int npost) {
    return modes_us(nx, ny, nz, nb, npre, npost) < planes_us(nx, ny, nz, nb, npre, npost);
}

}  // namespace smg
