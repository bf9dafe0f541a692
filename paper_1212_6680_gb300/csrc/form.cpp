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
// below do, sums of each form's launches, steps and waves on 152 SMs, fitted to 7880 applications timed in
// both forms (1 to 2048 by 1 to 512 by 1 to 1024 points, 1 to 32 vectors, (1,0) to (2,1) cycles; microseconds).  Of these,
// the form picked is more than 5 % slower than the other one in 1.9 %, and more than 15 % in 1 %.
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
    constexpr double kStep[10] = {1.71, 2.15, 2.51, 3.07, 4.39, 5.63, 7.35, 13.3, 14.9, 15.8};
    constexpr int kRows[10] = {1, 2, 3, 4, 6, 8, 8, 16, 16, 16};
    const int q = static_cast<int>(div_up(nx, 32));
    const int c = nx > 512 ? 7 + static_cast<int>(div_up(nx, 512)) - 2 : nx > 256 ? 6 : q <= 4 ? q - 1 : q <= 6 ? 4 : 5;
    const int W = nx > 512 ? static_cast<int>(div_up(nx, 512)) : nx > 256 ? 2 : 1, K = kRows[c], teams = 16 / W;
    const double line = W == 1 ? 0.78 + 3.77 * K : 4.87 * K;  // FP64 issue of a line's two solves a sweep
    auto relax = [&](int planes, int most) {
        if (planes == 0) return 0.0;
        const long long p = static_cast<long long>(planes) * nb;
        int R = 1;
        while (2 * R <= most && p * 2 * R <= kSMs) R *= 2;
        const double waves = static_cast<double>(div_up(p, kSMs)), rounds = static_cast<double>(solve_rounds(ny, R, teams));
        double t = 2.36 + waves * (rounds * kStep[c] + 2.0 * ny / R / teams * line);
        if (R > 1) t += (div_up(p * R, 128) - 1) * rounds * 0.7 * K;  // clusters fill 128 of the SMs at most
        return t;
    };
    double t = relax(1, 16);
    for (int n = nz; n > 1; n /= 2) t += (npre + npost) * (relax((n + 1) / 2, 8) + relax(n / 2, 8)) + 8.6;
    return t;
}

double modes_us(int nx, int ny, int nz, int nb, int npre, int npost) {
    constexpr double kPass[5] = {4.89, 9.09, 9.87, 10.8, 19.6};     // one plane on each group of lanes
    constexpr int kTables[5] = {6000, 9000, 18000, 28000, 90000};      // shared memory beside the vectors, about
    const ModalConfig cfg = modal_config(ny, true);
    const int ci = ny <= 32 ? 0 : ny <= 64 ? 1 : ny <= 128 ? 2 : ny <= 256 ? 3 : 4;
    const int L = levels_of(nz), nh = (nx + 1) / 2, sweeps = npre + npost;
    const long long stages = div_up(nh, 16);
    const long long tiles = div_up(static_cast<long long>(nz) * ((ny + 3) / 4 * 4), 64) * div_up(nh, 32) * nb;
    double t = 35.9 * div_up(tiles, kSMs) * stages + 63.2e-6 * nx * ny * nz * nb;
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
    t += 56.2 * lt + 7.1 * waves;
    for (int l = lt; l + 1 < L; ++l) {
        const int n = nz >> l;
        t += sweeps * (waves * kPass[ci] * (div_up((n + 1) / 2, groups) + div_up(n / 2, groups)) + 8.49 * ctas / kSMs * n / groups * cfg.G / 32);
    }
    for (int l = 0; l < lt; ++l) t += 52.0e-6 * ctas * cfg.G * cfg.K * (nz >> l) * sweeps;
    return t;
}

}  // namespace

bool mode_space_faster(int nx, int ny, int nz, int nb, int npre, int npost) {
    constexpr double kMargin = 0.95;
    return modes_us(nx, ny, nz, nb, npre, npost) < kMargin * planes_us(nx, ny, nz, nb, npre, npost);
}

}  // namespace smg
