// Planes per task of the 3D TMA pass (host code).
//
// A task is a 64 x 8 column of one grid over a chunk of planes; the SMs take tasks in turn (b, b + G,
// ...), x fastest, then y, then the chunks.  A pass lasts as long as its busiest SM, so the chunk is
// the one that makes the largest sum of task costs on an SM smallest.  Costs in planes:
//   - a plane of undamped points costs 1, and TASK_DAMP more where damping acts: of its two halves
//     of 32 columns (a warp each), those that hold a damped column, or all in a damped row or plane;
//   - a task costs TASK_START planes of its own (its 2 R warm-up stages carry two planes of the
//     twenty, and the stages of one task overlap the last of the one before);
//   - a shorter chunk has to be CHUNK_MARGIN better than the longer ones.
// Damped columns are why counting planes alone misleads: one long task an SM leaves some SMs with
// nothing but damped columns, many short ones mix them.  On 192 x 192 x 192, 2 chunks (one task an SM,
// 96 planes on the busiest) take 216 us a Faber degree, 6 chunks (also 96 planes) 202, 14 chunks 189.
// Fitted on 335 (size, chunk) pairs of 22 grids from 64 x 64 x 64 to 400 x 400 x 400 with layers of 10
// to 40 points: at each the choice is within 2.5 % of the best chunk measured, and no slower than that
// of the rule before (rounds of tasks x (planes + R) smallest).  Before and now, us a Faber degree:
// 192 x 192 x 192 216 and 189, 64 x 64 x 64 38 and 31, 210 x 99 x 233 200 and 185, 100 x 95 x 260 100
// and 95, 128 x 128 x 128 78 and 74, 111 x 222 x 177 141 and 138, 251 x 229 x 197 308 and 306; the same
// chunk at the others.  Chunks under 12 planes were not measured.
#pragma once

#include <algorithm>
#include <vector>

namespace ewv {

struct Grid3 {
    int nx, ny, nz, pml;
    bool fs;              // free surface: no damping at the first planes
};
constexpr double TASK_DAMP = 0.2, TASK_START = 0.5, CHUNK_MARGIN = 0.02;
constexpr int MIN_PLANES = 12;

// Cost of the busiest of nsm SMs with kc planes a task; bx, by: columns and rows of a task.
inline double busiest_sm(const std::vector<Grid3>& grids, int kc, int nsm, int bx, int by) {
    long long tasks = 0;
    for (const Grid3& g : grids)
        tasks += (long long)((g.nx + bx - 1) / bx) * ((g.ny + by - 1) / by) * ((g.nz + kc - 1) / kc);
    std::vector<double> sm((size_t)std::max(1LL, std::min<long long>(nsm, tasks)), 0.0);
    auto damped = [](int lo, int hi, int n, int pml) { return lo < pml || hi > n - pml; };
    size_t b = 0;
    for (const Grid3& g : grids)
        for (int k0 = 0; k0 < g.nz; k0 += kc) {
            const int k1 = std::min(k0 + kc, g.nz);
            const int bottom = std::max(0, k1 - std::max(k0, g.nz - g.pml));
            const int top = g.fs ? 0 : std::max(0, std::min(k1, g.pml) - k0);
            const int dz = std::min(k1 - k0, top + bottom);              // damped planes
            for (int y0 = 0; y0 < g.ny; y0 += by) {
                const bool row = damped(y0, std::min(y0 + by, g.ny), g.ny, g.pml);
                for (int x0 = 0; x0 < g.nx; x0 += bx) {
                    double f = 0.0;
                    for (int x = x0; x < x0 + bx && x < g.nx; x += bx / 2)
                        if (row || damped(x, std::min(x + bx / 2, g.nx), g.nx, g.pml)) f += 0.5;
                    sm[b] += TASK_START + (k1 - k0 - dz) * (1.0 + TASK_DAMP * f) + dz * (1.0 + TASK_DAMP);
                    if (++b == sm.size()) b = 0;
                }
            }
        }
    return *std::max_element(sm.begin(), sm.end());
}

inline int planes_per_task(const std::vector<Grid3>& grids, int nsm, int bx, int by) {
    int nz = 1;
    for (const Grid3& g : grids) nz = std::max(nz, g.nz);
    int best_kc = nz;
    double best = -1.0;
    for (int n = 1; n == 1 || nz / n >= MIN_PLANES; ++n) {
        const int kc = (nz + n - 1) / n;
        const double cost = busiest_sm(grids, kc, nsm, bx, by);
        if (best < 0.0 || cost < best * (1.0 - CHUNK_MARGIN)) {
            best = cost;
            best_kc = kc;
        }
    }
    return best_kc;
}

}  // namespace ewv
