// Planes per task of the 3D TMA pass (host code).
//
// A task is a 64 x 8 column of one grid over a chunk of planes; the SMs take tasks in turn (b, b + G,
// ...), x fastest, then y, then the chunks, and a pass lasts as long as its busiest SM.  Two rules:
//   - by rounds: the chunk that makes rounds of tasks x (planes + R) smallest (the 2 R warm-up stages
//     of a task carry two planes of the twenty);
//   - by cost: the chunk that makes the largest sum of task costs on an SM smallest.  In planes, a
//     plane costs 1, and TASK_DAMP more where damping acts (of its two halves of 32 columns, a warp
//     each, those that hold a damped column, or all in a damped row or plane); a task TASK_START of its
//     own; and few long tasks an SM FEW_TASKS / (tasks an SM) more, since nothing evens out what
//     differs between tasks and between SMs.
// The second is taken where it promises COST_MARGIN, the first otherwise.  By rounds alone, 192 x 192 x
// 192 gave each SM one task of 96 planes: 216 us a Faber degree, where 32-plane chunks (three of 32 on
// the busiest) take 202 and 12-plane chunks 191.
// Fitted on 899 chunks of 61 grids from 64 x 64 x 64 to 400 x 400 x 400 with layers of 10 to 40 points
// (Faber, low-storage HORK and leap-frog): at none is the choice slower than by rounds or than 32-plane
// chunks; it is within 1 % of the best chunk measured on average (4.4 % by rounds) and 9 % at worst.
// us a Faber degree by rounds and now: 192 x 192 x 192 216 and 191, 227 x 112 x 249 226 and 201, 256 x 128 x
// 128 145 and 130, 64 x 64 x 64 38 and 31, 100 x 95 x 260 100 and 95, 128 x 128 x 128 78 and 74.  Chunks under
// 12 planes were not measured.
#pragma once

#include <algorithm>
#include <vector>

namespace ewv {

struct Grid3 {
    int nx, ny, nz, pml;
    bool fs;              // free surface: no damping at the first planes
};
constexpr double TASK_DAMP = 0.15, TASK_START = 1.5, FEW_TASKS = 0.12, COST_MARGIN = 0.03;
constexpr int MIN_PLANES_ROUNDS = 16, MIN_PLANES_COST = 12;

inline long long tasks_of(const std::vector<Grid3>& grids, int kc, int bx, int by) {
    long long tasks = 0;
    for (const Grid3& g : grids)
        tasks += (long long)((g.nx + bx - 1) / bx) * ((g.ny + by - 1) / by) * ((g.nz + kc - 1) / kc);
    return tasks;
}

// Cost of the busiest of nsm SMs with kc planes a task; bx, by: columns and rows of a task.
inline double busiest_sm(const std::vector<Grid3>& grids, int kc, int nsm, int bx, int by) {
    const long long tasks = tasks_of(grids, kc, bx, by);
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
                    double f = 0.0, all = 0.0;      // damped halves, and those with points
                    for (int x = x0; x < x0 + bx && x < g.nx; x += bx / 2) {
                        if (row || damped(x, std::min(x + bx / 2, g.nx), g.nx, g.pml)) f += 0.5;
                        all += 0.5 * (std::min(y0 + by, g.ny) - y0) / by;
                    }
                    sm[b] += TASK_START + (k1 - k0) + TASK_DAMP * ((k1 - k0 - dz) * f + dz * all);
                    if (++b == sm.size()) b = 0;
                }
            }
        }
    const long long most = (tasks + (long long)sm.size() - 1) / (long long)sm.size();
    return *std::max_element(sm.begin(), sm.end()) * (1.0 + FEW_TASKS / (double)most);
}

inline int planes_per_task(const std::vector<Grid3>& grids, int nsm, int bx, int by, int R) {
    int nz = 1;
    for (const Grid3& g : grids) nz = std::max(nz, g.nz);
    long long rounds_best = -1;
    double cost_best = -1.0;
    int kc_rounds = nz, kc_cost = nz;
    for (int n = 1; n == 1 || nz / n >= MIN_PLANES_COST; ++n) {
        const int kc = (nz + n - 1) / n;
        const long long rounds = (tasks_of(grids, kc, bx, by) + nsm - 1) / nsm * (kc + R);
        if ((n == 1 || nz / n >= MIN_PLANES_ROUNDS) && (rounds_best < 0 || rounds < rounds_best)) {
            rounds_best = rounds;
            kc_rounds = kc;
        }
        const double cost = busiest_sm(grids, kc, nsm, bx, by);
        if (cost_best < 0.0 || cost < cost_best) {
            cost_best = cost;
            kc_cost = kc;
        }
    }
    return cost_best < (1.0 - COST_MARGIN) * busiest_sm(grids, kc_rounds, nsm, bx, by) ? kc_cost : kc_rounds;
}

}  // namespace ewv
