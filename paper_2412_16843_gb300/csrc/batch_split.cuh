// CTAs an instance of a batched step (host code, no CUDA).
//
// One CTA an instance does the most work a second when instances abound, but
// the launch ends with its slowest instance: of 64 instances of 2k to 131k
// cells the largest was alone on one SM for most of the launch.  Larger
// clusters shorten that tail and leave fewer slots.  For every cluster size n
// the instances (largest first) are laid out over its slots, and the size with
// the earliest end is taken, a larger one only for a gain of 3 %.  A step of c cells on n CTAs is taken as
// (a + 0.009 us (n - 1)) c / n plus 0.6 ms of barriers and shared-memory
// multigrid tails; a, by precision and threads, is the cost a cell measured on
// single instances of 131k cells.  How many V-cycles an instance needs is not
// known beforehand: in FP32, where the solve is most of a step, the slowest of
// many large instances took up to 1.35 times the typical one, so 0.4 of the
// largest instance's step is added to the end (in FP64 the stages are most of
// a step, and nothing is added).
//
// Measured, ms a step of the whole batch (FP32, 1024 threads; resident clusters
// on 152 SMs 152, 76, 36, 15, 7); * is the size taken:
//   CTAs          1       2       4       8      16
//   sweep, 64   26.8    14.8     8.4     7.7*   12.5
//   sweep, 160  30.6    17.1    12.7*   20.2    33.7
//   sweep, 512  34.5    31.0*   38.3    62.6   104.5
// Over 142 batches measured at every size (8 to 512 instances of the 2D sweep,
// 8 to 160 3D grids of 16^3 to 64^3, both precisions, 256 to 1024 threads) the
// size taken is within 2 % of the fastest in 133, 16 % off at most and 0.5 % on
// average.
#pragma once

#include <algorithm>
#include <functional>
#include <vector>

namespace cdi {

// cells[n]: the instances' cell counts in decreasing order; slots[k]: clusters
// of 2^k CTAs resident at once, k < sizes.  Returns log2 of the cluster size.
inline int batch_split_choice(const long* cells, int n, const int* slots, int sizes, bool fp64, int threads) {
    const double a = fp64 ? (threads == 256 ? 0.85 : threads == 512 ? 0.72 : 0.68)
                          : (threads == 256 ? 0.42 : threads == 512 ? 0.25 : 0.19);
    int best = 0;
    double best_end = 0.0;
    for (int k = 0; k < sizes; ++k) {
        const int ctas = 1 << k;
        auto step = [&](long c) { return (a + 0.009 * (ctas - 1)) * (double)c / ctas + 600.0; };
        std::vector<double> end(std::max(1, std::min(slots[k], n)), 0.0);  // a min-heap of the slots' ends
        for (int i = 0; i < n; ++i) {
            std::pop_heap(end.begin(), end.end(), std::greater<double>());
            end.back() += step(cells[i]);
            std::push_heap(end.begin(), end.end(), std::greater<double>());
        }
        const double t = *std::max_element(end.begin(), end.end()) + (fp64 ? 0.0 : 0.4) * step(cells[0]);
        if (k == 0 || t < 0.97 * best_end) {
            best_end = t;
            best = k;
        }
    }
    return best;
}

}  // namespace cdi
