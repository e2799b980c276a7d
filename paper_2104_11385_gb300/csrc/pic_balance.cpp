// pic_balance.cpp -- the load-balancing routine of arXiv 2104.11385 Sec. 2.2,
// host C++: load-balance efficiency (Eq. 1), the knapsack and Morton
// space-filling-curve policies, the improvement threshold, the Sec. 4 speedup
// model, and the cutting of boxes into work units for the persistent kernel.
#include "pic_balance.h"

#include <algorithm>
#include <cmath>
#include <numeric>

namespace pic {

double lb_efficiency(const double* costs, const int32_t* assign, int64_t nboxes, int n_workers) {
    std::vector<double> load(n_workers, 0.0);
    for (int64_t b = 0; b < nboxes; ++b) load[assign[b]] += costs[b];
    double total = 0.0, mx = 0.0;
    for (int w = 0; w < n_workers; ++w) {
        total += load[w];
        mx = std::max(mx, load[w]);
    }
    if (mx == 0.0) return 1.0;
    return (total / (double)n_workers) / mx;
}

// Greedy longest-processing-time-first with a cap on boxes per worker.
void knapsack(const double* costs, int64_t nboxes, int n_workers, double cap_factor,
              int32_t* assign) {
    std::vector<int64_t> order(nboxes);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(),
                     [&](int64_t a, int64_t b) { return costs[a] > costs[b]; });
    const int64_t cap_ceil = (nboxes + n_workers - 1) / n_workers;
    const int64_t cap_f = (int64_t)std::floor(cap_factor * (double)nboxes / (double)n_workers);
    const int64_t cap = std::max(cap_ceil, cap_f);
    // min-heap keyed by (load, worker id) over workers below the cap; a worker
    // that reaches the cap leaves the heap
    using Entry = std::pair<double, int>;
    auto cmp = [](const Entry& a, const Entry& b) {
        return a.first > b.first || (a.first == b.first && a.second > b.second);
    };
    std::vector<Entry> heap;
    heap.reserve(n_workers);
    for (int w = 0; w < n_workers; ++w) heap.push_back({0.0, w});
    std::make_heap(heap.begin(), heap.end(), cmp);
    std::vector<int64_t> cnt(n_workers, 0);
    for (int64_t b : order) {
        std::pop_heap(heap.begin(), heap.end(), cmp);
        Entry e = heap.back();
        heap.pop_back();
        assign[b] = e.second;
        e.first += costs[b];
        if (++cnt[e.second] < cap) {
            heap.push_back(e);
            std::push_heap(heap.begin(), heap.end(), cmp);
        }
    }
}

uint64_t morton_key(int dim, int64_t bx, int64_t by, int64_t bz) {
    // spread the bits of each coordinate with shift-and-mask steps
    auto spread3 = [](uint64_t v) {
        v &= 0x1fffffull;
        v = (v | (v << 32)) & 0x1f00000000ffffull;
        v = (v | (v << 16)) & 0x1f0000ff0000ffull;
        v = (v | (v << 8)) & 0x100f00f00f00f00full;
        v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
        v = (v | (v << 2)) & 0x1249249249249249ull;
        return v;
    };
    auto spread2 = [](uint64_t v) {
        v &= 0xffffffffull;
        v = (v | (v << 16)) & 0x0000ffff0000ffffull;
        v = (v | (v << 8)) & 0x00ff00ff00ff00ffull;
        v = (v | (v << 4)) & 0x0f0f0f0f0f0f0f0full;
        v = (v | (v << 2)) & 0x3333333333333333ull;
        v = (v | (v << 1)) & 0x5555555555555555ull;
        return v;
    };
    if (dim == 3)
        return spread3((uint64_t)bx) | (spread3((uint64_t)by) << 1) | (spread3((uint64_t)bz) << 2);
    return spread2((uint64_t)bx) | (spread2((uint64_t)bz) << 1);
}

void sfc(const double* costs, const int32_t* ijk, int64_t nboxes, int dim, int n_workers,
         int32_t* assign) {
    std::vector<std::pair<uint64_t, int64_t>> keyed(nboxes);
    for (int64_t b = 0; b < nboxes; ++b)
        keyed[b] = {morton_key(dim, ijk[3 * b], ijk[3 * b + 1], ijk[3 * b + 2]), b};
    std::sort(keyed.begin(), keyed.end());
    double total = 0.0;
    for (const auto& kb : keyed) total += costs[kb.second];
    double prefix = 0.0;
    int w = 0;
    for (const auto& kb : keyed) {
        assign[kb.second] = w;
        prefix += costs[kb.second];
        if (w < n_workers - 1 && prefix * (double)n_workers >= (double)(w + 1) * total) ++w;
    }
}

bool adopt(double e_old, double e_new, double theta) { return e_new >= (1.0 + theta) * e_old; }

double predicted_speedup(double e0, double x) { return std::pow(1.0 / e0, x); }

// Cuts boxes into units: a box of cost c gets ceil(c / target) units (at most
// one per min_particles particles, at least one), target = total /
// (n_workers * split).  Unit cost = box cost / units.
std::vector<Unit> make_units(const double* costs, const int64_t* np, int64_t nboxes, int n_workers,
                             int split, int64_t min_particles, bool allow_split) {
    double total = 0.0;
    for (int64_t b = 0; b < nboxes; ++b) total += costs[b];
    const double target = total / ((double)n_workers * (double)std::max(1, split));
    std::vector<Unit> units;
    units.reserve(nboxes);
    for (int64_t b = 0; b < nboxes; ++b) {
        int64_t k = 1;
        if (allow_split && target > 0.0 && costs[b] > target) {
            k = (int64_t)std::ceil(costs[b] / target);
            int64_t kmax = std::max<int64_t>(1, np[b] / std::max<int64_t>(1, min_particles));
            k = std::min(k, kmax);
            k = std::min<int64_t>(k, 1 << 20);
        }
        for (int64_t c = 0; c < k; ++c) units.push_back(Unit{(int32_t)b, (int32_t)c, (int32_t)k, costs[b] / (double)k});
    }
    return units;
}

// A unit costs about 14 us of scheduling, tile staging and partly filled rounds
// before any balance is gained (128^3 foil, 8.4 M particles on 304 CTAs: 1.48 ms
// in units of 1725 particles, 1.31 ms in units of 6900), so units hold at least
// 4096 particles, or a quarter of a worker's share where that is less.  Where a
// quarter is below 1024 it is too little, and 1024 may leave workers without a
// unit: there they hold what gives no more units than workers (or a worker's
// share, if the boxes alone are more), between 256, one round of a CTA's
// threads, and 1024.  Particle kernel per step, 304 CTAs, with units of 256 /
// 1024 / this rule: foil of 64^3 cells and 131 thousand particles, quadratic,
// 178 / 211 / 165 us, 262 thousand, linear, 137 / 99 / 102, 32^3 plasma 133 / 92 / 81.
int64_t min_unit_particles(const int64_t* np, int64_t nboxes, int n_workers) {
    int64_t total = 0;
    for (int64_t b = 0; b < nboxes; ++b) total += np[b];
    const int64_t nw = std::max(1, n_workers), quarter = total / (4 * nw);
    if (quarter >= 1024) return std::min<int64_t>(4096, quarter);
    auto fits = [&](int64_t m) {
        int64_t units = 0;
        for (int64_t b = 0; b < nboxes; ++b) units += std::max<int64_t>(1, np[b] / m);
        return units <= nw;
    };
    int64_t lo = 256, hi = 1024;
    if (!fits(hi)) return std::min(hi, std::max(lo, total / nw));
    while (lo < hi) {
        const int64_t m = (lo + hi) / 2;
        if (fits(m)) hi = m;
        else lo = m + 1;
    }
    return hi;
}

// A mapping with at most half as many units as persistent CTAs (8 boxes on 152
// SMs) would leave most of the chip idle, so each unit is then cut into equal
// parts that different CTAs pull, down to 256 particles (one round of a CTA's
// threads).  The plan itself, its costs and its efficiency stay per unit.  16^3
// cells in 8 boxes, 32768 particles, one CTA per SM: the particle kernel takes 40
// us against 137.
int64_t unit_share(int64_t nu, int ctas, int64_t np) {
    if (nu <= 0 || 2 * nu > ctas) return 1;
    return std::max<int64_t>(1, std::min<int64_t>(ctas / nu, np / nu / 256));
}

}  // namespace pic
