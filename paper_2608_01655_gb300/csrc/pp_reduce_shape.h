// How many CTAs share an item of the exact reduction: plain C++, no device.
#pragma once

#include <algorithm>
#include <cstddef>

namespace pp {

constexpr int kPortable = 8;     // CTAs of a cluster that every device takes
constexpr int kReduceCtas = 128;            // of all items in flight (16 clusters of 8, 15 of which run at a time on 152
                                            // SMs: a batch of 16 685 us; all at once on 6 CTAs each, 712)

// What an item may cost, in microseconds, see set_spending.
struct Spending {
    float price = 0.f;              // of one price
    float sweep[2] = {};            // of a sweep of all rows: at most 128 columns, more
    int evals[2] = {};              // prices tried at most (0: the sweep takes the item)
};

// Layout of an instance's reduction.  bins = 0: this tree is not reduced.
struct ReduceShape {
    int bins = 0, nslots = 0, nstreams = 0, nlev = 0, ntop = 0, toptiles = 0, max_kids = 0;
    int ncl = 0, cl[8] = {}, acc[8] = {}, path[8] = {}, acc_global = 0;      // cluster sizes, largest first
    int wide = 0;                   // clusters above the portable size that fit the device
    Spending spending[8];           // by cluster size
    size_t item_bytes = 0;          // scratch of one item
};

// `wide` clusters of the largest size, above the portable one, run at a time:
// with none the sizes above it are left out, and without any other the tree
// is not reduced
inline void set_wide(ReduceShape &r, int wide)
{
    r.wide = wide;
    if (wide > 0) return;
    int drop = 0;
    while (drop < r.ncl && r.cl[drop] > kPortable) ++drop;
    for (int x = drop; x < r.ncl; ++x) {
        r.cl[x - drop] = r.cl[x];
        r.acc[x - drop] = r.acc[x];
        r.path[x - drop] = r.path[x];
        r.spending[x - drop] = r.spending[x];
    }
    r.ncl -= drop;
    if (r.ncl == 0) r.bins = 0;
}

// As many CTAs per item as the items in flight leave SMs for (whole plans,
// 16 CTAs an item against 8: 2 starts of 200,000 rows 11.9 and 15.7 ms, 8
// starts of 20,000 10.4 and 11.1 although one start in eight waits; 16
// starts of 50,000 41.7 and 29.3, half of them waiting)
inline int cluster_index(const ReduceShape &r, int items)
{
    int x = 0;
    while (x + 1 < r.ncl && ((r.cl[x] > kPortable && items * 7 > r.wide * 8) || r.cl[x] * items > kReduceCtas)) ++x;
    return x;
}

// No more is spent on an item before it is left to the sweep than a sweep of
// all rows would take, so that one which the reduction cannot solve takes about
// twice as long as without it at most (with 16 prices and three DPs for every
// item, up to 5.6 times).
// A price, by the tiles that follow one another: 3.3 us on a star of 800 rows
// (one tile), 5.0 on a random tree of 800 (6), 12.5 on a chain of 800 (25), 6.0
// on a random tree of 1,600 on 6 CTAs (4, and 2 in the last bin), 10.9 on
// chains of 256 (18 and 1).  The exact evaluation with the losses takes two.
// A sweep: pruning and walk, then 0.035 to 0.045 us a row of at most 128
// columns of unit weights, 0.065 to 0.1 of more, 0.18 to 0.4 with weights
// (0.25 here: they sooner pay).
// A tree whose sweep takes less than six prices is left to it at once: three
// prices, the exact evaluation and a DP would not fit (chains of 400 and 800
// rows, 128 columns at most: 85 and 115 us with the prices, 55 and 72 without).
inline void set_spending(ReduceShape &r, int n, int max_weight, int max_evals)
{
    for (int x = 0; x < r.ncl; ++x) {
        Spending &s = r.spending[x];
        s.price = 2.6f + 0.4f * (float)(r.path[x] + r.toptiles) + (r.cl[x] > 1 ? 1.f : 0.f);
        for (int many = 0; many < 2; ++many) {
            s.sweep[many] = 25.f + (float)n * (max_weight > 1 ? 0.25f : many ? 0.07f : 0.04f);
            s.evals[many] = s.sweep[many] < 6 * s.price ? 0 : std::min(max_evals, (int)(s.sweep[many] / s.price) - 2);
        }
    }
}

}  // namespace pp
