// How many CTAs share an item of the exact reduction: plain C++, no device.
#pragma once

namespace pp {

constexpr int kPortable = 8;     // CTAs of a cluster that every device takes
constexpr int kReduceCtas = 128;            // of all items in flight (16 clusters of 8, 15 of which run at a time on 152
                                            // SMs: a batch of 16 685 us; all at once on 6 CTAs each, 712)

// Layout of an instance's reduction.  bins = 0: this tree is not reduced.
struct ReduceShape {
    int bins = 0, nslots = 0, nstreams = 0, nlev = 0, ntop = 0, max_kids = 0;
    int ncl = 0, cl[8] = {}, acc[8] = {}, acc_global = 0;      // cluster sizes, largest first
    int wide = 0;                   // clusters above the portable size that fit the device
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

}  // namespace pp
