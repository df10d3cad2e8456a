// Exact reduction of the capacity-k tree knapsack (Eq. 9) before its sweep.
//
// For a price lambda >= 0 per slot (a Lagrange multiplier of the budget), let
//   f(v) = p_v - lambda w_v + sum over the children c of v of max(0, f(c)),
//   L    = sum over the roots r of max(0, f(r)) + lambda k.
// L bounds every parent-closed set within the budget from above (relaxed
// precedence-constrained knapsack: the best closed set at price lambda, plus
// the price of the whole budget).  Let S be that best closed set (f > 0 along
// the whole path from the root).  Any closed set that holds a chunk v outside
// S has at most L - lin(v), lin(v) = sum over v's path of max(0, -f); any
// closed set without a chunk v of S at most L - lout(v), lout(v) = min over
// v's path of f.  So with V the value of any feasible set, every chunk whose
// loss (lin or lout) exceeds L - V is decided: it is the same in every optimal
// set, and the set that the backtracking of Eq. 9 returns is one of those.
// Only the undecided chunks need the DP, with the budget that the chunks
// decided "in" leave over; their optimum and their lexicographically smallest
// optimal set, joined with the decided chunks, are Eq. 9's.
//
// V comes from the DP itself: take the rows whose loss is at most some t, run
// the DP on them (V), and accept if L - V <= t, else repeat with t = L - V,
// which is then large enough by construction.  Losses are compared through
// their keys (an order-preserving 11-bit code of the loss rounded down), so
// every test errs on the side of keeping a row.  The rows kept also have to
// hang together: below a row that is decided out every row is, as it is for
// the losses themselves (lin grows down a path) and for the rounded ones, which
// are sums of whole numbers (loss_tile).
//
// A prefix tree of 50,000 chunks with the planner's profits leaves 222
// undecided rows (the mean of a plan's updates) of the 16,000 to 37,000 that the
// pruned sweep keeps, and a budget of a few hundred slots instead of 4,096: 0.17
// ms an item, where that sweep took 1.3.  More undecided rows than fit on chip
// (chunks in long chains that are worth taking only whole) go to pp_dp.cu's
// kernels with what is left of the budget; where no V is found (ties that leave
// nearly everything undecided), or none before as much time is spent as they
// take, those kernels get every row.
//
// Layout.  f is a Lindley recursion along every heavy path of the tree
// (y_i = max(0, d_i + y_(i+1)), d_i the row's own term plus its light
// children), so a path is a scan of the maps x -> max(m, s + x), and losses
// are scans the other way.  Heavy paths bound the dependent levels by
// log2(n) + 1 for every tree shape (6 to 9 on the prefix trees here, whose
// depth is 72 and more).  Rows are laid out by (bin, level, path), bottom of
// the path first, in tiles of 32 (one per warp step).  A bin is a set of
// whole subtrees of at most n / (2 bins) rows; a CTA of the item's cluster
// walks one bin or several side by side, so that levels are separated by block
// barriers only.  The few nodes above all bins form a last bin that one warp
// of every CTA walks for itself, after the cluster barrier that ends an
// evaluation.  How many CTAs share an item is decided at the launch, from the
// items that are in flight together.
#include <algorithm>
#include <climits>
#include <cstring>

#include "pp_prune.cuh"

namespace pp {

namespace {

constexpr unsigned kAll = 0xffffffffu;
constexpr int kThreads = 1024;              // per CTA
constexpr int kWarps = kThreads / 32;
constexpr int kMaxLevels = 20;              // of a bin (heavy paths: log2 of its rows, plus one)
constexpr int kMaxEvals = 16;               // prices tried per item
constexpr int kPasses = 5;                  // thresholds tried per item
constexpr int kRowCap = 1024;               // undecided rows the on-chip DP takes
constexpr int kFirstRows = 192;             // most rows of the first threshold
constexpr int kMoreRows = 640;              // of the next, where the first gave no V or a poor one
constexpr float kPassUs = 6.f;              // a threshold without its DP, and a row of the DP, us
constexpr float kRowUs = 0.08f, kWeightedRowUs = 0.11f;
constexpr int kColCap = 1024;               // its columns (budget left over)
constexpr int kPool = 112 << 10;            // its decisions, stack and row buffers, bytes
constexpr int kKeyBase = (127 << 5) - 1;    // float bits >> 18 of 1.0, minus 1
constexpr int kBins = 2048;                 // keys of 0 .. 2^62
constexpr int kKeyPad = 0xffff;
constexpr int64_t kBig = (int64_t)1 << 61;
constexpr int kMaxWeight = 1 << 22;         // weights ride in the slot code
constexpr int kMaxPathRows = 1024;          // trees with longer heavy paths are left to the sweep
constexpr int kMaxKids = 65535;             // light children of a row: its 16-bit limbs add up in 32 bits
constexpr int kRing = 3;                    // tiles of a warp in flight or in use
constexpr int kMaxTiles = 64;               // of a warp, all levels together
constexpr size_t kRingBytes = (size_t)kWarps * kRing * 512;
constexpr int kMaxBins = 16;
constexpr int kMaxTop = 256;                // rows of the last bin (every CTA walks it)
// the search's 32-bit units: the first price is 2^11 to 2^12 of them
constexpr int kUnitBits = 11;
constexpr int kClipRow = 1 << 24, kClipPath = 1 << 26, kClipPrice = 1 << 19;

// slot info.  x: bits 0-4 lanes to the left in the same path and tile, 5 the
// path comes from the previous tile, 6 top of its path, 7 its parent is in
// the last bin, 8.. weight.  y: accumulator (low half), the parent's
// accumulator for a path's top (high half); kNone: none, a root
constexpr int kCont = 32, kTop = 64, kUp = 128, kWeightShift = 8;
constexpr int kNone = 0xffff;

struct Tab {
    int n, bins, CL, nslots, ntop;
    const int2 *info;
    const int *pos;              // position of the slot's row (-1 pad)
    const uint8_t *form;         // of a tile: 1 on level 0 (paths without light children), 3 there and its first
                                 // path comes from the tile before, 0 above
    const int2 *stream;          // first tile, tiles: what one warp walks in sequence
    const int *lev;              // stream boundaries of the levels
    const int *binlev;           // [bins + 2] boundaries of a bin's entries in lev
    const int *binslot;          // [bins + 2] first slot of a bin
    const int *nacc;             // [bins + 1] accumulators of a bin
};

struct Scal {                    // per item, zeroed by the kernel
    unsigned long long maxp;
    unsigned long long sumL;
    unsigned long long sumZ[kMaxEvals];
    unsigned long long vfix[kPasses];
    unsigned long long wfix[kPasses];
    int verdict[kPasses];
    int key[kPasses];
};

struct Args {
    Tab t;
    const int64_t *profit;       // [batch][n]
    const int32_t *order;        // null: profits in preorder
    const int32_t *next, *wpre;
    const int32_t *item_budget, *item_active;
    int32_t max_budget;
    int64_t *best;
    unsigned long long *rows_kept;
    DpWork w;
    size_t item_bytes;           // of w.red_scratch
    int64_t total_weight;
    float mean_weight;           // of a row
    int32_t max_weight;
    int32_t clip_kid;            // the search's bound on what a light child adds
    Spending spending;
    const int2 *pspan;           // the pruned sweep's: see prune_item
    int32_t stack_depth;
    int32_t *status;
};

__host__ __device__ inline size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }

// Accumulators: what a row's light children add to it.  The search adds
// 32-bit values and sizes; the exact evaluation adds four 16-bit limbs,
// because shared memory adds 32-bit words natively and 64-bit ones in a
// compare-and-swap loop.  Integer sums do not depend on the order of the
// additions.  `down` is what the light children read on the way down.
constexpr size_t kAccBytes = 8 + 16 + 8;
struct Down {                    // what a row passes to its light children: lin (units), lout
    int a;
    float b;
};
struct Acc {
    int4 *limb;
    int2 *s;                     // search: value, size
    Down *down;
};
__host__ __device__ inline Acc acc_at(char *base, size_t count)
{
    Acc a;
    a.limb = (int4 *)base;
    a.s = (int2 *)(base + count * 16);
    a.down = (Down *)(base + count * 24);
    return a;
}

// one item's scratch
struct Scratch1 {
    Scal *s;
    unsigned *hist;              // [2][kBins] profits per slot (weights), losses (rows)
    int64_t *prof, *f;           // [nslots]
    int *unit;                   // [nslots] profits in the search's units
    uint16_t *key;               // [nslots]
    int2 *tops;                  // [3][ntop] what the bins add to the last one: search (three prices in turn)
    int4 *topl;                  // [ntop] exact evaluation
    char *own;                   // accumulators of the bins when they are not in shared memory
};
__host__ __device__ inline size_t carve(char *base, int nslots, int ntop, bool acc_global, Scratch1 *o)
{
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *p = base + off;
        off += up16(bytes);
        return p;
    };
    Scratch1 x;
    x.s = (Scal *)take(sizeof(Scal));
    x.hist = (unsigned *)take(2 * kBins * 4);
    x.prof = (int64_t *)take((size_t)nslots * 8);
    x.f = (int64_t *)take((size_t)nslots * 8);
    x.unit = (int *)take((size_t)nslots * 4);
    x.key = (uint16_t *)take((size_t)nslots * 2);
    x.tops = (int2 *)take((size_t)ntop * 3 * 8);
    x.topl = (int4 *)take((size_t)ntop * 16);
    x.own = take(acc_global ? (size_t)(nslots + 32) * kAccBytes : 0);
    if (o) *o = x;
    return off;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ int cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}

// order-preserving code of a value >= 0, in [0, kBins): 32 codes per octave
__device__ __forceinline__ int code_of(int64_t v)
{
    if (v <= 0) return 0;
    return (int)(__float_as_uint(__ll2float_rd(v)) >> 18) - kKeyBase;
}
__device__ __forceinline__ float code_edge(int code) { return __uint_as_float((unsigned)(code + kKeyBase) << 18); }


__device__ __forceinline__ int64_t limbs(const int4 l)
{
    return (int64_t)((unsigned long long)(unsigned)l.x + ((unsigned long long)(unsigned)l.y << 16) +
                     ((unsigned long long)(unsigned)l.z << 32) + ((unsigned long long)(unsigned)l.w << 48));
}
__device__ __forceinline__ void limb_add(int4 *a, int64_t v)
{
    int *l = (int *)a;
    atomicAdd(l, (int)(v & 0xffff));
    atomicAdd(l + 1, (int)((v >> 16) & 0xffff));
    atomicAdd(l + 2, (int)((v >> 32) & 0xffff));
    atomicAdd(l + 3, (int)(v >> 48));
}
__device__ __forceinline__ void pair_add(int2 *a, int y, int z)
{
    atomicAdd((int *)a, y);
    atomicAdd((int *)a + 1, z);
}
// accumulators in global memory are added to in L2: read there
template <bool GLOBAL, typename T>
__device__ __forceinline__ T acc_ld(const T *p)
{
    if constexpr (GLOBAL) return __ldcg(p);
    else return *p;
}

// An entry of a warp's list of tiles: bits 0-15 the tile of the CTA's, 16-20
// its level, 21-25 its bin
__device__ __forceinline__ int tile_of(unsigned en) { return (int)(en & 0xffffu); }
__device__ __forceinline__ int level_of(unsigned en) { return (int)(en >> 16 & 31u); }
__device__ __forceinline__ int bin_of(unsigned en) { return (int)(en >> 21); }

// The tiles that a warp walks, its lanes' slots (info and a value) copied to
// shared memory two tiles ahead.  Asynchronous copies: registers loaded for
// the next trip of a loop are waited for at its back edge, which puts L2's
// latency (300 to 500 cycles) on every tile.
template <typename V, int DIR>
struct Feed {
    const int2 *info;                        // of this lane's slot of the bin's first tile
    const V *val;
    const unsigned *list;
    int2 *ri;                                // this lane's column of the ring
    V *rv;
    int n, i, h;                             // tiles, the one in hand, its ring slot

    __device__ __forceinline__ Feed(const int2 *info_, const V *val_, const unsigned *list_, int n_, unsigned char *ring)
        : info(info_ + (threadIdx.x & 31)), val(val_ + (threadIdx.x & 31)), list(list_), n(n_)
    {
        ri = (int2 *)(ring + (threadIdx.x >> 5) * (kRing * 512)) + (threadIdx.x & 31);
        rv = (V *)(ring + (threadIdx.x >> 5) * (kRing * 512) + kRing * 256) + (threadIdx.x & 31);
        i = DIR > 0 ? 0 : n - 1;
        h = 0;
        issue(i, 0);
        issue(i + DIR, 1);
    }
    __device__ __forceinline__ void issue(int x, int to)
    {
        if (x >= 0 && x < n) {
            const int slot = tile_of(list[x]) * 32;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(ri + to * 32)),
                         "l"(__cvta_generic_to_global(info + slot)) : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(rv + to * 32)),
                         "l"(__cvta_generic_to_global(val + slot)), "n"((int)sizeof(V)) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    __device__ __forceinline__ bool more() const { return DIR > 0 ? i < n : i >= 0; }
    __device__ __forceinline__ unsigned entry() const { return list[i]; }
    // the slots of the tile in hand; the one after next is started
    __device__ __forceinline__ void take(int2 &c, V &v)
    {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        c = ri[h * 32];
        v = rv[h * 32];
        issue(i + 2 * DIR, h == 0 ? 2 : h - 1);
        h = h == 2 ? 0 : h + 1;
        i += DIR;
    }
};

// ---- one tile of the search: f, and the size of the best closed set below
// (and with) every row, at a price of `lam` units; `out` the lanes with f <= 0
struct STile {
    int f, z;
    unsigned out;
};
__device__ __forceinline__ STile search_tile(int code, int p, int2 kids, int lam, int &carryY, int &carryZ)
{
    const int lane = threadIdx.x & 31;
    const int off = code & 31, w = code >> kWeightShift;
    const int d = min(p - min(lam * min(w, 4095), kClipRow) + kids.x, kClipRow);
    const bool cont = code & kCont;
    const int cy = cont ? carryY : 0;
    int ps = w + kids.y;
    // inclusive scan of x -> max(m, s + x) along the path
    int m = 0, sm = d;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int m2 = __shfl_up_sync(kAll, m, o), s2 = __shfl_up_sync(kAll, sm, o), p2 = __shfl_up_sync(kAll, ps, o);
        if (off >= o) {
            m = max(m, sm + m2);
            sm += s2;
        }
        if (lane >= o) ps += p2;
    }
    const int y = min(max(m, sm + cy), kClipPath);
    const int yp = __shfl_up_sync(kAll, y, 1);
    STile r;
    r.f = d + (off ? yp : cy);
    r.out = __ballot_sync(kAll, r.f <= 0);
    const unsigned neg = r.out & ((2u << lane) - (1u << (lane - off)));    // in this path, up to here
    const int at = neg ? 31 - __clz((int)neg) : lane - off - 1;
    const int pb = __shfl_sync(kAll, ps, at & 31);
    r.z = ps - (at >= 0 ? pb : 0) + (!neg && cont ? carryZ : 0);
    carryY = __shfl_sync(kAll, y, 31);
    carryZ = __shfl_sync(kAll, r.z, 31);
    return r;
}

// The search over a bin: levels from the leaves up, a block barrier between
// them.  A tile without a row of positive f has none at any higher price:
// `keep` gets the others, the list to walk if this price turns out to be a
// lower bound; their number is returned.  own.s[na] stays zero (rows without
// light children read it).
template <bool GLOBAL>
__device__ __forceinline__ int search_bin(const int2 *info, const int *val, const unsigned *list, int n, unsigned *keep,
                                          int nlev, const Acc &own, const int *base, int na, int2 *tops, int lam, int clip,
                                          unsigned char *ring, int &rootZ)
{
    const int lane = threadIdx.x & 31;
    Feed<int, 1> feed(info, val, list, n, ring);
    int lev = 0, carryY = 0, carryZ = 0, kept = 0;
    unsigned prev = 0;
    while (feed.more()) {
        const unsigned en = feed.entry();
        for (; lev < level_of(en); ++lev) __syncthreads();
        int2 c;
        int p;
        feed.take(c, p);
        const int ac = c.y & 0xffff, up = (unsigned)c.y >> 16;
        const int a0 = base[bin_of(en)];
        const int2 kids = acc_ld<GLOBAL>(own.s + min(a0 + ac, na));
        if (en != prev + 1) carryY = carryZ = 0;         // not the same path's next tile
        prev = en;
        const STile r = search_tile(c.x, p, kids, lam, carryY, carryZ);
        if (r.out != kAll) {
            if (lane == 0) keep[kept] = en;
            ++kept;
        }
        if ((c.x & kTop) && r.f > 0) {
            if (up == kNone) rootZ += r.z;
            else if (c.x & kUp) pair_add(tops + up, min(r.f, clip), r.z);
            else pair_add(own.s + a0 + up, min(r.f, clip), r.z);
        }
    }
    for (++lev; lev < nlev; ++lev) __syncthreads();
    return kept;
}

// The last bin, by one warp (every CTA does it for itself): its tiles in
// order; `loc`: what the bins have added, then its own paths.  The slots come
// from shared memory if there are at most kTopSlots (two trips to L2 less a
// price).
constexpr int kTopSlots = 256;
__device__ __forceinline__ int search_top(const Tab &t, const Scratch1 &g, const int4 *slots, const int2 *tops, int2 *loc,
                                          int lam, int clip)
{
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < t.ntop; i += 32) loc[i] = __ldcg(tops + i);
    __syncwarp();
    int rootZ = 0, carryY = 0, carryZ = 0;
    const int s0 = t.binslot[t.bins], ns = t.nslots - s0;
    for (int s = lane; s < ns; s += 32) {
        int4 c;
        if (ns <= kTopSlots) {
            c = slots[s];
        } else {
            const int2 i = __ldg(t.info + s0 + s);
            c = make_int4(i.x, i.y, __ldcg(g.unit + s0 + s), 0);
        }
        const int ac = c.y & 0xffff, up = (unsigned)c.y >> 16;
        const int2 kids = ac != kNone ? loc[ac] : make_int2(0, 0);
        const STile r = search_tile(c.x, c.z, kids, lam, carryY, carryZ);
        if ((c.x & kTop) && r.f > 0) {
            if (up == kNone) rootZ += r.z;
            else pair_add(loc + up, min(r.f, clip), r.z);
        }
        __syncwarp();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rootZ += __shfl_xor_sync(kAll, rootZ, o);
    return rootZ;
}

// ---- one tile of the exact evaluation at the price lam
__device__ __forceinline__ int64_t exact_tile(int code, int64_t p, int64_t kids, int64_t lam, int64_t &carryY)
{
    const int off = code & 31;
    const bool cont = code & kCont;
    const int64_t d = p - lam * (code >> kWeightShift) + kids;
    int64_t m = 0, sm = d;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t m2 = __shfl_up_sync(kAll, m, o), s2 = __shfl_up_sync(kAll, sm, o);
        if (off >= o) {
            const int64_t v = sm + m2;
            m = m > v ? m : v;
            sm += s2;
        }
    }
    const int64_t v = sm + (cont ? carryY : 0);
    const int64_t y = m > v ? m : v;
    int64_t yp = __shfl_up_sync(kAll, y, 1);
    if (off == 0) yp = cont ? carryY : 0;
    carryY = __shfl_sync(kAll, y, 31);
    return d + yp;
}

// f of every row of a bin to f, the roots' share of L to rootY
template <bool GLOBAL>
__device__ __forceinline__ void exact_bin(const int2 *info, const int64_t *val, int64_t *fout, int4 *topl,
                                          const unsigned *list, int n, int nlev, const Acc &own, const int *base, int na, int64_t lam,
                                          unsigned char *ring, int64_t &rootY)
{
    const int lane = threadIdx.x & 31;
    Feed<int64_t, 1> feed(info, val, list, n, ring);
    int lev = 0;
    int64_t carryY = 0;
    unsigned prev = 0;
    while (feed.more()) {
        const unsigned en = feed.entry();
        for (; lev < level_of(en); ++lev) __syncthreads();
        int2 c;
        int64_t p;
        feed.take(c, p);
        const int ac = c.y & 0xffff, up = (unsigned)c.y >> 16;
        const int a0 = base[bin_of(en)];
        const int64_t kids = limbs(acc_ld<GLOBAL>(own.limb + min(a0 + ac, na)));
        if (en != prev + 1) carryY = 0;
        prev = en;
        const int64_t f = exact_tile(c.x, p, kids, lam, carryY);
        fout[tile_of(en) * 32 + lane] = f;
        if ((c.x & kTop) && f > 0) {
            if (up == kNone) rootY += f;
            else if (c.x & kUp) limb_add(topl + up, f);
            else limb_add(own.limb + a0 + up, f);
        }
    }
    for (++lev; lev < nlev; ++lev) __syncthreads();
}
// the last bin, by one warp of every CTA (they write the same f)
__device__ __forceinline__ int64_t exact_top(const Tab &t, const Scratch1 &g, int4 *loc, int64_t lam)
{
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < t.ntop; i += 32) loc[i] = __ldcg(g.topl + i);
    __syncwarp();
    int64_t rootY = 0, carryY = 0;
    for (int s = t.binslot[t.bins] + lane; s < t.nslots; s += 32) {
        const int2 c = __ldg(t.info + s);
        const int ac = c.y & 0xffff, up = (unsigned)c.y >> 16;
        const int64_t kids = ac != kNone ? limbs(loc[ac]) : 0;
        const int64_t f = exact_tile(c.x, __ldcg(g.prof + s), kids, lam, carryY);
        g.f[s] = f;
        if ((c.x & kTop) && f > 0) {
            if (up == kNone) rootY += f;
            else limb_add(loc + up, f);
        }
        __syncwarp();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rootY += __shfl_xor_sync(kAll, rootY, o);
    return rootY;
}

// ---- one tile of the losses, from the top of a path down: `a` the sum of
// max(0, -f) over the path from the root, `b` the smallest f on it.  Sums in
// units of 2^shift, each row's share rounded down to them and no more than
// kLossCap: a loss is only ever underestimated, which keeps rows.  Below a row
// that is decided out every row has to be, so no row's sum may lie below its
// parent's: whole numbers add up to the same in any order (sums of floats did
// not, and a row stayed undecided under a parent that was out; with a running
// maximum over them, five more shuffles a tile, the paper-scale plan took 27.73
// ms, with whole numbers 27.53).
constexpr int kLossCap = 1 << 30;
constexpr int kLossBits = 20;                // of a price times a mean weight: 0.1 of it, the first threshold, is 2^17
__device__ __forceinline__ void loss_tile(int code, int64_t f, int shift, bool child, Down up, int &ca, float &cb, int &a,
                                          float &b)
{
    const int lane = threadIdx.x & 31;
    const unsigned starts = __ballot_sync(kAll, (code & 31) == 0);
    const unsigned tops = __ballot_sync(kAll, (code & kTop) != 0);
    const unsigned after = lane < 31 ? starts >> (lane + 1) : 0u;
    const int rem = after ? __ffs((int)after) - 1 : 31 - lane;    // lanes to the right in this path
    b = __ll2float_rd(f);
    const unsigned long long loss = f < 0 ? (unsigned long long)-f >> shift : 0;
    a = loss < kLossCap ? (int)loss : kLossCap;
    if (child) {                             // a path's top below some row: `up` is that row's
        a = min(a + up.a, kLossCap);
        b = fminf(b, up.b);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a2 = __shfl_down_sync(kAll, a, o);
        const float b2 = __shfl_down_sync(kAll, b, o);
        if (rem >= o) {
            a = min(a + a2, kLossCap);
            b = fminf(b, b2);
        }
    }
    if (!((tops >> (lane + rem)) & 1u)) {       // the path goes on in the next tile
        a = min(a + ca, kLossCap);
        b = fminf(b, cb);
    }
    ca = __shfl_sync(kAll, a, 0);
    cb = __shfl_sync(kAll, b, 0);
}
// key of a row (15 bits) and whether it is in S (bit 15)
__device__ __forceinline__ int loss_code(int a, float b, int shift)
{
    const bool in = b > 0.f;
    const float v = in ? b : __int2float_rd(a);
    const int k = v < 1.f ? 0 : min((int)(__float_as_uint(v) >> 18) - kKeyBase + (in ? 0 : 32 * shift), kBins - 1);
    return k | (in ? 0x8000 : 0);
}

// losses of one bin, levels from the top down, and their histogram
template <bool GLOBAL>
__device__ __forceinline__ void loss_bin(const int2 *info, const int64_t *fin, uint16_t *key, const unsigned *list, int n,
                                         int nlev, const Acc &own, const int *base, const Down *topd, int shift,
                                         unsigned char *ring, unsigned *hist)
{
    const int lane = threadIdx.x & 31;
    Feed<int64_t, -1> feed(info, fin, list, n, ring);
    int lev = nlev - 1;
    int ca = 0;
    float cb = 0.f;
    while (feed.more()) {
        const unsigned en = feed.entry();
        for (; lev > level_of(en); --lev) __syncthreads();
        int2 c;
        int64_t f;
        feed.take(c, f);
        const int ac = c.y & 0xffff, up = (unsigned)c.y >> 16;
        const bool child = (c.x & kTop) && up != kNone;
        const int a0 = base[bin_of(en)];
        Down from = {0, 0.f};
        if (child) {
            if (c.x & kUp) from = topd[up];
            else {
                const int2 d = acc_ld<GLOBAL>((const int2 *)(own.down + a0 + up));
                from = {d.x, __int_as_float(d.y)};
            }
        }
        int a;                               // (a path that goes on does so in the tile just done)
        float b;
        loss_tile(c.x, f, shift, child, from, ca, cb, a, b);
        if (ac != kNone) own.down[a0 + ac] = {a, b};
        const int code = (c.x >> kWeightShift) ? loss_code(a, b, shift) : kKeyPad;      // (a pad weighs nothing)
        if (code != kKeyPad) atomicAdd(hist + (code & 0x7fff), 1u);
        key[tile_of(en) * 32 + lane] = (uint16_t)code;
    }
    for (; lev > 0; --lev) __syncthreads();
}
// the last bin, by one warp; one CTA (`write`) keeps its keys
__device__ __forceinline__ void loss_top(const Tab &t, const Scratch1 &g, Down *topd, int shift, unsigned *hist, bool write)
{
    const int lane = threadIdx.x & 31;
    int ca = 0;
    float cb = 0.f;
    for (int s = t.nslots - 32 + lane; s >= t.binslot[t.bins]; s -= 32) {
        const int2 c = __ldg(t.info + s);
        const int ac = c.y & 0xffff, up = (unsigned)c.y >> 16;
        const bool child = (c.x & kTop) && up != kNone;
        int a;
        float b;
        loss_tile(c.x, g.f[s], shift, child, child ? topd[up] : Down{0, 0.f}, ca, cb, a, b);
        if (ac != kNone) topd[ac] = {a, b};
        if (write) {
            const int code = (c.x >> kWeightShift) ? loss_code(a, b, shift) : kKeyPad;
            if (code != kKeyPad) atomicAdd(hist + (code & 0x7fff), 1u);
            g.key[s] = (uint16_t)code;
        }
        __syncwarp();
    }
}

// exclusive scan over the block (one value per thread) and its total
__device__ int block_scan(int v, int *total, int *sh)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kAll, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    int w = lane < kWarps ? sh[lane] : 0;    // every warp scans the warps' totals
    const int mine = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kAll, w, o);
        if (lane >= o) w += y;
    }
    *total = __shfl_sync(kAll, w, 31);
    const int before = __shfl_sync(kAll, w - mine, wid);
    __syncthreads();
    return before + x - v;
}

// ---------------------------------------------------------------------------
// The price.  |S| falls with the price; the one wanted is where it passes k.
// Its first guess is the k-th largest profit per slot (chunks taken without
// their prefixes: within ~15% on the prefix trees here), the second scales
// that curve through the first point, then the bracket is closed by
// interpolating logarithms (|S| falls like a power).  3 to 7 prices; a search
// from price 0 by the tangents of L took 9 to 10.
// ---------------------------------------------------------------------------
enum : int { kGo = 0, kStop = 1, kSlack = 2, kCoarser = 3, kTooDear = 4 };
constexpr int kCoarserBits = 6;

struct Search {                              // prices in units
    float x0, x1, z0, z1;                    // price and |S| of the ends with |S| > k and <= k
    int have, side;                          // bit 0, 1: that end is there; steps in a row to one side
    int max_evals;                           // prices that may be tried
    float left;                              // us that may still be spent before the item is left to the sweep
};

// weight of the rows worth at least lam per slot, and its inverse (cum[c]:
// weight of the codes >= c)
__device__ float rank_at(const int *cum, float lam)
{
    const int c = lam < 1.f ? 0 : min((int)(__float_as_uint(lam) >> 18) - kKeyBase, kBins - 1);
    const float lo = code_edge(c), hi = code_edge(c + 1);
    const int n0 = cum[c], n1 = c + 1 < kBins ? cum[c + 1] : 0;
    return n0 - (n0 - n1) * ((lam - lo) / (hi - lo));
}
__device__ float price_of_rank(const int *cum, float rank)
{
    int a = 1, b = kBins;                    // the last code with cum >= rank
    while (b - a > 1) {
        const int m = (a + b) >> 1;
        if (cum[m] >= rank) a = m;
        else b = m;
    }
    const float lo = code_edge(a), hi = code_edge(a + 1);
    const int n0 = cum[a], n1 = a + 1 < kBins ? cum[a + 1] : 0;
    float fr = n0 > n1 ? (n0 - rank) / (n0 - n1) : 0.f;
    fr = fminf(fmaxf(fr, 0.f), 1.f);
    return lo + (hi - lo) * fr;
}

// what to do after the price `lam` (units of 2^shift) gave |S| = Z: try `nx`
// (kGo), stop and use `nx` (kStop), the budget does not bind (kSlack), or go on
// in units of 2^(shift + kCoarserBits) with `nx` of them (kCoarser): where few
// chunks have a profit whole paths are taken for one, and the price may be far
// above the k-th largest profit per slot, which the units were chosen by
__device__ int next_price(Search &b, const int *cum, float k, int maxlam, float unit, int evals, int lam, float Z, int &nx)
{
    if (Z > k) {
        b.x0 = (float)lam;
        b.z0 = Z;
        b.side = b.side > 0 ? b.side + 1 : 1;
        b.have |= 1;
    } else {
        if (lam == 0) return kSlack;
        b.x1 = (float)lam;
        b.z1 = Z;
        b.side = b.side < 0 ? b.side - 1 : -1;
        b.have |= 2;
    }
    if ((Z - k) * (Z - k) <= 0.05f * k) {    // |S| is so near k that L is flat
        nx = lam;
        return kStop;
    }
    if (lam == kClipPrice && Z > k && evals < b.max_evals) {
        b.x0 *= 1.f / (1 << kCoarserBits);
        nx = lam >> (kCoarserBits - 3);
        return kCoarser;
    }
    float x;
    if (b.have == 3) {
        // L's slope is k - |S|, so these bound what a better price could still give
        const float d = b.x1 - b.x0, e0 = (b.z0 - k) * d, e1 = (k - b.z1) * d;
        if (fminf(e0, e1) <= 0.1f * b.x0 || d <= 1.f || evals >= b.max_evals) {
            nx = (int)(e0 < e1 ? b.x0 : b.x1);
            return kStop;
        }
        if (b.x0 > 0.f) {
            float s = __log2f(b.z0 / k) / __log2f(b.z0 / fmaxf(b.z1, 1.f));
            s = fminf(fmaxf(s, 0.15f), 0.85f);
            if (b.side >= 2 || b.side <= -2) s = 0.5f * s + 0.25f;      // creeping from one side
            if (evals > 5) s = fminf(fmaxf(s, 0.2f), 0.8f);
            x = b.x0 * exp2f(__log2f(b.x1 / b.x0) * s);
        } else {
            x = 0.5f * b.x1;
        }
        x = fminf(fmaxf(x, b.x0 + 1.f), b.x1 - 1.f);
    } else {
        if (evals >= b.max_evals) {
            nx = lam;
            return kStop;
        }
        const bool above = Z > k;            // the price has to rise
        const float l1 = fmaxf((float)lam, 1.f), c = rank_at(cum, l1 * unit);
        if (Z > 0.f && c > 0.f && evals < 6) {
            x = price_of_rank(cum, k * c / Z) / unit;
            const float step = evals == 1 ? 0.015f : evals == 2 ? 0.04f : evals == 3 ? 0.1f : 0.3f;
            x = above ? fmaxf(x, l1) * (1.f + step) : fminf(x, l1) * (1.f - step);
        } else if (!above && evals < 5) {
            // nothing is worth that much, a little less (close profits) or much
            // less (for what lies above it)
            x = l1 * (evals == 1 ? 0.96f : evals == 2 ? 0.5f : 0.25f);
        } else {
            x = above ? (float)maxlam : 0.f;
        }
        x = above ? fmaxf(x, b.x0 + 1.f) : fminf(x, b.x1 - 1.f);
    }
    nx = min(max((int)x, 0), maxlam);
    return kGo;
}

// ---------------------------------------------------------------------------
// Eq. 9 over the undecided rows, in shared memory
// ---------------------------------------------------------------------------
struct __align__(16) Row {
    int64_t p;
    int w, info;                             // flags below, stack level << 8
};
struct Rows {                                // in sweep order (last position first)
    Row row[kRowCap + 8];                    // (read up to eight at a time)
    int2 step[kRowCap];                      // the walk's: weight, row that a skip goes to (-1 past the last)
    int pos[kRowCap], last[kRowCap + 8];
    unsigned leaf[kRowCap / 32];             // bit: a skip goes to the next row
};
constexpr int kPush = 1, kReload = 2, kZeroTop = 4, kFromCur = 8;

// One column per thread (column j = 1 + thread), as many warps as that takes.
// The row just computed goes through shared memory (any weight is then one
// load at j - w; `guard` words left of column 0 read as never worth taking),
// a barrier of these warps per row; the scalars of four rows are read at once
// and decision bits packed per thread over 32 rows.  Several columns per
// thread of one warp took 100 (2 columns) to 310 ns (8) a row: a single warp
// issues every instruction of a row in turn.
__device__ __forceinline__ void dp_rows(const Rows &R, int T, int act, int guard, int64_t *rowb, int64_t *stk,
                                        uint32_t *bits, int64_t *result, int kc)
{
    const int tid = threadIdx.x, cols = act * 32, pitch = cols + 1 + guard;
    int64_t cur = 0, top = 0;
    uint32_t wb = 0;
    int64_t *const b0 = rowb + guard + 1 + tid, *const b1 = b0 + pitch;     // this column in the two row buffers
    for (int r0 = 0; r0 < T; r0 += 4) {
        Row x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = R.row[r0 + u];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (r0 + u >= T) break;
            const int64_t *prev = u & 1 ? b1 : b0;
            int64_t *out = u & 1 ? b0 : b1;
            const int64_t tv = x[u].p + prev[-x[u].w];
            const int64_t sk = (x[u].info & kFromCur) ? cur : top;
            const bool take = tv > sk;
            cur = take ? tv : sk;
            *out = cur;
            if (take) wb |= 1u << ((r0 + u) & 31);
            if (x[u].info & (kPush | kReload | kZeroTop)) {
                int64_t *sl = stk + (x[u].info >> 8) * cols + tid;
                if (x[u].info & kPush) *sl = top = cur;
                else top = (x[u].info & kReload) ? *sl : 0;
            }
            if (act == 1) __syncwarp();
            else asm volatile("bar.sync 1, %0;" ::"r"(cols) : "memory");
        }
        if ((r0 & 31) == 28 || r0 + 4 >= T) {
            bits[(r0 >> 5) * cols + tid] = wb;
            wb = 0;
        }
    }
    if (kc == 1 + tid) *result = cur;
}

// Unit weights and at most 128 columns: one warp, C columns per lane (column
// j = 1 + lane * C + c) in registers, the column shift a shuffle, no barrier:
// 38 to 80 ns a row (C and stack rows) against 98 with a barrier per row.  Instead of decision
// bits it keeps, per row and column, the first row taken from there on, plus
// 1 (0: none; following skips changes nothing), so the walk takes one step per
// chunk.
constexpr int kUnitCols = 128;
template <int C>
__device__ __forceinline__ void dp_unit(const Rows &R, int T, int64_t *stk, uint16_t *stf, uint16_t *first,
                                        int64_t *result, int kc)
{
    constexpr int cols = 32 * C;
    const int lane = threadIdx.x & 31;
    int64_t cur[C], top[C];
    int fc[C], ft[C];                        // first row taken from the row just computed, from the top
#pragma unroll
    for (int c = 0; c < C; ++c) {
        cur[c] = top[c] = 0;
        fc[c] = ft[c] = 0;
    }
    constexpr int U = 4;                     // rows unrolled (no-op rows past the last)
    constexpr int kOps = kPush | kReload | kZeroTop;
    for (int r0 = 0; r0 < T; r0 += U) {
        Row x[U];
        int ops = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            x[u] = R.row[r0 + u];
            ops |= x[u].info;
        }
        auto row = [&](const int u, const bool stack) {
            int64_t up = __shfl_up_sync(kAll, cur[C - 1], 1);
            up = lane ? up : 0;
            const bool same = x[u].info & kFromCur;
#pragma unroll
            for (int c = C - 1; c >= 0; --c) {
                const int64_t sk = same ? cur[c] : top[c];
                const int64_t tv = x[u].p + (c ? cur[c > 0 ? c - 1 : 0] : up);
                const bool take = tv > sk;
                cur[c] = take ? tv : sk;
                fc[c] = take ? r0 + u + 1 : same ? fc[c] : ft[c];
            }
            uint16_t *fo = first + (r0 + u) * cols + lane * C;
            if (C == 4) *(uint2 *)fo = make_uint2(fc[0] | fc[C > 1 ? 1 : 0] << 16, fc[C > 2 ? 2 : 0] | fc[C > 3 ? 3 : 0] << 16);
            else if (C == 2) *(unsigned *)fo = fc[0] | fc[C > 1 ? 1 : 0] << 16;
            else *fo = (uint16_t)fc[0];
            if (stack && (x[u].info & kOps)) {
                const int at = (x[u].info >> 8) * cols + lane;       // (a lane's own cells: no exchange)
                if (x[u].info & kPush) {
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        stk[at + 32 * c] = top[c] = cur[c];
                        stf[at + 32 * c] = (uint16_t)(ft[c] = fc[c]);
                    }
                } else {
                    const bool re = x[u].info & kReload;
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        top[c] = re ? stk[at + 32 * c] : 0;
                        ft[c] = re ? stf[at + 32 * c] : 0;
                    }
                }
            }
        };
        if ((ops & kOps) == 0) {
#pragma unroll
            for (int u = 0; u < U; ++u) row(u, false);
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) row(u, true);
        }
    }
#pragma unroll
    for (int c = 0; c < C; ++c)
        if (kc == 1 + lane * C + c) *result = cur[c];
}

// the rows of an item that stays unsolved (not inlined: its registers are not
// the reduction's)
__device__ __noinline__ void prune_left(const Args &A, int item, const uint32_t *ud)
{
    prune_item(A.t.n, item, A.profit, A.order, A.next, A.pspan, A.wpre, A.w, ud, 1, A.stack_depth, A.status, A.rows_kept);
}

}  // namespace

template <bool SMEM>                         // accumulators of the bins in shared memory
__global__ void __launch_bounds__(kThreads) k_reduce(const __grid_constant__ Args A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned char leaf[kWarps * kMaxTiles];   // tiles of level 0: see the gather
    __shared__ unsigned lists[3][kWarps][kMaxTiles];    // a warp's tiles: all; two that the search shortens in turn
    __shared__ int4 s_top[kMaxTop];          // the last bin's own sums, then what it passes down
    __shared__ int4 slots[kTopSlots];        // of the last bin: info, profit in units
    __shared__ int sh[kWarps];
    __shared__ int base[kMaxBins + 1];       // of a bin's accumulators among the CTA's
    __shared__ int s_a, s_b, s_flag, s_lam;
    __shared__ Search s_search;
    __shared__ int64_t s_val;
    const Tab &t = A.t;
    const int CL = t.CL, cr = CL > 1 ? cluster_rank() : 0;
    const int item = blockIdx.x / CL;
    chain_wait();
    if (A.w.clear && cr == 0 && threadIdx.x == 0) A.w.clear[item] = 0;
    const int n = t.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t *red = A.w.red + item;
    if (A.item_active && !A.item_active[item]) return;      // uniform over the cluster
    const int32_t kreq = A.item_budget[item];
    if (kreq < 0 || kreq > A.max_budget) {                  // the DP's kernel reports it
        if (cr == 0 && tid == 0) *red = 0;
        prune_left(A, item, nullptr);
        return;
    }
    const int64_t k = kreq < A.total_weight ? kreq : A.total_weight;     // more changes nothing
    if (A.spending.evals[k > 128] == 0 && k > 0) {           // (the same in every CTA)
        if (cr == 0 && tid == 0) *red = 0;
        prune_left(A, item, nullptr);
        return;
    }
    Scratch1 g;
    carve(A.w.red_scratch + (size_t)item * A.item_bytes, t.nslots, t.ntop, !SMEM, &g);
    const int words = (n + 31) / 32;
    uint32_t *taken = A.w.taken + (size_t)item * words, *freeb = A.w.undecided + (size_t)item * words;
    const int64_t *P = A.profit + (size_t)item * n;
    for (int i = cr * kThreads + tid; i < words; i += CL * kThreads) taken[i] = freeb[i] = 0;
    if (k == 0) {                            // nothing fits
        if (cr == 0 && tid == 0) {
            A.best[item] = 0;
            A.w.nkept[item] = 0;
            *red = 1;
        }
        return;
    }
    const int per = t.bins / CL, bin0 = cr * per;            // this CTA's bins
    const int lo = t.binslot[bin0], hi = t.binslot[bin0 + per];
    if (tid < 32) {
        const int mine = lane < per ? __ldg(t.nacc + bin0 + lane) : 0;
        int x = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kAll, x, o);
            if (lane >= o) x += y;
        }
        if (lane <= per) base[lane] = x - mine;
    }
    __syncthreads();
    const int na = base[per];
    const Acc own = acc_at(SMEM ? (char *)smem : g.own + (size_t)(lo + cr) * kAccBytes, na + 1);   // (one reads as zero)
    unsigned char *ring = smem + (SMEM ? up16((size_t)(na + 1) * kAccBytes) : 0);
    unsigned *hist = (unsigned *)(ring + kRingBytes);
    const int top0 = t.binslot[t.bins];
    const bool has_top = top0 < t.nslots;
    const int2 *info = t.info + lo;
    auto sync_all = [&] {
        if (CL > 1) cluster_sync();
        else __syncthreads();
    };

    // ---- clear what is added to; this bin's streams
    if (cr == 0) {
        for (int i = tid; i < (int)(sizeof(Scal) / 8); i += kThreads) ((unsigned long long *)g.s)[i] = 0;
        for (int i = tid; i < 2 * kBins; i += kThreads) g.hist[i] = 0;
        for (int i = tid; i < 3 * t.ntop; i += kThreads) g.tops[i] = make_int2(0, 0);
        for (int i = tid; i < t.ntop; i += kThreads) g.topl[i] = make_int4(0, 0, 0, 0);
    }
    for (int i = tid; i < kBins; i += kThreads) hist[i] = 0;
    // this warp's tiles: of every level the bins' streams go round the warps
    int tiles = 0, nlev = 0;
    {
        const int e0 = __ldg(t.binlev + bin0), e1 = __ldg(t.binlev + bin0 + per);
        const int q0 = __ldg(t.lev + e0);
        // (at most kMaxBins (kMaxLevels + 1) entries, then at most kWarps kMaxTiles streams)
        int *lev = (int *)ring;
        int2 *stream = (int2 *)(ring + kMaxBins * (kMaxLevels + 1) * 4);
        const int ns = __ldg(t.lev + e1 - 1) - q0;
        for (int i = tid; i < e1 - e0; i += kThreads) lev[i] = __ldg(t.lev + e0 + i) - q0;
        for (int i = tid; i < ns; i += kThreads) stream[i] = __ldg(t.stream + q0 + i);
        const int from = lane < per ? __ldg(t.binlev + bin0 + lane) - e0 : 0;       // a lane per bin
        const int levels = lane < per ? __ldg(t.binlev + bin0 + lane + 1) - 1 - e0 - from : 0;
        nlev = __reduce_max_sync(kAll, levels);
        __syncthreads();
        for (int l = 0, at = 0; l < nlev; ++l) {
            int first = 0, c = 0;
            if (l < levels) {
                first = lev[from + l];
                c = lev[from + l + 1] - first;
            }
            int x = c;
#pragma unroll
            for (int o = 1; o < kMaxBins; o <<= 1) {
                const int y = __shfl_up_sync(kAll, x, o);
                if (lane >= o) x += y;
            }
            const int j = (warp - at - (x - c)) & (kWarps - 1);     // which of the bin's streams is this warp's
            for (unsigned m = __ballot_sync(kAll, j < c); m; m &= m - 1) {
                const int bb = __ffs((int)m) - 1;
                const int2 st = stream[__shfl_sync(kAll, first + j, bb)];
                for (int i = lane; i < st.y; i += 32)
                    lists[0][warp][tiles + i] = (unsigned)bb << 21 | (unsigned)l << 16 | (unsigned)(st.x - (lo >> 5) + i);
                tiles += st.y;
            }
            at += __shfl_sync(kAll, x, kMaxBins - 1);
        }
    }
    for (int i = tid; i < (hi - lo) >> 5; i += kThreads) leaf[i] = 0;
    sync_all();

    // ---- gather the profits into the slots; weights by profit per slot
    // (from every tile up to 16,384 slots, then from a sample of the tiles)
    int64_t mx = 0;
    const int every = t.nslots > 16384 ? 31 - __clz(t.nslots >> 13) : 0;
    auto gather = [&](int from, int to) {
        constexpr int U = 4;                 // loads in flight per thread
        for (int s0 = from + tid; s0 < to; s0 += U * kThreads) {
            int x[U], form[U];
            int64_t p[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int s = s0 + u * kThreads;
                x[u] = s < to ? __ldg(t.pos + s) : -1;
                form[u] = s < min(to, hi) ? __ldg(t.form + (s >> 5)) : 0;      // (the last bin's tiles are in no list)
            }
            if (A.order)
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (x[u] >= 0) x[u] = __ldg(A.order + x[u]);
#pragma unroll
            for (int u = 0; u < U; ++u) p[u] = x[u] >= 0 ? P[x[u]] : 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int s = s0 + u * kThreads;
                if (s >= to) break;
                g.prof[s] = p[u];
                mx = p[u] > mx ? p[u] : mx;
                // a warp's slots are a tile; its form if there is no profit in it
                if (!__any_sync(kAll, p[u] > 0) && form[u] && lane == 0) leaf[(s - lo) >> 5] = (unsigned char)form[u];
                if (p[u] > 0 && ((s >> 5) & ((1 << every) - 1)) == 0) {
                    const int w = __ldg(&t.info[s].x) >> kWeightShift;
                    const int c = w == 1 ? code_of(p[u]) : code_of((int64_t)((float)p[u] / (float)w));
                    atomicAdd(hist + c, (unsigned)w << every);
                }
            }
        }
    };
    gather(lo, hi);
    if (cr == 0 && has_top) gather(top0, t.nslots);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int64_t y = __shfl_xor_sync(kAll, mx, o);
        mx = y > mx ? y : mx;
    }
    if (lane == 0 && mx > 0) atomicMax(&g.s->maxp, (unsigned long long)mx);
    __syncthreads();
    for (int i = tid; i < kBins; i += kThreads)
        if (hist[i]) atomicAdd(g.hist + i, hist[i]);
    sync_all();
    const int64_t maxp = (int64_t)__ldcg(&g.s->maxp);
    {
        // leaf tiles without a profit leave the lists: at any price nothing in
        // them is taken (on the planner's later sweeps, most of the tree)
        int kept = 0;
        int prev = -2;
        bool pd = false;
        for (int i = 0; i < tiles; ++i) {
            const unsigned en = lists[0][warp][i];
            const int q = tile_of(en), fl = leaf[q];
            const bool d = (fl & 1) && (!(fl & 2) || (pd && q == prev + 1));
            __syncwarp();
            if (d) g.key[lo + q * 32 + lane] = kKeyPad;
            else if (lane == 0) lists[0][warp][kept] = lists[1][warp][kept] = en;
            kept += !d;
            pd = d;
            prev = q;
        }
        tiles = kept;
    }
    int *cum = (int *)hist;                  // weight of the codes >= c
    {
        constexpr int V = kBins / kThreads;
        int c[V], sum = 0;
#pragma unroll
        for (int v = V - 1; v >= 0; --v) {
            c[v] = sum;                      // of the codes above, in this thread's run
            sum += (int)__ldcg(g.hist + tid * V + v);
        }
        int tot;
        const int before = block_scan(sum, &tot, sh);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int mine = (int)__ldcg(g.hist + tid * V + v);
            cum[tid * V + v] = tot - before - sum + c[v] + mine;
        }
        __syncthreads();
    }

    // ---- the price
    // lambda k, and lambda times the weight of a tile's 32 rows (what a scan sums
    // before it takes the maximum), have to stay within int64 (a product: the
    // division, with one of the mean weight further on, was 0.8 us an item)
    const unsigned long long slots_most = k > 32 * A.max_weight ? k : 32 * A.max_weight, top_profit = maxp;
    const bool too_large = __umul64hi(top_profit, slots_most) != 0 || top_profit * slots_most > (unsigned long long)kBig;
    int64_t lam = 0, L = 0;
    if (!too_large) {
        const float guess = cum[0] <= k ? 0.f : fminf(fmaxf(price_of_rank(cum, (float)k), 1.f), (float)maxp);
        int shift = max(0, (int)(__float_as_uint(fmaxf(guess, 1.f)) >> 23) - 127 - kUnitBits);
        int price = (int)(guess * exp2f((float)-shift));
        if (tid == 0) {                      // (shared; the search's thread)
            s_search = Search();
            s_search.max_evals = A.spending.evals[k > 128];
            s_search.left = A.spending.sweep[k > 128];
        }
        auto to_units = [&](int from, int to) {
            for (int s = from + tid; s < to; s += kThreads) {
                const int64_t p = g.prof[s] >> shift;
                g.unit[s] = (int)(p > kClipRow ? kClipRow : p < -kClipRow ? -kClipRow : p);
            }
        };
        bool low = false;                    // the last price was a lower bound
        int at = 1, alive = tiles, kept = 0;
        int ev = 0;
        for (;;) {
            const int maxlam = (int)min((maxp >> shift) + 1, (int64_t)kClipPrice);
            to_units(lo, hi);
            if (has_top && t.nslots - top0 > kTopSlots) {
                if (cr == 0) to_units(top0, t.nslots);
            } else if (tid < t.nslots - top0) {
                const int64_t p = __ldcg(g.prof + top0 + tid) >> shift;
                const int2 i = __ldg(t.info + top0 + tid);
                slots[tid] = make_int4(i.x, i.y, (int)(p > kClipRow ? kClipRow : p < -kClipRow ? -kClipRow : p), 0);
            }
            for (;; ++ev) {
                for (int i = tid; i <= na; i += kThreads) own.s[i] = make_int2(0, 0);
                // (the set that the last price but one's sums were read from)
                if (low) {                       // fewer tiles to walk from now on
                    at ^= 3;
                    alive = kept;
                }
                if (cr == 0)
                    for (int i = tid; i < t.ntop; i += kThreads) g.tops[(ev + 1) % 3 * t.ntop + i] = make_int2(0, 0);
                int2 *tops = g.tops + ev % 3 * t.ntop;
                int rz = 0;
                __syncthreads();
                kept = search_bin<!SMEM>(info, g.unit + lo, lists[at][warp], alive, lists[at ^ 3][warp], nlev, own, base, na, tops,
                                         price, A.clip_kid, ring, rz);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) rz += __shfl_xor_sync(kAll, rz, o);
                if (lane == 0 && rz) atomicAdd(&g.s->sumZ[ev], (unsigned long long)rz);
                sync_all();
                if (warp == 0) {
                    const int bins = lane == 0 ? (int)__ldcg(&g.s->sumZ[ev]) : 0;
                    int z = has_top ? search_top(t, g, slots, tops, (int2 *)s_top, price, A.clip_kid) : 0;
                    if (lane == 0) {
                        z += bins;
                        int nx = price;
                        s_flag = next_price(s_search, cum, (float)k, maxlam, exp2f((float)shift), ev + 1, price, (float)z, nx);
                        if (s_flag == kStop || s_flag == kSlack) {
                            // (the exact evaluation and the losses take two prices)
                            s_search.left -= (float)(ev + 3) * A.spending.price;
                            if (s_search.left < kPassUs) s_flag = kTooDear;
                        }
                        s_lam = nx;
                        s_a = z > k;
                    }
                }
                __syncthreads();
                price = s_lam;
                low = s_a;
                if (s_flag != kGo) break;
                __syncthreads();
            }
            if (s_flag != kCoarser) break;
            ++ev;
            shift += kCoarserBits;
            sync_all();                      // no CTA reads the old units any more
        }
        if (s_flag == kSlack) price = 0;
        lam = (int64_t)price << shift;
        if (s_flag != kTooDear) {
            // ---- exactly there: f of every row, L
            for (int i = tid; i <= na; i += kThreads) own.limb[i] = make_int4(0, 0, 0, 0);
            __syncthreads();
            int64_t ry = 0;
            exact_bin<!SMEM>(info, g.prof + lo, g.f + lo, g.topl, lists[0][warp], tiles, nlev, own, base, na, lam, ring, ry);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) ry += __shfl_xor_sync(kAll, ry, o);
            if (lane == 0 && ry) atomicAdd(&g.s->sumL, (unsigned long long)ry);
            sync_all();
            if (warp == 0) {
                ry = has_top ? exact_top(t, g, s_top, lam) : 0;
                if (lane == 0) s_val = (int64_t)__ldcg(&g.s->sumL) + ry + lam * k;
            }
            __syncthreads();
            L = s_val;
        }
    }
    const bool give_up = too_large || s_flag == kTooDear;

    // ---- losses and their histogram
    unsigned *ghist = g.hist + kBins;
    if (!give_up) {
        // (at price 0 the largest profit stands for it)
        const float unit = lam > 0 ? (float)lam * A.mean_weight : (float)maxp;
        const int shift = max(0, (int)(__float_as_uint(fmaxf(unit, 1.f)) >> 23) - 127 - kLossBits);
        for (int i = tid; i < kBins; i += kThreads) hist[i] = 0;
        __syncthreads();
        if (has_top) {
            if (warp == 0) loss_top(t, g, (Down *)s_top, shift, hist, cr == 0);
            __syncthreads();
        }
        loss_bin<!SMEM>(info, g.f + lo, g.key + lo, lists[0][warp], tiles, nlev, own, base, (const Down *)s_top, shift, ring, hist);
        __syncthreads();
        for (int i = tid; i < kBins; i += kThreads)
            if (hist[i]) atomicAdd(ghist + i, hist[i]);
        sync_all();
    }
    // the largest key up to `most` whose rows, and all below, are at most
    // `rows` (but at least key 0), and their number
    auto up_to = [&](int rows, int most, int &key_out) {
        constexpr int V = kBins / kThreads;
        int c[V], sum = 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            c[v] = (int)__ldcg(ghist + tid * V + v);
            sum += c[v];
        }
        if (tid == 0) s_a = s_b = 0;
        int tot;
        int ex = block_scan(sum, &tot, sh);              // (orders the line above too)
        int last = -1, cnt = 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            ex += c[v];
            const int q = tid * V + v;
            if (q == 0 || (q <= most && ex <= rows)) {
                last = q;
                cnt = ex;
            }
        }
        if (last >= 0) {
            atomicMax(&s_a, last);
            atomicMax(&s_b, cnt);
        }
        __syncthreads();
        key_out = s_a;
        const int r = s_b;
        __syncthreads();
        return r;
    };

    int verdict = 3, key = 0, pass = 0, vkey = -1;      // vkey: the smallest sure key so far (first CTA)
    bool sure = false;           // the key comes from a V: no row above it is undecided
    // time of a threshold with T rows, and the rows that what is left to spend
    // allows for one more after it (one that is sure to succeed is not refused)
    auto pass_us = [&](int T) { return kPassUs + (float)T * (A.max_weight > 1 ? kWeightedRowUs : kRowUs); };
    auto rows_left = [&](float more) {
        const float us = s_search.left - more - kPassUs;
        return (int)fminf(fmaxf(us * (A.max_weight > 1 ? 1.f / kWeightedRowUs : 1.f / kRowUs), 0.f), (float)kRowCap);
    };
    if (!give_up) {
        int T = 0;
        // first the rows whose loss is within 0.1 of the price of a chunk's
        // slots (most gaps are), at most kFirstRows; none at price 0 (see
        // kleft < 0 below)
        if (lam == 0) {
            key = -1;
        } else {
            T = up_to(min(kFirstRows, rows_left(0.f)), code_of((int64_t)(0.1f * (float)lam * A.mean_weight)), key);
        }
        for (; pass < kPasses; ++pass) {
            const bool big = T > (sure ? kRowCap : rows_left(0.f));       // the same in every CTA
            verdict = 3;
            if (big && !sure) break;
            // ---- decided rows: value and weight of those in; the others' positions
            if (pass > 0) {
                for (int i = cr * kThreads + tid; i < words; i += CL * kThreads) freeb[i] = 0;
                sync_all();
            }
            unsigned long long vf = 0, wf = 0;
            auto classify = [&](int a, int b) {
#pragma unroll 4
                for (int s = a + tid; s < b; s += kThreads) {
                    const int c = g.key[s];
                    const int kk = c & 0x7fff;
                    if (c == kKeyPad) continue;
                    if (kk <= key) {
                        const int x = __ldg(t.pos + s);
                        atomicOr(freeb + (x >> 5), 1u << (x & 31));
                    } else if (c & 0x8000) {
                        vf += (unsigned long long)g.prof[s];
                        wf += (unsigned)(__ldg(&t.info[s].x) >> kWeightShift);
                    }
                }
            };
            classify(lo, hi);
            if (cr == 0 && has_top) classify(top0, t.nslots);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                vf += __shfl_xor_sync(kAll, vf, o);
                wf += __shfl_xor_sync(kAll, wf, o);
            }
            if (lane == 0) {
                if (vf) atomicAdd(&g.s->vfix[pass], vf);
                if (wf) atomicAdd(&g.s->wfix[pass], wf);
            }
            sync_all();
            if (big) {
                verdict = 4;
                break;
            }
            // ---- the first CTA: DP over the undecided rows, on chip
            if (cr == 0) {
                Rows &R = *(Rows *)smem;
                unsigned char *pool = smem + up16(sizeof(Rows));
                const int64_t vfix = (int64_t)__ldcg(&g.s->vfix[pass]);
                const int64_t kleft = k - (int64_t)__ldcg(&g.s->wfix[pass]);
                int out = 0, okey = 0;       // 1 solved, 2 again with okey (5: which is sure), 3 not reducible, 4 to the sweep
                if (kleft < 0) {                        // too few rows undecided: take more by rank
                    out = 2;
                    const int most = rows_left(kPassUs);
                    up_to(min(kFirstRows, most), kBins, okey);
                    if (okey <= key) up_to(min(kMoreRows, most), kBins, okey);
                    if (okey <= key) up_to(most, kBins, okey);
                    if (okey <= key) out = 3;
                } else {
                    // rows in sweep order from the bitmap
                    const int per = (words + kThreads - 1) / kThreads;
                    const int w0 = min(words, tid * per), w1 = min(words, w0 + per);
                    int c = 0;
#pragma unroll 4
                    for (int i = w0; i < w1; ++i) c += __popc(__ldcg(freeb + i));
                    int tot;
                    int ex = block_scan(c, &tot, sh);
                    if (c)
                        for (int i = w0; i < w1; ++i) {
                            uint32_t m = __ldcg(freeb + i);
                            while (m) {
                                const int x = i * 32 + __ffs((int)m) - 1;
                                m &= m - 1;
                                R.pos[T - 1 - ex] = x;
                                ++ex;
                            }
                        }
                    __syncthreads();
                    int wsum = 0;                       // capped: far above every column cap
                    for (int r = tid; r < (T + 31 & ~31); r += kThreads) {
                        bool leaf = false;
                        if (r < T) {
                            const int x = R.pos[r];
                            const int w = __ldg(A.wpre + x);
                            R.row[r].p = P[A.order ? __ldg(A.order + x) : x];
                            R.row[r].w = w;
                            wsum += min(w, 1 << 18);
                            R.last[r] = -1;
                            // the first undecided row at or after next(x), -1: none
                            const int nx = __ldg(A.next + x);
                            int a = 0, b = r;           // rows 0..a-1 have pos >= nx
                            while (a < b) {
                                const int mid = (a + b) >> 1;
                                if (R.pos[mid] >= nx) a = mid + 1;
                                else b = mid;
                            }
                            R.step[r] = make_int2(w, a - 1);
                            leaf = a == r;
                        }
                        const unsigned lm = __ballot_sync(kAll, leaf);
                        if (lane == 0) R.leaf[r >> 5] = lm;
                    }
                    int wtot;
                    block_scan(wsum, &wtot, sh);
                    const int kc = (int)(kleft < wtot ? kleft : wtot);
                    // stack plan, as the pruned sweep's: a row read through the
                    // stack is pushed when computed and popped after its last reader
                    for (int r = tid; r < T; r += kThreads) {
                        const int sk = R.step[r].y;
                        if (sk >= 0 && sk != r - 1) atomicMax(&R.last[sk], r);
                    }
                    if (tid == 0) s_a = 0;
                    __syncthreads();
                    int depth = 0;
                    for (int base = 0; base < T; base += kThreads) {
                        const int r = base + tid;
                        int sk = -1;
                        bool pop = false, push = false;
                        if (r < T) {
                            sk = R.step[r].y;
                            pop = sk >= 0 && sk != r - 1 && R.last[sk] == r;
                            push = R.last[r] >= 0;
                        }
                        int dt;
                        const int ex2 = block_scan((int)push - (int)pop, &dt, sh) + depth;
                        if (r < T) {
                            const int dd = ex2 - (int)pop;
                            int fl = 0, lvl = 0;
                            if (push) {
                                fl = kPush;
                                lvl = dd;
                                atomicMax(&s_a, dd + 1);
                            } else if (pop && dd > 0) {
                                fl = kReload;
                                lvl = dd - 1;
                            } else if (pop) {
                                fl = kZeroTop;
                            }
                            if (sk >= 0 && sk == r - 1 && R.last[r - 1] < 0) fl |= kFromCur;
                            R.row[r].info = fl | (lvl << 8);
                        }
                        depth += dt;
                    }
                    __syncthreads();
                    const int levels = s_a;
                    const int act = max(1, (kc + 31) / 32);          // warps that hold columns
                    const int cols = act * 32;
                    const int guard = min(A.max_weight, cols);
                    const int pitch = cols + 1 + guard;
                    const size_t need = (size_t)2 * pitch * 8 + (size_t)levels * cols * 8 + (size_t)((T + 31) / 32) * cols * 4;
                    const int C = kc <= 32 ? 1 : kc <= 64 ? 2 : 4;   // columns per lane of the one-warp kernel
                    const size_t uneed = (size_t)levels * 32 * C * 10 + (size_t)(T + 6) * 32 * C * 2 + 16;
                    const bool unit = A.max_weight == 1 && kc <= kUnitCols && uneed <= (size_t)kPool;
                    const int ucols = 32 * C;
                    if (kc > kColCap || (!unit && need > (size_t)kPool)) {
                        out = sure ? 4 : 3;
                    } else {
                        int64_t *rowb = (int64_t *)pool;             // [2][guard + 1 + cols]
                        int64_t *stk = rowb + 2 * pitch;             // [levels][cols]
                        uint32_t *bits = (uint32_t *)(stk + (size_t)levels * cols);   // [T / 32][cols]
                        int64_t *ustk = (int64_t *)pool;             // [levels][ucols]
                        // [T + 4][ucols], two rows of zeros (and a little) before
                        uint16_t *first = (uint16_t *)(ustk + (size_t)levels * ucols) + 8 + 2 * ucols;
                        uint16_t *stf = first + (size_t)(T + 4) * ucols;     // [levels][ucols]
                        if (unit)
                            for (int i = tid; i < 8 + 2 * ucols; i += kThreads) first[i - 8 - 2 * ucols] = 0;
                        if (!unit) {
                            for (int i = tid; i < 2 * pitch; i += kThreads) rowb[i] = i % pitch < guard ? -2 * kBig : 0;
                            for (int r = tid; r < T; r += kThreads)
                                if (R.row[r].w > cols) R.row[r].w = cols + 1;    // never fits: column 0's guard
                        }
                        if (tid == 0) s_val = 0;
                        if (tid < 4) {
                            R.row[T + tid].p = -kBig;                // no-op rows: never taken
                            R.row[T + tid].w = 0;
                            R.row[T + tid].info = kFromCur;
                        }
                        __syncthreads();
                        if (!unit) {
                            if (warp < act) dp_rows(R, T, act, guard, rowb, stk, bits, &s_val, kc);
                        } else if (warp == 0) {
                            if (C == 1) dp_unit<1>(R, T, ustk, stf, first, &s_val, kc);
                            else if (C == 2) dp_unit<2>(R, T, ustk, stf, first, &s_val, kc);
                            else dp_unit<4>(R, T, ustk, stf, first, &s_val, kc);
                        }
                        __syncthreads();
                        const int64_t V = vfix + s_val;
                        // at price 0 with |S| <= k, S is Eq. 9's set: a chunk is
                        // taken iff what it brings is positive
                        const int need_key = key < 0 ? -1 : code_of(L - V);
                        if (need_key <= key) {
                            out = 1;
                            // walk the decisions: in a 32-row word of the column, the
                            // next row that is taken or whose skip is no leaf's
                            if (tid == 0) {
                                int r = T - 1, j = kc;
                                int m = 0;                   // rows taken (plus 1), listed in R.last
                                if (unit) {
                                    // Four steps a trip, nothing tested in between (a branch a
                                    // step: 94 ns each, so 26): after a 0 the walk stays in
                                    // the zeros.  What it reads left of
                                    // column 1, after kc steps, is not listed.
                                    for (; m < kc; m += 4) {
                                        int v = 0;
#pragma unroll
                                        for (int u = 0; u < 4; ++u) {
                                            v = first[r * ucols + j - 1];
                                            R.last[m + u] = v;
                                            r = v - 2;
                                            --j;
                                        }
                                        if (v == 0) break;
                                    }
                                    m = min(m + 4, kc);
                                }
                                while (!unit && r >= 0 && j > 0) {
                                    const int blk = r >> 5;
                                    const uint32_t word = bits[blk * cols + j - 1];
                                    const uint32_t cand = (word | ~R.leaf[blk]) & (0xffffffffu >> (31 - (r & 31)));
                                    const int rr = (r & ~31) + 31 - __clz((int)cand);      // below the block if none
                                    const int2 st = R.step[max(rr, 0)];
                                    const bool none = cand == 0, take = (cand & word) >> (rr & 31) & 1u;
                                    if (!none && take) R.last[m++] = rr + 1;
                                    j -= !none && take ? st.x : 0;
                                    r = none || take ? rr - !none : st.y;
                                }
                                s_a = m;
                                A.best[item] = V;
                                A.w.nkept[item] = T;
                                if (A.rows_kept) atomicAdd(A.rows_kept, (unsigned long long)T);
                            }
                            __syncthreads();
                            for (int i = tid; i < s_a; i += kThreads) {
                                if (R.last[i] == 0) continue;
                                const int x = R.pos[R.last[i] - 1];
                                atomicOr(taken + (x >> 5), 1u << (x & 31));
                            }
                        } else {
                            out = 5;
                            okey = vkey = vkey < 0 ? need_key : min(vkey, need_key);
                            int same;
                            if (pass < kPasses - 2 && up_to(INT_MAX, okey, same) > kRowCap) {
                                // a V from more rows may need fewer (an item of 50,000
                                // rows: 16,299 left by the V of 591 rows, 1,447 by that of
                                // 1,010; the sweep of the former took 1.5 ms)
                                int more;
                                const int most = rows_left(pass_us(T));
                                up_to(T < kMoreRows * 7 / 8 ? min(kMoreRows, most) : most, kBins, more);
                                if (more > key) {
                                    out = 2;
                                    okey = more;
                                }
                            }
                        }
                    }
                }
                if (out == 3 && vkey >= 0) {
                    out = 5;
                    okey = vkey;
                }
                if (tid == 0) {
                    g.s->key[pass] = okey;
                    g.s->verdict[pass] = out;
                }
            }
            if (tid == 0) s_search.left -= pass_us(T);
            sync_all();
            verdict = __ldcg(&g.s->verdict[pass]);
            if (verdict != 2 && verdict != 5) break;
            sure = verdict == 5;
            key = __ldcg(&g.s->key[pass]);
            int same;
            T = up_to(INT_MAX, key, same);
        }
    }
    const int state = verdict == 1 ? 1 : verdict == 4 ? 2 : 0;
    chain_release();
    // ---- the decided "in" rows join the set
    if (state) {
        auto mark = [&](int a, int b) {
#pragma unroll 4
            for (int s = a + tid; s < b; s += kThreads) {
                const int c = g.key[s];
                if (c == kKeyPad || !(c & 0x8000) || (c & 0x7fff) <= key) continue;
                const int x = __ldg(t.pos + s);
                atomicOr(taken + (x >> 5), 1u << (x & 31));
            }
        };
        mark(lo, hi);
        if (cr == 0 && has_top) mark(top0, t.nslots);
    }
    if (cr == 0 && tid == 0) {
        *red = state;
        if (state == 2) {
            A.w.left[item] = (int32_t)(k - (int64_t)__ldcg(&g.s->wfix[pass]));
            A.w.base[item] = (int64_t)__ldcg(&g.s->vfix[pass]);
        }
    }
    if (state != 1) prune_left(A, item, state == 2 ? freeb : nullptr);
}

// ---------------------------------------------------------------------------
// host: the layout (see the top of the file), one device block per instance
// ---------------------------------------------------------------------------
// Bins of a tree: the most CTAs that can share an item.  One price costs
// 12.4 us on 6 CTAs and 8.6 on 8 (50,000 rows), 19.5 on 8 and 11.3 on 16
// (200,000 rows): 32 warps on four schedulers issue some 150 instructions a
// tile each.  But more bins put more rows into the last one and more padding
// into the tiles: at 10,000 rows 8 CTAs are 6% slower than 6.  Below 1,536
// rows one CTA is as fast as any cluster.
static int bins_of(int n) { return n <= 1536 ? 1 : n <= 12288 ? 6 : 16; }

bool build_reduce_tables(int32_t n, const std::vector<int32_t> &par, const std::vector<int32_t> &next,
                         const std::vector<int32_t> &wpre, int64_t total_weight, int32_t max_weight,
                         ReduceTables *out)
{
    ReduceTables &R = *out;
    R = ReduceTables();
    if (n < kReduceMinRows || max_weight > kMaxWeight || total_weight >= ((int64_t)1 << 30)) return false;
    int NB = bins_of(n);
    // rows of a subtree that stays in one bin: half a CTA's share, more
    // if that leaves too many rows above the bins
    std::vector<int32_t> kids(n, 0), heavy(n, -1), best(n, 0);
    for (int32_t i = 0; i < n; ++i) {
        const int p = par[i];
        if (p < 0) continue;
        if (++kids[p] > kMaxKids) return false;
        R.max_kids = std::max(R.max_kids, kids[p]);
    }
    int limit = n;
    if (NB > 1) {
        limit = std::max(64, n / (2 * NB));
        for (;; limit *= 2) {
            int above = 0;
            for (int32_t i = 0; i < n; ++i) above += next[i] - i > limit;
            if (above <= kMaxTop) break;
            if (limit >= n / 2) {
                NB = 1;
                limit = n;
                break;
            }
        }
    }
    auto is_top = [&](int i) { return next[i] - i > limit; };
    // bins: subtrees below the limit, each to the emptiest bin
    std::vector<int32_t> bin(n), level(n, 0), acc(n, -1);
    std::vector<int64_t> load(NB, 0);
    for (int32_t i = 0; i < n; ++i) {
        const int p = par[i];
        if (is_top(i)) bin[i] = NB;
        else if (p >= 0 && bin[p] != NB) bin[i] = bin[p];
        else {
            const int b = (int)(std::min_element(load.begin(), load.end()) - load.begin());
            bin[i] = b;
            load[b] += next[i] - i;
        }
        const int sz = next[i] - i;
        if (p >= 0 && bin[p] == bin[i] && sz > best[p]) {
            best[p] = sz;
            heavy[p] = i;
        }
    }
    R.nacc.assign(NB + 1, 0);
    int maxlev = 0;
    for (int32_t i = n - 1; i >= 0; --i) {
        const int p = par[i];
        maxlev = std::max(maxlev, level[i]);
        if (p < 0) continue;
        if (heavy[p] == i) level[p] = std::max(level[p], level[i]);
        else if (bin[p] == bin[i]) level[p] = std::max(level[p], level[i] + 1);
        if (heavy[p] != i && acc[p] < 0) acc[p] = R.nacc[bin[p]]++;
    }
    for (int b = 0; b <= NB; ++b)
        if (R.nacc[b] >= kNone) return false;
    // path tops grouped by (bin, level)
    const int nl = maxlev + 1;
    if (nl > kMaxLevels) return false;
    std::vector<int32_t> start((size_t)(NB + 1) * nl + 1, 0), rows((size_t)(NB + 1) * nl, 0), tops, len(n, 0);
    for (int32_t i = n - 1; i >= 0; --i) len[i] = 1 + (heavy[i] >= 0 ? len[heavy[i]] : 0);
    auto path_top = [&](int i) { return par[i] < 0 || heavy[par[i]] != i; };
    for (int32_t i = 0; i < n; ++i)
        if (path_top(i)) {
            const size_t q = (size_t)bin[i] * nl + level[i];
            start[q + 1]++;
            rows[q] += len[i];
            if (len[i] > kMaxPathRows) return false;
        }
    for (size_t q = 0; q + 1 < start.size(); ++q) start[q + 1] += start[q];
    tops.resize(start.back());
    {
        std::vector<int32_t> at(start.begin(), start.end() - 1);
        for (int32_t i = 0; i < n; ++i)
            if (path_top(i)) tops[at[(size_t)bin[i] * nl + level[i]]++] = i;
    }
    R.info.reserve((size_t)n + 32 * 64);
    R.pos.reserve((size_t)n + 32 * 64);
    std::vector<int32_t> path, to(tops.size()), mine[kWarps];
    for (int b = 0; b <= NB; ++b) {
        R.binslot.push_back((int32_t)R.info.size());
        R.binlev.push_back((int32_t)R.lev.size());
        int levels = nl;
        while (levels > 0 && rows[(size_t)b * nl + levels - 1] == 0) --levels;
        for (int l = 0; l < levels; ++l) {
            const size_t q = (size_t)b * nl + l;
            R.lev.push_back((int32_t)R.stream.size());
            // streams, at most one per warp: the fewest tiles each (one, where
            // the level has rows for no more) that take every path, in the
            // first stream with room (the next stream only: 15% more tiles);
            // a longer path has a stream of its own
            int room = (rows[q] + 32 * kWarps - 1) / (32 * kWarps) * 32, streams = 0;
            int used[kWarps];
            for (;; room += 32) {
                streams = 0;
                bool fits = true;
                for (int x = start[q]; x < start[q + 1] && fits; ++x) {
                    const int l1 = len[tops[x]];
                    int y = 0;
                    while (y < streams && used[y] + l1 > room) ++y;
                    fits = y < kWarps;
                    if (!fits) break;
                    if (y == streams) used[streams++] = 0;
                    used[y] += l1;
                    to[x] = y;
                }
                if (fits) break;
            }
            for (int x = start[q]; x < start[q + 1]; ++x) mine[to[x]].push_back(tops[x]);
            for (int st = 0; st < streams; ++st) {
                const int tile0 = (int)(R.info.size() / 32);
                for (int topn : mine[st]) {
                    path.clear();
                    for (int v = topn; v >= 0; v = heavy[v]) path.push_back(v);
                const int first = (int)R.info.size();            // the path's first slot
                    for (int y = (int)path.size() - 1; y >= 0; --y) {
                        const int v = path[y];
                        const int s = (int)R.info.size(), t0 = s & ~31;
                        int code = (s - std::max(first, t0)) | (first < t0 ? kCont : 0) | (v == topn ? kTop : 0) |
                                   (wpre[v] << kWeightShift);
                        int up = kNone;
                        if (v == topn && par[v] >= 0) {
                            up = acc[par[v]];
                            if (bin[par[v]] != bin[v]) code |= kUp;
                        }
                        if (s == t0) R.form.push_back(l == 0 ? (first < t0 ? 3 : 1) : 0);
                        R.info.push_back({code, (acc[v] < 0 ? kNone : acc[v]) | (int)((unsigned)up << 16)});
                        R.pos.push_back(v);
                    }
                }
                while (R.info.size() % 32) {
                    R.info.push_back({0, kNone | (int)((unsigned)kNone << 16)});
                    R.pos.push_back(-1);
                }
                R.stream.push_back({tile0, (int)(R.info.size() / 32) - tile0});
                mine[st].clear();
            }
        }
        R.lev.push_back((int32_t)R.stream.size());
    }
    R.binslot.push_back((int32_t)R.info.size());
    R.binlev.push_back((int32_t)R.lev.size());
    // the cluster sizes: every warp's tiles have to fit its list (streams go
    // round the warps as the kernel deals them)
    for (int cl = NB; cl >= 1; --cl) {
        if (NB % cl) continue;
        const int per = NB / cl;
        int most = 0, acc_most = 0, longest = 0;
        for (int r = 0; r < cl; ++r) {
            int tiles[kWarps] = {}, at = 0, accs = 0, path = 0;
            for (int l = 0; l < kMaxLevels; ++l) {
                int level[kWarps] = {};
                for (int b = r * per; b < (r + 1) * per; ++b) {
                    const int e = R.binlev[b] + l;
                    if (e + 1 >= R.binlev[b + 1]) continue;
                    for (int x = R.lev[e]; x < R.lev[e + 1]; ++x) level[at++ % kWarps] += R.stream[x].tiles;
                }
                for (int q = 0; q < kWarps; ++q) tiles[q] += level[q];
                path += *std::max_element(level, level + kWarps);
            }
            longest = std::max(longest, path);
            for (int b = r * per; b < (r + 1) * per; ++b) accs += R.nacc[b];
            most = std::max(most, *std::max_element(tiles, tiles + kWarps));
            acc_most = std::max(acc_most, accs);
        }
        if (most > kMaxTiles || acc_most >= kNone) break;
        R.cluster.push_back({cl, acc_most, longest});
    }
    if (R.cluster.empty()) return false;
    R.bins = NB;
    return true;
}

static size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

// device block: info | positions | forms | streams | levels | binlev | binslot | nacc
size_t reduce_tables_bytes(const ReduceTables &R)
{
    return al(R.info.size() * 8) + al(R.info.size() * 4) + al(R.form.size()) + al(R.stream.size() * 8) +
           al(R.lev.size() * 4) + al(R.binlev.size() * 4) +
           al(R.binslot.size() * 4) + al(R.nacc.size() * 4);
}

void reduce_tables_pack(const ReduceTables &R, char *dst)
{
    auto put = [&](const void *src, size_t bytes) {
        std::memcpy(dst, src, bytes);
        dst += al(bytes);
    };
    put(R.info.data(), R.info.size() * 8);
    put(R.pos.data(), R.info.size() * 4);
    put(R.form.data(), R.form.size());
    put(R.stream.data(), R.stream.size() * 8);
    put(R.lev.data(), R.lev.size() * 4);
    put(R.binlev.data(), R.binlev.size() * 4);
    put(R.binslot.data(), R.binslot.size() * 4);
    put(R.nacc.data(), R.nacc.size() * 4);
}

static Tab device_tab(const pp_instance *inst)
{
    const ReduceShape &r = inst->red;
    char *p = (char *)inst->d_red;
    auto take = [&](size_t bytes) {
        char *q = p;
        p += al(bytes);
        return q;
    };
    Tab t;
    t.n = inst->n;
    t.bins = r.bins;
    t.nslots = r.nslots;
    t.ntop = r.ntop;
    t.info = (const int2 *)take((size_t)r.nslots * 8);
    t.pos = (const int *)take((size_t)r.nslots * 4);
    t.form = (const uint8_t *)take((size_t)r.nslots / 32);
    t.stream = (const int2 *)take((size_t)r.nstreams * 8);
    t.lev = (const int *)take((size_t)r.nlev * 4);
    t.binlev = (const int *)take((size_t)(r.bins + 2) * 4);
    t.binslot = (const int *)take((size_t)(r.bins + 2) * 4);
    t.nacc = (const int *)take((size_t)(r.bins + 1) * 4);
    return t;
}

// shared memory of the scans, with up to `acc` accumulators of a CTA there
static size_t scan_bytes(int acc, bool acc_smem)
{
    return (acc_smem ? up16((size_t)(acc + 1) * kAccBytes) : 0) + kRingBytes + kBins * 4;
}
constexpr size_t kAccLimit = (size_t)192 << 10;

ReduceShape reduce_shape(const ReduceTables &R, int32_t n, int32_t max_weight)
{
    ReduceShape s;
    s.bins = R.bins;
    s.nslots = (int)R.info.size();
    s.nstreams = (int)R.stream.size();
    s.nlev = (int)R.lev.size();
    s.ntop = R.nacc[R.bins];
    s.toptiles = (s.nslots - R.binslot[R.bins]) / 32;
    s.max_kids = R.max_kids;
    for (const auto &c : R.cluster) {
        s.cl[s.ncl] = c.cl;
        s.path[s.ncl] = c.path;
        s.acc[s.ncl++] = c.acc;
        if (scan_bytes(c.acc, true) > kAccLimit) s.acc_global = 1;
    }
    s.item_bytes = al(carve(nullptr, s.nslots, s.ntop, s.acc_global, nullptr));
    set_spending(s, n, max_weight, kMaxEvals);
    return s;
}

// scratch of one item in the DP workspace, 0 when the instance has no reduction
size_t reduce_item_bytes(const pp_instance *inst)
{
    return inst->red.bins ? inst->red.item_bytes : 0;
}

// Once per instance: the kernels' attributes, and how many clusters above the
// portable size the device holds at once.  Attributes belong to the process, so
// every instance sets the same: all the shared memory that the device allows.
pp_status reduce_device(ReduceShape *r)
{
    if (!r->ncl) return PP_OK;
    int dev = 0, limit = 0;
    PP_CUDA(cudaGetDevice(&dev));
    PP_CUDA(cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    for (const void *fn : {(const void *)k_reduce<true>, (const void *)k_reduce<false>}) {
        cudaFuncAttributes at;
        PP_CUDA(cudaFuncGetAttributes(&at, fn));
        PP_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, limit - (int)at.sharedSizeBytes));
        PP_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    }
    if (r->cl[0] <= kPortable) return PP_OK;
    const bool acc_smem = scan_bytes(r->acc[0], true) <= kAccLimit;
    const auto kern = acc_smem ? k_reduce<true> : k_reduce<false>;
    const size_t smem = std::max(scan_bytes(r->acc[0], acc_smem), up16(sizeof(Rows)) + kPool);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(r->cl[0]);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = r->cl[0];
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int wide = 0;
    if (cudaOccupancyMaxActiveClusters(&wide, kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        wide = 0;
    }
    set_wide(*r, wide);
    return PP_OK;
}

pp_status launch_reduce(pp_instance *inst, int batch, const int64_t *profit, bool by_node,
                        const int32_t *item_budget, const int32_t *item_active, int64_t *best, const DpWork &work,
                        cudaStream_t st, int32_t max_budget, unsigned long long *rows_kept)
{
    const ReduceShape &r = inst->red;
    Args a;
    a.t = device_tab(inst);
    a.profit = profit;
    a.order = by_node ? inst->d_order : nullptr;
    a.next = inst->d_next;
    a.wpre = inst->d_wpre;
    a.item_budget = item_budget;
    a.item_active = item_active;
    a.max_budget = max_budget;
    a.best = best;
    a.rows_kept = rows_kept;
    a.w = work;
    a.item_bytes = reduce_item_bytes(inst);
    a.total_weight = inst->total_weight;
    a.mean_weight = (float)inst->total_weight / (float)inst->n;
    a.max_weight = inst->max_weight;
    a.pspan = inst->d_pspan;
    a.stack_depth = inst->stack_depth;
    a.status = inst->d_status;
    a.clip_kid = std::min(1 << 22, (1 << 30) / std::max(1, r.max_kids));
    const int x = cluster_index(r, std::max(work.items, batch));
    a.t.CL = r.cl[x];
    a.spending = r.spending[x];
    const bool acc_smem = scan_bytes(r.acc[x], true) <= kAccLimit;
    const size_t smem = std::max(scan_bytes(r.acc[x], acc_smem), up16(sizeof(Rows)) + kPool);
    const auto kern = acc_smem ? k_reduce<true> : k_reduce<false>;
    PP_CUDA(launch_chained(kern, dim3(r.cl[x] * batch), dim3(kThreads), smem, st, r.cl[x], a));
    return PP_OK;
}

}  // namespace pp
