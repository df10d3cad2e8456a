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
// their keys (an order-preserving 11-bit code of the loss), so every test
// errs on the side of keeping a row.
//
// A prefix tree of 50,000 chunks with the planner's profits leaves 10 to 1,500
// undecided rows of the 16,000 to 37,000 that the pruned sweep keeps, and a
// budget of a few hundred slots instead of 4,096.  More undecided rows than
// fit on chip (chunks in long chains that are worth taking only whole) go to
// pp_dp.cu's kernels with what is left of the budget; where no V is found
// (ties that leave nearly everything undecided) those kernels get every row.
//
// Layout.  f is a Lindley recursion along every heavy path of the tree
// (y_i = max(0, d_i + y_(i+1)), d_i the row's own term plus its light
// children), so a path is a scan of the maps x -> max(m, s + x), and losses
// are scans the other way.  Heavy paths bound the dependent levels by
// log2(n) + 1 for every tree shape (6 to 9 on the prefix trees here, whose
// depth is 72 and more).  Rows are laid out by (bin, level, path), bottom of
// the path first, in tiles of 32 (one per warp step).  A bin is a set of
// whole subtrees of at most n / (4 CL) rows, one bin per CTA of the cluster,
// so that levels are separated by block barriers only; the few nodes above
// all bins form a last bin that the first CTA walks after a cluster barrier.
#include <algorithm>
#include <climits>
#include <cstring>

#include "pp_internal.cuh"

namespace pp {

namespace {

constexpr unsigned kAll = 0xffffffffu;
constexpr int kThreads = 512;               // per CTA
constexpr int kWarps = kThreads / 32;
constexpr int kMaxEvals = 16;               // prices tried per item
constexpr int kPasses = 4;                  // thresholds tried per item
constexpr int kRowCap = 1024;               // undecided rows the on-chip DP takes
constexpr int kFirstRows = 256;             // rows of the first threshold (by rank of the loss)
constexpr int kColCap = 1024;               // its columns (budget left over)
constexpr int kPool = 64 << 10;             // its decision bits, stack and row buffers, bytes
constexpr int kKeyBase = (127 << 5) - 1;    // float bits >> 18 of 1.0, minus 1
constexpr int kBins = 2048;                 // keys of 0 .. 2^62
constexpr int kKeyPad = 0xffff;
constexpr int64_t kBig = (int64_t)1 << 61;
constexpr int kMaxWeight = (1 << 22);       // weights ride in the slot code
constexpr int kMaxPathRows = 4096;          // longer heavy paths are left to the sweep

// slot code: bits 0-4 lanes to the left in the same path and tile, 5 the path
// comes from the previous tile, 6 top of its path, 8.. weight
constexpr int kCont = 32, kTop = 64, kWeightShift = 8;

struct Tab {
    int n, CL, nslots, ntop;
    const int4 *slot;            // position (-1 pad), code, accumulator (-1 none), parent
    const int2 *stream;          // first tile, tiles: what one warp walks in sequence
    const int *lev;              // stream boundaries of the levels
    const int *binlev;           // [CL + 2] boundaries of a bin's entries in lev
    const int *binslot;          // [CL + 2] first slot of a bin
    const int *nacc;             // [CL + 1] accumulators of a bin
};

struct Scal {                    // per item, zeroed by the kernel
    unsigned long long maxp;
    unsigned long long sumL[kMaxEvals];
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
    int acc_smem;                // accumulators in shared memory
    int64_t total_weight;
    int32_t max_weight;
};

__host__ __device__ inline size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }

// one item's scratch
struct Scratch1 {
    Scal *s;
    unsigned *hist;              // [kBins]
    int64_t *prof, *f;           // [nslots]
    uint16_t *key;               // [nslots]
    long long *topY, *topLin, *topLout;      // [ntop]
    int *topZ;
    long long *accY, *accLin, *accLout;      // [nslots] when not in shared memory
    int *accZ;
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
    x.hist = (unsigned *)take(kBins * 4);
    x.topY = (long long *)take((size_t)ntop * 8);
    x.topZ = (int *)take((size_t)ntop * 4);
    x.topLin = (long long *)take((size_t)ntop * 8);
    x.topLout = (long long *)take((size_t)ntop * 8);
    x.prof = (int64_t *)take((size_t)nslots * 8);
    x.f = (int64_t *)take((size_t)nslots * 8);
    x.key = (uint16_t *)take((size_t)nslots * 2);
    const size_t na = acc_global ? (size_t)nslots : 0;
    x.accY = (long long *)take(na * 8);
    x.accZ = (int *)take(na * 4);
    x.accLin = (long long *)take(na * 8);
    x.accLout = (long long *)take(na * 8);
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

// order-preserving code of a loss >= 0, in [0, kBins)
__device__ __forceinline__ int loss_key(int64_t loss)
{
    if (loss <= 0) return 0;
    return (int)(__float_as_uint(__ll2float_rd(loss)) >> 18) - kKeyBase;
}

__device__ __forceinline__ int64_t sat(int64_t x) { return x < kBig ? x : kBig; }

// f, and the values and sizes of the best closed sets, of one bin at price lam
struct BinAcc {
    volatile long long *y, *lin, *lout;
    volatile int *z;
};

__device__ void eval_bin(const Tab &t, int b, const Scratch1 &g, const BinAcc &own, const BinAcc &top, int64_t lam,
                         int64_t &rootY, int &rootZ)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l0 = t.binlev[b], l1 = t.binlev[b + 1] - 1;
    for (int l = l0; l < l1; ++l) {
        const int s1 = t.lev[l + 1];
        for (int s = t.lev[l] + warp; s < s1; s += kWarps) {
            const int2 st = t.stream[s];
            int64_t carryY = 0;
            int carryZ = 0;
            for (int q = 0; q < st.y; ++q) {
                const int slot = (st.x + q) * 32 + lane;
                const int4 e = t.slot[slot];
                const int off = e.y & 31, w = e.y >> kWeightShift;
                const bool cont = e.y & kCont;
                int64_t d = g.prof[slot] - lam * w;
                int zz = w;
                if (e.z >= 0) {
                    d += own.y[e.z];
                    zz += own.z[e.z];
                    own.y[e.z] = 0;            // for the next price
                    own.z[e.z] = 0;
                }
                // inclusive scan of x -> max(m, s + x) along the path
                int64_t m = 0, sm = d;
                int ps = zz;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int64_t m2 = __shfl_up_sync(kAll, m, o), s2 = __shfl_up_sync(kAll, sm, o);
                    const int p2 = __shfl_up_sync(kAll, ps, o);
                    if (off >= o) {
                        const int64_t v = sm + m2;
                        m = m > v ? m : v;
                        sm += s2;
                    }
                    if (lane >= o) ps += p2;
                }
                const int64_t v = sm + (cont ? carryY : 0);
                const int64_t y = m > v ? m : v;
                int64_t yp = __shfl_up_sync(kAll, y, 1);
                if (off == 0) yp = cont ? carryY : 0;
                const int64_t f = d + yp;
                g.f[slot] = f;
                // size of the best closed set below (and with) this row
                const bool in = f > 0;
                const unsigned seg = (2u << lane) - (1u << (lane - off));
                const unsigned neg = __ballot_sync(kAll, !in) & seg;
                const int at = neg ? 31 - __clz((int)neg) : lane - off - 1;
                const int pp = __shfl_sync(kAll, ps, at & 31);
                int z = ps - (at >= 0 ? pp : 0);
                if (!neg && cont) z += carryZ;
                if ((e.y & kTop) && in) {
                    if (e.w == -1) {
                        rootY += f;
                        rootZ += z;
                    } else {
                        const BinAcc &to = e.w >= 0 ? own : top;
                        const int id = e.w >= 0 ? e.w : -2 - e.w;
                        atomicAdd((unsigned long long *)(to.y + id), (unsigned long long)f);
                        atomicAdd((int *)(to.z + id), z);
                    }
                }
                carryY = __shfl_sync(kAll, y, 31);
                carryZ = __shfl_sync(kAll, z, 31);
            }
        }
        __syncthreads();
    }
}

// losses of one bin, levels from the top down; keys to g.key, histogram in sh
__device__ void loss_bin(const Tab &t, int b, const Scratch1 &g, const BinAcc &own, const BinAcc &top, unsigned *hist)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l0 = t.binlev[b], l1 = t.binlev[b + 1] - 1;
    for (int l = l1 - 1; l >= l0; --l) {
        const int s1 = t.lev[l + 1];
        for (int s = t.lev[l] + warp; s < s1; s += kWarps) {
            const int2 st = t.stream[s];
            int64_t ca = 0, cb = kBig;
            for (int q = st.y - 1; q >= 0; --q) {
                const int slot = (st.x + q) * 32 + lane;
                const int4 e = t.slot[slot];
                const int64_t f = g.f[slot];
                const unsigned starts = __ballot_sync(kAll, (e.y & 31) == 0);
                const unsigned tops = __ballot_sync(kAll, (e.y & kTop) != 0);
                const unsigned after = lane < 31 ? starts >> (lane + 1) : 0u;
                const int rem = after ? __ffs((int)after) - 1 : 31 - lane;    // lanes to the right in this path
                int64_t a = f < 0 ? sat(-f) : 0, bb = f;
                if (e.y & kTop) {
                    int64_t bl = 0, bo = kBig;
                    if (e.w != -1) {
                        const BinAcc &to = e.w >= 0 ? own : top;
                        const int id = e.w >= 0 ? e.w : -2 - e.w;
                        bl = to.lin[id];
                        bo = to.lout[id];
                    }
                    a = sat(a + bl);
                    bb = bb < bo ? bb : bo;
                }
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int64_t a2 = __shfl_down_sync(kAll, a, o), b2 = __shfl_down_sync(kAll, bb, o);
                    if (rem >= o) {
                        a = sat(a + a2);
                        bb = bb < b2 ? bb : b2;
                    }
                }
                if (!((tops >> (lane + rem)) & 1u)) {       // the path goes on in the next tile
                    a = sat(a + ca);
                    bb = bb < cb ? bb : cb;
                }
                if (e.z >= 0) {
                    own.lin[e.z] = a;
                    own.lout[e.z] = bb;
                }
                int code = kKeyPad;
                if (e.x >= 0) {
                    const int k = loss_key(bb > 0 ? bb : a);
                    code = k | (bb > 0 ? 0x8000 : 0);
                    atomicAdd(hist + k, 1u);
                }
                g.key[slot] = (uint16_t)code;
                ca = __shfl_sync(kAll, a, 0);
                cb = __shfl_sync(kAll, bb, 0);
            }
        }
        __syncthreads();
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
    int before = 0, tot = 0;
#pragma unroll
    for (int i = 0; i < kWarps; ++i) {
        before += i < wid ? sh[i] : 0;
        tot += sh[i];
    }
    *total = tot;
    __syncthreads();
    return before + x - v;
}

// what the price search knows: a price with |S| > k and one with |S| <= k
struct Bracket {
    double x0, y0, z0, x1, y1, z1;
};

enum : int { kGo = 0, kStop = 1, kBack = 2, kSlack = 3 };

// what to do after the price lam gave L and |S| = Z: try `nx` (kGo), stop
// here (kStop), or go back to the better end of the bracket `nx` (kBack)
__device__ int next_price(Bracket &b, double k, int evals, int64_t lam, double L, double Z, int64_t &nx_out)
{
    if (Z > k) {
        b.x0 = (double)lam;
        b.y0 = L;
        b.z0 = Z;
    } else {
        b.x1 = (double)lam;
        b.y1 = L;
        b.z1 = Z;
    }
    // L is convex in the price: its minimum lies above the crossing of the
    // two tangents, so L - y bounds what a better price could still give
    const double x = ((b.y0 - (k - b.z0) * b.x0) - (b.y1 - (k - b.z1) * b.x1)) / (b.z0 - b.z1);
    const double y = b.y0 + (k - b.z0) * (x - b.x0);
    const double best = b.y0 < b.y1 ? b.y0 : b.y1;
    if (evals > 1 && (best - y <= 0.03 * x || b.x1 - b.x0 <= 1.0 || evals >= kMaxEvals - 1)) {
        nx_out = (int64_t)(b.y0 < b.y1 ? b.x0 : b.x1);
        return nx_out == lam ? kStop : kBack;
    }
    double nx = x;
    if (b.x0 > 0 && b.z1 > 0 && evals <= 5) {
        // |S| falls roughly like a power of the price: interpolate the logarithms
        const float s = __log2f((float)(b.z0 / k)) / __log2f((float)(b.z0 / b.z1));
        nx = b.x0 * (double)exp2f(__log2f((float)(b.x1 / b.x0)) * s);
    }
    nx = nx < b.x0 + 1.0 ? b.x0 + 1.0 : nx;
    nx = nx > b.x1 - 1.0 ? b.x1 - 1.0 : nx;
    nx_out = (int64_t)nx > 0 ? (int64_t)nx : 1;
    return kGo;
}

struct Rows {                                // undecided rows, in sweep order (last position first)
    int pos[kRowCap], w[kRowCap], skip[kRowCap], info[kRowCap], last[kRowCap];
    int64_t p[kRowCap];
};
constexpr int kPush = 1, kReload = 2, kZeroTop = 4, kFromCur = 8;      // info flags, level << 8

}  // namespace

__global__ void __launch_bounds__(kThreads) k_reduce(Args A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int sh[kWarps];
    __shared__ long long shL[kWarps];
    __shared__ int64_t s_lam;
    __shared__ int s_key, s_flag, s_T;
    __shared__ long long s_val;
    const Tab &t = A.t;
    const int CL = t.CL, cr = CL > 1 ? cluster_rank() : 0;
    const int item = blockIdx.x / CL;
    const int n = t.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t *red = A.w.red + item;
    if (A.item_active && !A.item_active[item]) return;      // uniform over the cluster
    const int32_t kreq = A.item_budget[item];
    if (kreq < 0 || kreq > A.max_budget) {                  // the pruned sweep's kernel reports it
        if (cr == 0 && tid == 0) *red = 0;
        return;
    }
    const int64_t k = kreq < A.total_weight ? kreq : A.total_weight;     // more changes nothing
    Scratch1 g;
    carve(A.w.red_scratch + (size_t)item * A.item_bytes, t.nslots, t.ntop, !A.acc_smem, &g);
    const int words = (n + 31) / 32;
    uint32_t *taken = A.w.taken + (size_t)item * words, *freeb = A.w.undecided + (size_t)item * words;
    const int64_t *P = A.profit + (size_t)item * n;

    // accumulators of this CTA's bin
    BinAcc own, top;
    const int na = t.nacc[cr];
    if (A.acc_smem) {
        own.y = (long long *)smem;
        own.lin = own.y + na;
        own.lout = own.lin + na;
        own.z = (int *)(own.lout + na);
    } else {
        const int s0 = t.binslot[cr];
        own.y = g.accY + s0;
        own.lin = g.accLin + s0;
        own.lout = g.accLout + s0;
        own.z = g.accZ + s0;
    }
    top.y = g.topY;
    top.lin = g.topLin;
    top.lout = g.topLout;
    top.z = g.topZ;

    // ---- gather the profits, clear what is added to
    for (int i = tid; i < na; i += kThreads) {
        own.y[i] = 0;
        own.z[i] = 0;
    }
    if (cr == 0) {
        for (int i = tid; i < t.ntop; i += kThreads) {
            top.y[i] = 0;
            top.z[i] = 0;
        }
        for (int i = tid; i < (int)(sizeof(Scal) / 8); i += kThreads) ((unsigned long long *)g.s)[i] = 0;
        for (int i = tid; i < kBins; i += kThreads) g.hist[i] = 0;
    }
    for (int i = cr * kThreads + tid; i < words; i += CL * kThreads) taken[i] = 0;
    if (k == 0) {                            // nothing fits
        if (cr == 0 && tid == 0) {
            A.best[item] = 0;
            A.w.nkept[item] = 0;
            *red = 1;
        }
        return;
    }
    const bool has_top = t.ntop > 0 || t.binslot[CL] < t.nslots;
    int64_t mx = 0;
    auto gather = [&](int lo, int hi) {
        for (int s = lo + tid; s < hi; s += kThreads) {
            const int x = t.slot[s].x;
            const int64_t p = x >= 0 ? P[A.order ? A.order[x] : x] : 0;
            g.prof[s] = p;
            mx = p > mx ? p : mx;
        }
    };
    const int lo = t.binslot[cr], hi = t.binslot[cr + 1];
    gather(lo, hi);
    if (cr == 0 && has_top) gather(t.binslot[CL], t.nslots);
    if (CL > 1) cluster_sync();              // the scalars are clear
    else __syncthreads();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int64_t y = __shfl_xor_sync(kAll, mx, o);
        mx = y > mx ? y : mx;
    }
    if (lane == 0 && mx > 0) atomicMax(&g.s->maxp, (unsigned long long)mx);
    auto sync_all = [&] {
        if (CL > 1) cluster_sync();
        else __syncthreads();
    };
    sync_all();
    const int64_t maxp = (int64_t) * (volatile unsigned long long *)&g.s->maxp;

    // ---- the price: |S| <= k at price 0 means that the budget does not bind
    int64_t lam = 0, L = 0;
    bool slack = false, give_up = maxp > kBig / (k > A.max_weight ? k : A.max_weight);
    Bracket br;
    br.x1 = (double)maxp;
    br.y1 = (double)maxp * (double)k;
    br.z1 = 0;
    br.x0 = br.y0 = br.z0 = 0;
    // one price: f of every row to g.f, the sums over the roots to slot `ev`
    auto evaluate = [&](int ev) {
        int64_t ry = 0;
        int rz = 0;
        eval_bin(t, cr, g, own, top, lam, ry, rz);
        if (has_top) {
            sync_all();
            if (cr == 0) eval_bin(t, CL, g, top, top, lam, ry, rz);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ry += __shfl_xor_sync(kAll, ry, o);
            rz += __shfl_xor_sync(kAll, rz, o);
        }
        if (lane == 0) {
            shL[warp] = ry;
            sh[warp] = rz;
        }
        __syncthreads();
        if (tid == 0) {
            unsigned long long a = 0, z = 0;
            for (int i = 0; i < kWarps; ++i) {
                a += (unsigned long long)shL[i];
                z += (unsigned long long)sh[i];
            }
            if (a) atomicAdd(&g.s->sumL[ev], a);
            if (z) atomicAdd(&g.s->sumZ[ev], z);
        }
        sync_all();
    };
    for (int ev = 0; !give_up; ++ev) {
        evaluate(ev);
        if (tid == 0) {
            const int64_t sl = (int64_t) * (volatile unsigned long long *)&g.s->sumL[ev] + lam * k;
            const int64_t sz = (int64_t) * (volatile unsigned long long *)&g.s->sumZ[ev];
            int64_t nx = 0;
            s_flag = lam == 0 && sz <= k ? kSlack : next_price(br, (double)k, ev + 1, lam, (double)sl, (double)sz, nx);
            s_val = sl;
            s_lam = nx;
        }
        __syncthreads();
        L = s_val;
        const int todo = s_flag;
        if (todo == kGo || todo == kBack) lam = s_lam;
        __syncthreads();
        if (todo == kGo) continue;           // (never at the last but one slot: next_price stops there)
        slack = todo == kSlack;
        if (todo == kBack) {
            evaluate(kMaxEvals - 1);
            L = (int64_t) * (volatile unsigned long long *)&g.s->sumL[kMaxEvals - 1] + lam * k;
        }
        break;
    }

    // ---- losses and their histogram
    unsigned *hist = (unsigned *)(smem + (A.acc_smem ? up16((size_t)na * 28) : 0));
    if (!give_up) {
        for (int i = tid; i < kBins; i += kThreads) hist[i] = 0;
        __syncthreads();
        if (has_top) {
            if (cr == 0) loss_bin(t, CL, g, top, top, hist);
            sync_all();
        }
        loss_bin(t, cr, g, own, top, hist);
        for (int i = tid; i < kBins; i += kThreads)
            if (hist[i]) atomicAdd(g.hist + i, hist[i]);
        sync_all();
    }
    // largest key whose rows, and all below, are at most `rows` (but at least key 0)
    auto key_of_rank = [&](int rows) {
        constexpr int V = kBins / kThreads;
        int c[V], sum = 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            c[v] = (int)*(volatile unsigned *)(g.hist + tid * V + v);
            sum += c[v];
        }
        int tot;
        int ex = block_scan(sum, &tot, sh);
        if (tid == 0) s_key = 0;
        __syncthreads();
        int last = -1;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            ex += c[v];
            if (ex <= rows) last = tid * V + v;
        }
        if (last > 0) atomicMax(&s_key, last);
        __syncthreads();
        const int r = s_key;
        __syncthreads();
        return r;
    };
    auto rows_up_to = [&](int key) {
        constexpr int V = kBins / kThreads;
        int sum = 0;
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (tid * V + v <= key) sum += (int)*(volatile unsigned *)(g.hist + tid * V + v);
        int tot;
        block_scan(sum, &tot, sh);
        return tot;
    };

    int verdict = 3, key = 0, pass = 0;
    bool sure = false;           // the key comes from a V: no row above it is undecided
    if (!give_up) {
        key = slack ? -1 : key_of_rank(kFirstRows);
        for (pass = 0; pass < kPasses; ++pass) {
            const int T = key < 0 ? 0 : rows_up_to(key);
            const bool big = T > kRowCap;                         // the same in every CTA
            if (big && !sure) {
                verdict = 3;
                break;
            }
            // ---- decided rows: value and weight of those in; the others' positions
            for (int i = cr * kThreads + tid; i < words; i += CL * kThreads) freeb[i] = 0;
            sync_all();
            unsigned long long vf = 0, wf = 0;
            auto classify = [&](int a, int b) {
                for (int s = a + tid; s < b; s += kThreads) {
                    const int c = g.key[s];
                    if (c == kKeyPad) continue;
                    const int kk = c & 0x7fff;
                    if (kk <= key) {
                        const int x = t.slot[s].x;
                        atomicOr(freeb + (x >> 5), 1u << (x & 31));
                    } else if (c & 0x8000) {
                        vf += (unsigned long long)g.prof[s];
                        wf += (unsigned)(t.slot[s].y >> kWeightShift);
                    }
                }
            };
            classify(lo, hi);
            if (cr == 0 && has_top) classify(t.binslot[CL], t.nslots);
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
                unsigned char *pool = smem + sizeof(Rows);
                const int64_t vfix = (int64_t) * (volatile unsigned long long *)&g.s->vfix[pass];
                const int64_t wfix = (int64_t) * (volatile unsigned long long *)&g.s->wfix[pass];
                const int64_t kleft = k - wfix;
                int out = 0, okey = 0;       // 1 solved, 2 again with okey (5: which is sure), 3 not reducible
                if (kleft < 0) {                        // too few rows undecided: take more by rank
                    out = 2;
                    okey = key_of_rank(pass == 0 ? 2 * kFirstRows : kRowCap);
                    if (okey <= key) out = 3;
                } else {
                    // rows in sweep order from the bitmap
                    const int per = (words + kThreads - 1) / kThreads;
                    const int w0 = min(words, tid * per), w1 = min(words, w0 + per);
                    int c = 0;
                    for (int i = w0; i < w1; ++i) c += __popc(*(volatile uint32_t *)(freeb + i));
                    int tot;
                    int ex = block_scan(c, &tot, sh);
                    for (int i = w0; i < w1; ++i) {
                        uint32_t m = *(volatile uint32_t *)(freeb + i);
                        while (m) {
                            const int x = i * 32 + __ffs((int)m) - 1;
                            m &= m - 1;
                            R.pos[T - 1 - ex] = x;
                            ++ex;
                        }
                    }
                    __syncthreads();
                    int64_t wsum = 0;
                    for (int r = tid; r < T; r += kThreads) {
                        const int x = R.pos[r];
                        R.p[r] = P[A.order ? A.order[x] : x];
                        R.w[r] = A.wpre[x];
                        wsum += R.w[r];
                        R.last[r] = -1;
                        // the first undecided row at or after next(x), -1: none
                        const int nx = A.next[x];
                        int a = 0, b = r;               // rows 0..a-1 have pos >= nx
                        while (a < b) {
                            const int mid = (a + b) >> 1;
                            if (R.pos[mid] >= nx) a = mid + 1;
                            else b = mid;
                        }
                        R.skip[r] = a - 1;
                    }
                    wsum = wsum < (1 << 30) ? wsum : (1 << 30);
                    int wtot;
                    block_scan((int)min(wsum, (int64_t)(1 << 20)), &wtot, sh);   // (2^20 is above every column cap)
                    const int kc = (int)(kleft < wtot ? kleft : wtot);
                    // stack plan, as the pruned sweep's: a row read through the
                    // stack is pushed when computed and popped after its last reader
                    for (int r = tid; r < T; r += kThreads) {
                        const int sk = R.skip[r];
                        if (sk >= 0 && sk != r - 1) atomicMax(&R.last[sk], r);
                    }
                    __syncthreads();
                    int depth = 0, deepest = 0;
                    for (int base = 0; base < T; base += kThreads) {
                        const int r = base + tid;
                        bool pop = false, push = false;
                        if (r < T) {
                            const int sk = R.skip[r];
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
                            } else if (pop && dd > 0) {
                                fl = kReload;
                                lvl = dd - 1;
                            } else if (pop) {
                                fl = kZeroTop;
                            }
                            const int sk = R.skip[r];
                            if (sk >= 0 && sk == r - 1 && R.last[r - 1] < 0) fl |= kFromCur;
                            R.info[r] = fl | (lvl << 8);
                            deepest = max(deepest, push ? dd + 1 : 0);
                        }
                        depth += dt;
                    }
                    if (tid == 0) s_T = 0;
                    __syncthreads();
                    if (deepest) atomicMax(&s_T, deepest);
                    __syncthreads();
                    const int levels = s_T;
                    const int nw = (kc + 31) / 32;                   // warps that hold columns
                    const size_t need = (size_t)T * nw * 4 + (size_t)(levels + 2) * nw * 32 * 8;
                    if (kc > kColCap || need > (size_t)kPool) {
                        out = 3;
                    } else {
                        // one column per thread (two above 512); column j = c + 1
                        int64_t *rowb = (int64_t *)pool;             // [2][nw * 32]
                        int64_t *stk = rowb + 2 * nw * 32;           // [levels][nw * 32]
                        uint32_t *bits = (uint32_t *)(stk + (size_t)levels * nw * 32);   // [T][nw]
                        const int cols = nw * 32;
                        const int act = min(nw, kWarps);             // warps in the loop
                        if (tid == 0) s_val = 0;
                        for (int c2 = tid; c2 < cols; c2 += kThreads) rowb[c2] = 0;
                        __syncthreads();
                        if (warp < act) {
                            int64_t cur[2] = {0, 0}, tp[2] = {0, 0};
                            const bool two = tid + kThreads < cols;  // uniform over the warp
                            for (int r = 0; r < T; ++r) {
                                const int64_t p = R.p[r];
                                const int w = R.w[r], info = R.info[r];
                                const int64_t *prev = rowb + (r & 1) * cols;
                                int64_t *outr = rowb + ((r + 1) & 1) * cols;
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    if (h == 1 && !two) break;
                                    const int j = tid + h * kThreads + 1;
                                    const int64_t sk = (info & kFromCur) ? cur[h] : tp[h];
                                    bool take = false;
                                    int64_t v = sk;
                                    if (j >= w) {
                                        const int64_t tv = p + (j > w ? prev[j - w - 1] : 0);
                                        take = tv > sk;
                                        v = take ? tv : sk;
                                    }
                                    cur[h] = v;
                                    outr[j - 1] = v;
                                    const unsigned m = __ballot_sync(kAll, take);
                                    if (lane == 0) bits[r * nw + ((j - 1) >> 5)] = m;
                                    const int lvl = info >> 8;
                                    if (info & kPush) {
                                        stk[lvl * cols + j - 1] = v;
                                        tp[h] = v;
                                    } else if (info & kReload) {
                                        tp[h] = stk[lvl * cols + j - 1];
                                    } else if (info & kZeroTop) {
                                        tp[h] = 0;
                                    }
                                }
                                if (act == 1) __syncwarp();
                                else asm volatile("bar.sync 1, %0;" ::"r"(act * 32) : "memory");
                            }
                            if (kc > 0) {
                                if (tid == (kc - 1) % kThreads) s_val = cur[(kc - 1) / kThreads];
                            }
                        }
                        __syncthreads();
                        const int64_t V = vfix + s_val;
                        const int need_key = slack ? -1 : loss_key(L - V);
                        if (slack || need_key <= key) {
                            out = 1;
                            // walk the decisions
                            if (tid == 0) {
                                int r = T - 1, j = kc;
                                while (r >= 0 && j > 0) {
                                    if ((bits[r * nw + ((j - 1) >> 5)] >> ((j - 1) & 31)) & 1u) {
                                        const int x = R.pos[r];
                                        atomicOr(taken + (x >> 5), 1u << (x & 31));
                                        j -= R.w[r];
                                        --r;
                                    } else {
                                        r = R.skip[r];
                                    }
                                }
                                A.best[item] = V;
                                A.w.nkept[item] = T;
                                if (A.rows_kept) atomicAdd(A.rows_kept, (unsigned long long)T);
                            }
                        } else {
                            out = 5;
                            okey = need_key;
                        }
                    }
                }
                if (tid == 0) {
                    g.s->key[pass] = okey;
                    g.s->verdict[pass] = out;
                }
            }
            sync_all();
            verdict = *(volatile int *)&g.s->verdict[pass];
            if (verdict != 2 && verdict != 5) break;
            sure = verdict == 5;
            key = *(volatile int *)&g.s->key[pass];
        }
    }
    const int state = verdict == 1 ? 1 : verdict == 4 ? 2 : 0;
    // ---- the decided "in" rows join the set
    if (state) {
        auto mark = [&](int a, int b) {
            for (int s = a + tid; s < b; s += kThreads) {
                const int c = g.key[s];
                if (c == kKeyPad || !(c & 0x8000) || (c & 0x7fff) <= key) continue;
                const int x = t.slot[s].x;
                atomicOr(taken + (x >> 5), 1u << (x & 31));
            }
        };
        mark(lo, hi);
        if (cr == 0 && has_top) mark(t.binslot[CL], t.nslots);
    }
    if (cr == 0 && tid == 0) {
        *red = state;
        if (state == 2) {
            A.w.left[item] = (int32_t)(k - (int64_t) * (volatile unsigned long long *)&g.s->wfix[pass]);
            A.w.base[item] = (int64_t) * (volatile unsigned long long *)&g.s->vfix[pass];
        }
    }
}

// ---------------------------------------------------------------------------
// host: the layout (see the top of the file), one device block per instance
// ---------------------------------------------------------------------------
// CTAs of an item's cluster: one per 6,144 rows (12 tiles per warp), at most 8
static int cluster_of(int n) { return n <= 6144 ? 1 : n <= 12288 ? 2 : n <= 24576 ? 4 : 8; }

bool build_reduce_tables(int32_t n, const std::vector<int32_t> &par, const std::vector<int32_t> &next,
                         const std::vector<int32_t> &wpre, int64_t total_weight, int32_t max_weight,
                         ReduceTables *out)
{
    ReduceTables &R = *out;
    R = ReduceTables();
    if (n < kReduceMinRows || max_weight > kMaxWeight || total_weight >= ((int64_t)1 << 30)) return false;
    const int CL = cluster_of(n);
    const int limit = CL == 1 ? n : std::max(64, n / (4 * CL));      // rows of a subtree that stays in one bin
    auto is_top = [&](int i) { return next[i] - i > limit; };
    // bins: subtrees below the limit, each to the emptiest bin
    std::vector<int32_t> bin(n), heavy(n, -1), best(n, 0), level(n, 0), acc(n, -1);
    std::vector<int64_t> load(CL, 0);
    for (int32_t i = 0; i < n; ++i) {
        const int p = par[i];
        if (is_top(i)) bin[i] = CL;
        else if (p >= 0 && bin[p] != CL) bin[i] = bin[p];
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
    R.nacc.assign(CL + 1, 0);
    int maxlev = 0;
    for (int32_t i = n - 1; i >= 0; --i) {
        const int p = par[i];
        maxlev = std::max(maxlev, level[i]);
        if (p < 0) continue;
        if (heavy[p] == i) level[p] = std::max(level[p], level[i]);
        else if (bin[p] == bin[i]) level[p] = std::max(level[p], level[i] + 1);
        if (heavy[p] != i && acc[p] < 0) acc[p] = R.nacc[bin[p]]++;
    }
    // path tops grouped by (bin, level)
    const int nl = maxlev + 1;
    std::vector<int32_t> start((size_t)(CL + 1) * nl + 1, 0), rows((size_t)(CL + 1) * nl, 0), tops, len(n, 0);
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
    R.slot.reserve((size_t)n + 32 * 64);
    std::vector<int32_t> path;
    for (int b = 0; b <= CL; ++b) {
        R.binslot.push_back((int32_t)R.slot.size());
        R.binlev.push_back((int32_t)R.lev.size());
        int levels = nl;
        while (levels > 0 && rows[(size_t)b * nl + levels - 1] == 0) --levels;
        for (int l = 0; l < levels; ++l) {
            const size_t q = (size_t)b * nl + l;
            R.lev.push_back((int32_t)R.stream.size());
            // streams of about equal length, one per warp of the CTA when there are rows for all
            const int ns = std::max(1, std::min(kWarps, (rows[q] + 63) / 64));
            const int want = (rows[q] + ns - 1) / ns;
            int in_stream = 0, tile0 = (int)(R.slot.size() / 32);
            auto close = [&] {
                if (in_stream == 0) return;
                while (R.slot.size() % 32) R.slot.push_back({-1, 0, -1, -1});
                const int tile1 = (int)(R.slot.size() / 32);
                R.stream.push_back({tile0, tile1 - tile0});
                tile0 = tile1;
                in_stream = 0;
            };
            for (int x = start[q]; x < start[q + 1]; ++x) {
                const int topn = tops[x];
                path.clear();
                for (int v = topn; v >= 0; v = heavy[v]) path.push_back(v);
                int first = (int)R.slot.size();            // the path's first slot
                for (int y = (int)path.size() - 1; y >= 0; --y) {
                    const int v = path[y];
                    const int s = (int)R.slot.size(), t0 = s & ~31;
                    int code = (s - std::max(first, t0)) | (first < t0 ? kCont : 0) | (v == topn ? kTop : 0) |
                               (wpre[v] << kWeightShift);
                    int pr = -1;
                    if (v == topn && par[v] >= 0)
                        pr = bin[par[v]] == bin[v] ? acc[par[v]] : -2 - acc[par[v]];
                    R.slot.push_back({v, code, acc[v], pr});
                }
                in_stream += (int)path.size();
                if (in_stream >= want) close();
            }
            close();
        }
        R.lev.push_back((int32_t)R.stream.size());
    }
    R.binslot.push_back((int32_t)R.slot.size());
    R.binlev.push_back((int32_t)R.lev.size());
    R.CL = CL;
    return true;
}

static size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

// device block: slots | streams | levels | binlev | binslot | nacc
size_t reduce_tables_bytes(const ReduceTables &R)
{
    return al(R.slot.size() * 16) + al(R.stream.size() * 8) + al(R.lev.size() * 4) + al(R.binlev.size() * 4) +
           al(R.binslot.size() * 4) + al(R.nacc.size() * 4);
}

void reduce_tables_pack(const ReduceTables &R, char *dst)
{
    auto put = [&](const void *src, size_t bytes) {
        std::memcpy(dst, src, bytes);
        dst += al(bytes);
    };
    put(R.slot.data(), R.slot.size() * 16);
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
    t.CL = r.CL;
    t.nslots = r.nslots;
    t.ntop = r.ntop;
    t.slot = (const int4 *)take((size_t)r.nslots * 16);
    t.stream = (const int2 *)take((size_t)r.nstreams * 8);
    t.lev = (const int *)take((size_t)r.nlev * 4);
    t.binlev = (const int *)take((size_t)(r.CL + 2) * 4);
    t.binslot = (const int *)take((size_t)(r.CL + 2) * 4);
    t.nacc = (const int *)take((size_t)(r.CL + 1) * 4);
    return t;
}

ReduceShape reduce_shape(const ReduceTables &R)
{
    ReduceShape s;
    s.CL = R.CL;
    s.nslots = (int)R.slot.size();
    s.nstreams = (int)R.stream.size();
    s.nlev = (int)R.lev.size();
    s.ntop = R.nacc[R.CL];
    s.max_acc = *std::max_element(R.nacc.begin(), R.nacc.end() - 1);
    // two CTAs fit on one SM: at most 104 KB each
    s.acc_smem = up16((size_t)s.max_acc * 28) + kBins * 4 <= (size_t)(104 << 10);
    return s;
}

// scratch of one item in the DP workspace, 0 when the instance has no reduction
size_t reduce_item_bytes(const pp_instance *inst)
{
    if (!inst->red.CL) return 0;
    return al(carve(nullptr, inst->red.nslots, inst->red.ntop, !inst->red.acc_smem, nullptr));
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
    a.acc_smem = r.acc_smem;
    a.total_weight = inst->total_weight;
    a.max_weight = inst->max_weight;
    const size_t scan = (r.acc_smem ? up16((size_t)r.max_acc * 28) : 0) + kBins * 4;
    const size_t smem = std::max(scan, sizeof(Rows) + kPool);
    PP_CUDA(cudaFuncSetAttribute(k_reduce, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(r.CL * batch);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = r.CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    PP_CUDA(cudaLaunchKernelEx(&cfg, k_reduce, a));
    return PP_OK;
}

}  // namespace pp
