// The pruned sweep's rows (Eq. 9), found by one cluster of CTAs per item: run
// by the exact reduction's kernel for the items that it leaves, and by a kernel
// of its own where there is no reduction.
#pragma once
#include "pp_internal.cuh"

namespace pp {

__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_nctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

// ===========================================================================
// Pruned sweep (one cluster of CTAs per item).  A strict descendant set with
// no positive profit is never worth taking: for a parent x whose strict
// descendants all have p <= 0, D[x+1][.] = D[next(x)][.] (selecting nothing
// below x is optimal) and every decision bit below x is "skip".  So the rows
// strictly below x can be removed from the sweep: row x then sees D[next(x)]
// as its row i+1, which is the same values, and no kept row's value or bit
// changes.  With `cnt` the prefix counts of positive profits in preorder, x
// has a positive strict descendant iff cnt[next(x)] - cnt[x + 1] > 0, and row
// i is kept iff it is a root or its parent has one.  A kept row i that is
// itself an identity (p_i <= 0 and no positive strict descendant: D[i] =
// D[next(i)], all bits "skip") is dropped as well.  For an item that the
// reduction has cut down (`ud`: its undecided rows) only those of them are kept:
// decided rows inside the optimal set are closed upwards and those outside it
// downwards, so the undecided rows in preorder form a forest of their own,
// with the same subtree ends, in which a row without a positive profit at or
// below it is never worth taking either (a caterpillar of 1,600 chunks with a
// tenth of the profits: 1,568 undecided rows, 883 of them kept).
// Kept rows are listed in sweep order (decreasing i); every position records
// the first kept row at or after it in preorder, so a skip to a dropped row
// lands where the all-"skip" walk through it would.
// ===========================================================================
__device__ __forceinline__ int block_exclusive_scan(int v, int *total, int *sh)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int w = lane < nw ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < nw) sh[lane] = w;           // inclusive warp totals
    }
    __syncthreads();
    const int before = wid > 0 ? sh[wid - 1] : 0;
    *total = sh[nw - 1];
    __syncthreads();                           // sh is reused by the next scan
    return before + x - v;
}

// Exclusive scan over the CTAs of the cluster of one value per CTA (`v`, the
// same in every thread of the CTA).  Returns this CTA's offset and the cluster
// total.  The cluster barriers also order the global writes made before the
// call against the reads of other CTAs after it.
__device__ __forceinline__ int ld_dsmem_s32(uint32_t addr)
{
    int v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ int cluster_exclusive_scan(int v, int *total, int *slot, int *bcast)
{
    const int CLn = (int)cluster_nctarank(), cr = (int)cluster_ctarank();
    if (threadIdx.x == 0) *slot = v;
    cluster_sync_all();
    if (threadIdx.x == 0) {
        int ex = 0, tot = 0;
        for (int c = 0; c < CLn; ++c) {
            const int x = ld_dsmem_s32(map_to_rank(smem_addr(slot), (uint32_t)c));
            ex += c < cr ? x : 0;
            tot += x;
        }
        bcast[0] = ex;
        bcast[1] = tot;
    }
    cluster_sync_all();           // every slot read: they may be written again
    *total = bcast[1];
    return bcast[0];
}

// One cluster of CL CTAs per item: every pass splits its index range into CL
// contiguous slices, each CTA walks its slice in tiles of T*V elements (V per
// thread, one block scan per tile), and the slices are joined by a scan over
// the cluster's CTAs.
// (as many CTAs as the cluster has, 1024 threads each; `order`: profits are by
// node id; `ud`: bitmap of the only rows to keep, of those that pruning keeps)
__device__ __forceinline__ void prune_item(int32_t n, int item, const int64_t *__restrict__ profit,
                                           const int32_t *__restrict__ order, const int32_t *__restrict__ next,
                                           const int2 *__restrict__ pspan, const int32_t *__restrict__ wpre,
                                           const DpWork &w, const uint32_t *ud, int prune, int stack_depth,
                                           int32_t *__restrict__ status, unsigned long long *__restrict__ rows_kept)
{
    constexpr int V = 4;
    __shared__ int sh[32];
    __shared__ int slot, bcast[2];
    const int CL = (int)cluster_nctarank(), cr = (int)cluster_ctarank();
    const int64_t *Pp = profit + (size_t)item * n;
    int32_t *cnt = w.cnt + (size_t)item * (n + 1);
    int32_t *rl = w.rowlist + (size_t)item * n;
    int32_t *kx = w.kidx + (size_t)item * n;
    const int T = blockDim.x, t = threadIdx.x, tile = T * V;
    auto pval = [&](int i) { return Pp[order ? order[i] : i]; };
    auto slice = [&](int len, int &lo, int &hi) {
        const int per = (len + CL - 1) / CL;
        lo = min(len, cr * per);
        hi = min(len, lo + per);
    };
    int lo, hi, total;

    // prefix counts of positive profits, preorder
    slice(n, lo, hi);
    int mine = 0;
    for (int i = lo + t; i < hi; i += T) mine += pval(i) > 0;
    block_exclusive_scan(mine, &total, sh);
    int carry = cluster_exclusive_scan(total, &total, &slot, bcast);
    const int npos = total;
    for (int base = lo; base < hi; base += tile) {
        int f[V], c = 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int i = base + t * V + v;
            f[v] = i < hi && pval(i) > 0;
            c += f[v];
        }
        int tt;
        int ex = block_exclusive_scan(c, &tt, sh) + carry;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int i = base + t * V + v;
            if (i < hi) {
                cnt[i] = ex;
                ex += f[v];
            }
        }
        carry += tt;
    }
    if (cr == 0 && t == 0) cnt[n] = npos;
    cluster_sync_all();                                   // cnt complete for every CTA

    // kept rows in sweep order r = n - 1 - i, their kept index, their total weight
    auto keep = [&](int r) -> bool {
        if (!prune) return true;
        const int i = n - 1 - r;
        if (ud && !((ud[i >> 5] >> (i & 31)) & 1u)) return false;
        const int2 sp = pspan[i];
        if (!(sp.x < 0 || cnt[sp.y] - cnt[sp.x] > 0)) return false;
        // an identity row (p <= 0 and no positive strict descendant, so D[i] =
        // D[next(i)] and every bit is "skip") is dropped too: a skip to it
        // lands on the first kept row after it, which holds the same values
        return cnt[next[i]] - cnt[i + 1] != 0 || pval(i) > 0;
    };
    slice(n, lo, hi);
    int kmine = 0;
    for (int r = lo + t; r < hi; r += T) kmine += keep(r);
    block_exclusive_scan(kmine, &total, sh);
    int kcarry = cluster_exclusive_scan(total, &total, &slot, bcast);
    const int nk = total;
    for (int base = lo; base < hi; base += tile) {
        bool kp[V];
        int kc = 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int r = base + t * V + v;
            kp[v] = r < hi && keep(r);
            kc += kp[v];
        }
        int tt;
        int ex = block_exclusive_scan(kc, &tt, sh) + kcarry;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int r = base + t * V + v;
            if (r < hi) {
                const int i = n - 1 - r;
                if (kp[v]) {
                    rl[ex] = i;
                    kx[i] = ex++;
                } else {
                    kx[i] = ex - 1;         // the first kept row at or after position i (-1: none)
                }
            }
        }
        kcarry += tt;
    }
    if (cr == 0 && t == 0) {
        w.nkept[item] = nk;
        if (rows_kept) atomicAdd(rows_kept, (unsigned long long)nk);
    }
    cluster_sync_all();                                   // rl and kx complete

    // per kept row: skip target, the DP's row stream (profit, metadata) and
    // the suffix weights of the traceback
    int32_t *sk = w.skip + (size_t)item * n;
    int32_t *ws = w.wsuf + (size_t)item * (n + 1);
    int64_t *rp = w.rowp + (size_t)item * n;
    int32_t *rm = w.rowm + (size_t)item * n;
    slice(nk, lo, hi);
    int wmine = 0;
    for (int q = lo + t; q < hi; q += T) wmine += wpre[rl[q]];
    block_exclusive_scan(wmine, &total, sh);
    int wtot;                                             // weight of all kept rows
    int wcarry = cluster_exclusive_scan(total, &wtot, &slot, bcast);
    for (int base = lo; base < hi; base += tile) {
        int wq[V], wl = 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int q = base + t * V + v;
            wq[v] = 0;
            if (q < hi) {
                const int i = rl[q];
                const int nx = next[i];
                sk[q] = nx < n ? kx[nx] : -1;
                wq[v] = wpre[i];
                rp[q] = pval(i);
                cnt[q] = -1;                    // cnt (done with) becomes last_top_reader
            }
            wl += wq[v];
        }
        int tt;
        int ex = block_exclusive_scan(wl, &tt, sh) + wcarry;   // weight of kept rows before q
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int q = base + t * V + v;
            if (q < hi) {
                ws[q] = wtot - ex;                                 // weight of kept rows q..nk-1
                ex += wq[v];
            }
        }
        wcarry += tt;
    }
    if (cr == 0 && t == 0) ws[nk] = 0;

    // Skip-row stack plan over the kept rows (the host's plan is for the
    // whole tree; after pruning many of its pushes have no reader left).  Kept row q reads row sk[q]: the row just
    // computed when sk[q] = q - 1, else the stack top (the zero row when the
    // stack is empty, which is the case whenever sk[q] = -1).  A row read
    // through the stack is pushed when computed and popped after its last
    // such reader; the rows pushed in between are popped before it, so
    // every read is of the top.
    int32_t *lr_ = cnt;                                   // last_top_reader[target]
    cluster_sync_all();                                   // sk and the -1s complete
    for (int q = lo + t; q < hi; q += T) {
        const int s = sk[q];
        if (s >= 0 && s != q - 1) atomicMax(lr_ + s, q);
    }
    cluster_sync_all();                                   // last readers complete
    auto delta = [&](int q, bool &pop, bool &push) {
        const int s = sk[q];
        pop = s >= 0 && s != q - 1 && lr_[s] == q;
        push = lr_[q] >= 0;
        return (int)push - (int)pop;
    };
    int dmine = 0;
    for (int q = lo + t; q < hi; q += T) {
        bool a, b;
        dmine += delta(q, a, b);
    }
    block_exclusive_scan(dmine, &total, sh);
    int dcarry = cluster_exclusive_scan(total, &total, &slot, bcast);
    for (int base = lo; base < hi; base += tile) {
        int dq[V], dl = 0;
        bool pq[V], uq[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int q = base + t * V + v;
            dq[v] = 0;
            pq[v] = uq[v] = false;
            if (q < hi) dq[v] = delta(q, pq[v], uq[v]);
            dl += dq[v];
        }
        int tt;
        int ex = block_exclusive_scan(dl, &tt, sh) + dcarry;   // stack depth before row q
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int q = base + t * V + v;
            if (q < hi) {
                const int s = sk[q];
                const int d = ex - (int)pq[v];            // after the pop
                int flags = 0, lvl = 0;
                if (uq[v]) {
                    flags = kWavePush;
                    lvl = d;
                } else if (pq[v] && d > 0) {
                    flags = kWaveReload;                  // the level below becomes the top
                    lvl = d - 1;
                } else if (pq[v]) {
                    flags = kWaveZeroTop;                 // the stack emptied: top = zero row
                }
                if ((flags & (kWavePush | kWaveReload)) && lvl >= stack_depth) {
                    // cannot happen (the plan of an ancestor-closed sub-forest is
                    // never deeper than the whole tree's): report, stay in bounds
                    atomicExch(status, (int32_t)PP_EBOUNDS);
                    flags = 0;
                    lvl = 0;
                }
                const int wq = wpre[rl[q]];
                // a row whose skip row is the row just computed reads it from the
                // stack top when that row was pushed (the push made it the top):
                // the same values, and sub-blocks without "cur" rows need no
                // per-row choice of skip source
                const bool cur = s >= 0 && s == q - 1 && lr_[q - 1] < 0;
                rm[q] = wave_pack(wq > 8 ? 8 : wq, cur ? kWaveCur : kWaveTop, flags, lvl);
                ex += dq[v];
            }
        }
        dcarry += tt;
    }
}

}  // namespace pp
