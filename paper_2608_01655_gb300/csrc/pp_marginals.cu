// Per-worker exact node marginals (Prop. 1) and the planner objective.
//   requester-side (Eq. 10):   p_h(b) = a_h(b) + 1{no holder l != h} Delta(b)
//   source-dependent (Eq. 7):  p_h(b) = sum_m [g_h,m(b) - max_{l in H_b \ h} g_l,m(b)]_+
// where g_h,m(b) = Lambda_m(b) q_{m<-h}(b) (Eq. 5) is precomputed per instance
// and the max over an empty holder set is 0.  Objectives: F (Eq. 4) and
// F_pair (Eq. 6).  All arithmetic is exact int64.
#include "pp_internal.cuh"

namespace pp {

__device__ __forceinline__ int64_t warp_sum64(int64_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// block-wide sum added atomically into *dst (integer addition is exact, so the
// result does not depend on the order of the atomics)
__device__ __forceinline__ void block_add64(int64_t v, int64_t *dst)
{
    __shared__ int64_t part[32];
    v = warp_sum64(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) part[wid] = v;
    __syncthreads();
    if (wid == 0) {
        int nw = (blockDim.x + 31) >> 5;
        int64_t x = lane < nw ? part[lane] : 0;
        x = warp_sum64(x);
        if (lane == 0 && x != 0) atomicAdd((unsigned long long *)dst, (unsigned long long)x);
    }
}

// Values of kReq requesters at once, so that a thread has that many loads in
// flight: one requester at a time, a thread waited for memory W times (1 + |H|)
// (20,000 chunks, 16 workers, 8 items: 58 and 61 us for marginals and objective).
constexpr int kReq = 8;
// g_{l,m}(i) of the requesters m0 .. m0 + kReq - 1 (0 past the last)
__device__ __forceinline__ void load_req(int32_t n, int32_t W, int32_t l, int32_t m0, int32_t i,
                                         const int64_t *__restrict__ g, int64_t (&x)[kReq])
{
    const int64_t *q = g + ((size_t)l * W + m0) * n + i;
#pragma unroll
    for (int u = 0; u < kReq; ++u) x[u] = m0 + u < W ? __ldg(q + (size_t)u * n) : 0;
}
// their largest over the holders, 0 without one
__device__ __forceinline__ void best_of(int32_t n, int32_t W, uint32_t holders, int32_t m0, int32_t i,
                                        const int64_t *__restrict__ g, int64_t (&v)[kReq])
{
#pragma unroll
    for (int u = 0; u < kReq; ++u) v[u] = 0;
    for (uint32_t o = holders; o; o &= o - 1) {
        int64_t x[kReq];
        load_req(n, W, __ffs((int)o) - 1, m0, i, g, x);
#pragma unroll
        for (int u = 0; u < kReq; ++u) v[u] = x[u] > v[u] ? x[u] : v[u];
    }
}

// Marginal of one chunk at preorder position i for worker h; `others` is the
// holder mask without bit h.
template <int MODE>
__device__ __forceinline__ int64_t marginal_at(int32_t n, int32_t W, int32_t h, int32_t i,
                                               uint32_t others, const int64_t *__restrict__ a,
                                               const int64_t *__restrict__ delta,
                                               const int64_t *__restrict__ g)
{
    if (MODE == 0) {
        int64_t p = a[(size_t)h * n + i];
        if (others == 0) p += delta[i];
        return p;
    } else {
        int64_t p = 0;
        for (int32_t m0 = 0; m0 < W; m0 += kReq) {
            int64_t mine[kReq], v[kReq];
            load_req(n, W, h, m0, i, g, mine);
            best_of(n, W, others, m0, i, g, v);
#pragma unroll
            for (int u = 0; u < kReq; ++u) p += mine[u] > v[u] ? mine[u] - v[u] : 0;
        }
        return p;
    }
}

// grid: (blocks over positions, batch).  BYNODE: masks / profits indexed by
// node id (ABI); otherwise by preorder position (planner).  oldsum (optional)
// is added the sum of p_h over the chunks worker h currently holds, which equals
// G(T) - G(T_-h, {}) by Prop. 1 and is the refinement's acceptance threshold.
template <bool BYNODE, int MODE>
__global__ void __launch_bounds__(256) k_marginals(int32_t n, int32_t W,
                                                    const int32_t *__restrict__ worker,
                                                    const uint32_t *__restrict__ mask,
                                                    const int32_t *__restrict__ order,
                                                    const int64_t *__restrict__ a,
                                                    const int64_t *__restrict__ delta,
                                                    const int64_t *__restrict__ g,
                                                    const int32_t *__restrict__ item_active,
                                                    int64_t *__restrict__ profit,
                                                    int64_t *__restrict__ oldsum,
                                                    int32_t *__restrict__ status)
{
    chain_wait();
    chain_release();
    const int item = blockIdx.y;
    if (item_active && !item_active[item]) return;
    const int32_t h = worker[item];
    const uint32_t *M = mask + (size_t)item * n;
    int64_t *P = profit + (size_t)item * n;
    if (h < 0 || h >= W) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicExch(status, (int32_t)PP_EBOUNDS);
        for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
            P[i] = 0;
        return;
    }
    const uint32_t hb = 1u << h;
    int64_t held = 0;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int32_t idx = BYNODE ? order[i] : i;
        const uint32_t mk = M[idx];
        const int64_t p = marginal_at<MODE>(n, W, h, i, mk & ~hb, a, delta, g);
        P[idx] = p;
        if (mk & hb) held += p;
    }
    if (oldsum) block_add64(held, oldsum + item);
}

template <bool BYNODE, int MODE>
static cudaError_t marg_launch(pp_instance *inst, dim3 grid, const int32_t *worker, const uint32_t *mask,
                               const int32_t *item_active, int64_t *profit, int64_t *oldsum, cudaStream_t st)
{
    return launch_chained(k_marginals<BYNODE, MODE>, grid, dim3(256), 0, st, 1, inst->n, inst->W, worker, mask,
                          inst->d_order, inst->d_a, inst->d_delta, inst->d_g, item_active, profit, oldsum,
                          inst->d_status);
}

pp_status launch_marginals(pp_instance *inst, int batch, const int32_t *worker,
                           const uint32_t *mask, bool by_node, const int32_t *item_active,
                           int64_t *profit, int64_t *oldsum, cudaStream_t st)
{
    if (batch <= 0 || inst->n == 0) return PP_OK;
    int bx = (inst->n + 255) / 256;
    int cap = (2 * inst->sm_count * 8 + batch - 1) / batch;   // ~16 blocks per SM overall
    if (bx > cap) bx = cap;
    if (bx < 1) bx = 1;
    dim3 grid(bx, batch);
    const auto go = inst->mode == 0 ? (by_node ? marg_launch<true, 0> : marg_launch<false, 0>)
                                    : (by_node ? marg_launch<true, 1> : marg_launch<false, 1>);
    PP_CUDA(go(inst, grid, worker, mask, item_active, profit, oldsum, st));
    return PP_OK;
}

// ---------------------------------------------------------------------------
// Source-dependent marginals from top-2 holder tables (Section IV-C: keeping
// the largest and second-largest current holder value of every requester-
// chunk pair gives every leave-one-worker-out marginal in O(M^2 n) per sweep).
// Per start s, requester m and position i: v1 = max over the holders l of
// g_{l,m}(i), l1 = the first holder reaching it, v2 = the largest value among
// the other holders (0 with fewer than two).  Then
//   max_{l in H_b \ h} g_{l,m}(b) = (l1 == h) ? v2 : v1,
// which is exact also under ties (then v2 = v1).  The tables hold for the
// holder masks `seen`; a marginal pass first applies the change of the chunks
// whose mask differs (the step before changed one worker's bit).
// A marginal depends on the other workers' holdings alone, so each worker's
// marginals are kept (`marg`), with a bit per worker and chunk that says
// which are stale: a changed chunk makes every worker's stale but the changed
// one's.  After the greedy pass few are, and a pass reads 28 bytes a chunk
// instead of 17 W.
// ---------------------------------------------------------------------------
// Apply worker h's change at chunk i to the top-2 entry of requester m (tb =
// the start's table base): h joined -> insert its value; h left -> rebuild the
// entry where it was the top holder or tied the second.
__device__ __forceinline__ void top2_apply(int32_t n, int32_t W, int32_t h, int32_t m, int32_t i, uint32_t mk, bool now,
                                           size_t tb, const int64_t *__restrict__ g, const Top2 &t)
{
    const size_t q = tb + (size_t)m * n + i;
    const int64_t x = g[((size_t)h * W + m) * n + i], a = t.v1[q], b = t.v2[q];
    const int l1 = t.l1[q];
    if (now) {
        if (l1 < 0 || x > a) {
            t.v2[q] = l1 < 0 ? 0 : a;
            t.v1[q] = x;
            t.l1[q] = (int8_t)h;
        } else if (x > b) {
            t.v2[q] = x;
        }
        return;
    }
    if (l1 != h && x < b) return;
    int64_t b1 = 0, b2 = 0;
    int id1 = -1;
    for (uint32_t o = mk; o;) {
        constexpr int U = 4;                 // holders whose loads are in flight
        int id[U];
        int64_t y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            id[u] = o ? __ffs(o) - 1 : -1;
            o &= o - 1;
            if (id[u] >= 0) y[u] = g[((size_t)id[u] * W + m) * n + i];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (id[u] < 0) break;
            if (id1 < 0 || y[u] > b1) {
                b2 = id1 < 0 ? 0 : b1;
                b1 = y[u];
                id1 = id[u];
            } else if (y[u] > b2) {
                b2 = y[u];
            }
        }
    }
    t.v1[q] = b1;
    t.v2[q] = b2;
    t.l1[q] = (int8_t)id1;
}

// requester m's share of worker h's marginal at chunk i
__device__ __forceinline__ int64_t top2_share(int32_t n, int32_t W, int32_t h, int32_t m, int32_t i, size_t tb,
                                              const int64_t *__restrict__ g, const Top2 &t)
{
    const size_t q = tb + (size_t)m * n + i;
    const int64_t a = g[((size_t)h * W + m) * n + i], b = t.v1[q], c = t.v2[q];
    const int64_t other = t.l1[q] == h ? c : b;
    return a > other ? a - other : 0;
}

// A lane per chunk; a changed chunk's tables, and a stale marginal unless many
// lanes have one, are the work of G lanes, a lane per requester: one lane
// alone waited for memory W times (and W times per holder in a rebuild), which
// was 53 us a pass whatever n.  Changed chunks lie next to one another
// (subtrees), so a warp's 32 chunks are four runs of 8 (a sector of masks)
// from the four quarters of the order, and 32 / G chunks are done at once.
template <int G>                             // lanes per chunk: the power of two from W on, at least 8
__global__ void __launch_bounds__(256) k_marginals_top2(int32_t n, int32_t W, const int32_t *__restrict__ worker,
                                                         const uint32_t *__restrict__ mask,
                                                         const int64_t *__restrict__ g, Top2 t,
                                                         const int32_t *__restrict__ item_active,
                                                         int64_t *__restrict__ profit, int64_t *__restrict__ oldsum,
                                                         int32_t *__restrict__ status)
{
    constexpr unsigned kAllLanes = 0xffffffffu;
    chain_wait();
    chain_release();
    const int item = blockIdx.y;
    if (item_active && !item_active[item]) return;
    const int32_t h = worker[item];
    const uint32_t *M = mask + (size_t)item * n;
    int64_t *P = profit + (size_t)item * n;
    if (h < 0 || h >= W) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicExch(status, (int32_t)PP_EBOUNDS);
        for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) P[i] = 0;
        return;
    }
    const int lane = threadIdx.x & 31;
    const size_t tb = (size_t)item * W * n;
    int64_t *marg = t.marg + tb + (size_t)h * n;
    uint32_t *seen = t.seen + (size_t)item * n, *stale = t.stale + (size_t)item * n;
    int64_t held = 0;
    constexpr int kAtOnce = 32 / G;
    const int m = lane % G;                  // requester, where lanes share a chunk
    const int32_t units = (n + 31) / 32, dw = gridDim.x * blockDim.x / 32;
    for (int32_t x0 = (blockIdx.x * blockDim.x + threadIdx.x) / 32; x0 < units; x0 += dw) {
        const int32_t i = ((lane >> 3) * units + x0) * 8 + (lane & 7);
        const bool in = i < n;
        // the lane whose chunk this lane's group takes of the lanes in `c` (-1: none)
        auto mine = [&](unsigned c) {
            for (int q = 0; q < lane / G; ++q) c &= c - 1;
            return __ffs((int)c) - 1;
        };
        auto rest = [](unsigned c) {
#pragma unroll
            for (int q = 0; q < kAtOnce; ++q) c &= c - 1;
            return c;
        };
        const uint32_t mk = in ? M[i] : 0, was = in ? seen[i] : 0, st = in ? stale[i] : 0;
        int64_t p = in ? marg[i] : 0;
        uint32_t s = st;
        if (mk != was) {
            seen[i] = mk;
            s |= ~(mk ^ was);
        }
        for (unsigned c = __ballot_sync(kAllLanes, mk != was); c; c = rest(c)) {
            const int src = mine(c);
            const uint32_t now = __shfl_sync(kAllLanes, mk, src & 31), x = now ^ __shfl_sync(kAllLanes, was, src & 31);
            const int32_t at = __shfl_sync(kAllLanes, i, src & 31);
            if (src >= 0 && m < W) top2_apply(n, W, __ffs(x) - 1, m, at, now, (now & x) != 0, tb, g, t);
        }
        __syncwarp();                        // the tables' new entries, before the shares below
        const bool old = (s >> h) & 1u;
        const unsigned all = __ballot_sync(kAllLanes, old);
        if (__popc(all) <= 8) {
            for (unsigned c = all; c; c = rest(c)) {
                const int src = mine(c);
                const int32_t at = __shfl_sync(kAllLanes, i, src & 31);
                int64_t v = src >= 0 && m < W ? top2_share(n, W, h, m, at, tb, g, t) : 0;
#pragma unroll
                for (int q = G / 2; q > 0; q >>= 1) v += __shfl_xor_sync(kAllLanes, v, q);
                const int rank = __popc(c & ((1u << lane) - 1));       // which group took this lane's chunk
                v = __shfl_sync(kAllLanes, v, rank * G & 31);
                if ((c >> lane & 1u) && rank < kAtOnce) p = v;
            }
        } else if (old) {
            p = 0;
#pragma unroll 4
            for (int32_t r = 0; r < W; ++r) p += top2_share(n, W, h, r, i, tb, g, t);
        }
        if (old) {
            marg[i] = p;
            s &= ~(1u << h);
        }
        if (s != st) stale[i] = s;
        if (in) P[i] = p;
        if ((mk >> h) & 1u) held += p;
    }
    if (oldsum) block_add64(held, oldsum + item);
}

pp_status launch_marginals_top2(pp_instance *inst, int batch, const int32_t *worker,
                                const uint32_t *mask, const int32_t *item_active, const Top2 &t2,
                                int64_t *profit, int64_t *oldsum, cudaStream_t st)
{
    if (batch <= 0 || inst->n == 0) return PP_OK;
    int bx = (inst->n + 255) / 256;
    int cap = (2 * inst->sm_count * 8 + batch - 1) / batch;
    if (bx > cap) bx = cap;
    if (bx < 1) bx = 1;
    const auto kern = inst->W <= 8 ? k_marginals_top2<8> : inst->W <= 16 ? k_marginals_top2<16> : k_marginals_top2<32>;
    PP_CUDA(launch_chained(kern, dim3(bx, batch), dim3(256), 0, st, 1, inst->n, inst->W, worker, mask,
                           inst->d_g, t2, item_active, profit, oldsum, inst->d_status));
    return PP_OK;
}

// ---------------------------------------------------------------------------
// Objective of holder masks (planner, preorder) or of [W][n] byte placements
// by node id (ABI).  Eq. 4: sum over held (m, b) of a_m(b) plus Delta(b) once
// per covered chunk.  Eq. 6: sum_b sum_m max_{h in H_b} g_h,m(b).
// ---------------------------------------------------------------------------
template <bool FROM_BYTES, int MODE>
__global__ void __launch_bounds__(256) k_objective(int32_t n, int32_t W,
                                                    const uint32_t *__restrict__ mask,
                                                    const uint8_t *__restrict__ chosen,
                                                    const int32_t *__restrict__ order,
                                                    const int64_t *__restrict__ a,
                                                    const int64_t *__restrict__ delta,
                                                    const int64_t *__restrict__ g,
                                                    int64_t *__restrict__ obj)
{
    const int item = blockIdx.y;
    int64_t acc = 0;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        uint32_t mk = 0;
        if (FROM_BYTES) {
            const int32_t b = order[i];
            for (int32_t m0 = 0; m0 < W; m0 += kReq) {
                uint8_t c[kReq];
#pragma unroll
                for (int u = 0; u < kReq; ++u)
                    c[u] = m0 + u < W ? __ldg(chosen + ((size_t)item * W + m0 + u) * n + b) : 0;
#pragma unroll
                for (int u = 0; u < kReq; ++u) mk |= c[u] ? 1u << (m0 + u) : 0u;
            }
        } else {
            mk = mask[(size_t)item * n + i];
        }
        if (mk == 0) continue;
        if (MODE == 0) {
            uint32_t o = mk;
            while (o) {
                int m = __ffs(o) - 1;
                o &= o - 1;
                acc += a[(size_t)m * n + i];
            }
            acc += delta[i];
        } else {
            for (int32_t m0 = 0; m0 < W; m0 += kReq) {
                int64_t v[kReq];
                best_of(n, W, mk, m0, i, g, v);
#pragma unroll
                for (int u = 0; u < kReq; ++u) acc += v[u];
            }
        }
    }
    block_add64(acc, obj + item);
}

pp_status launch_objective(pp_instance *inst, int batch, const uint32_t *mask,
                           const uint8_t *chosen, int64_t *obj, cudaStream_t st)
{
    if (batch <= 0) return PP_OK;
    PP_CUDA(cudaMemsetAsync(obj, 0, sizeof(int64_t) * batch, st));
    if (inst->n == 0) return PP_OK;
    int bx = (inst->n + 255) / 256;
    int cap = (2 * inst->sm_count * 8 + batch - 1) / batch;
    if (bx > cap) bx = cap;
    if (bx < 1) bx = 1;
    dim3 grid(bx, batch);
    const int32_t n = inst->n, W = inst->W;
    if (chosen) {
        if (inst->mode == 0)
            k_objective<true, 0><<<grid, 256, 0, st>>>(n, W, nullptr, chosen, inst->d_order, inst->d_a,
                                                       inst->d_delta, inst->d_g, obj);
        else
            k_objective<true, 1><<<grid, 256, 0, st>>>(n, W, nullptr, chosen, inst->d_order, inst->d_a,
                                                       inst->d_delta, inst->d_g, obj);
    } else {
        if (inst->mode == 0)
            k_objective<false, 0><<<grid, 256, 0, st>>>(n, W, mask, nullptr, inst->d_order, inst->d_a,
                                                        inst->d_delta, inst->d_g, obj);
        else
            k_objective<false, 1><<<grid, 256, 0, st>>>(n, W, mask, nullptr, inst->d_order, inst->d_a,
                                                        inst->d_delta, inst->d_g, obj);
    }
    PP_CUDA(cudaGetLastError());
    return PP_OK;
}

}  // namespace pp

using namespace pp;

extern "C" pp_status pp_marginals(pp_instance *inst, int32_t batch, const int32_t *worker,
                                  const uint32_t *holder_mask, int64_t *profit, void *stream)
{
    if (!inst) return fail(PP_EINVAL, "null instance");
    if (batch < 0) return fail(PP_EINVAL, "batch must be >= 0");
    if (batch == 0 || inst->n == 0) return PP_OK;
    if (!worker || !holder_mask || !profit) return fail(PP_EINVAL, "null device pointer");
    return launch_marginals(inst, batch, worker, holder_mask, true, nullptr, profit, nullptr,
                            (cudaStream_t)stream);
}

extern "C" pp_status pp_objective(pp_instance *inst, int32_t batch, const uint8_t *chosen,
                                  int64_t *obj, void *stream)
{
    if (!inst) return fail(PP_EINVAL, "null instance");
    if (batch < 0) return fail(PP_EINVAL, "batch must be >= 0");
    if (batch == 0) return PP_OK;
    if (!obj || (inst->n > 0 && !chosen)) return fail(PP_EINVAL, "null device pointer");
    return launch_objective(inst, batch, nullptr, chosen, obj, (cudaStream_t)stream);
}
