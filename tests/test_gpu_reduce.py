"""The exact reduction before the tree DP's sweep (csrc/pp_reduce.cu), bit for
bit against the oracle: trees around its tile, stream and cluster boundaries,
budgets that bind or do not, ties that leave it more undecided rows than it
takes, and paths too long for it.  Everything is integer: equality."""
import threading

import numpy as np
import pytest

from paper_2608_01655_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_01655_gb300 import build
    build.build()
    from paper_2608_01655_gb300 import binding
    return binding


def _tree(rng, shape, n):
    if shape == "random":
        return np.array([-1] + [int(rng.integers(v)) if rng.random() < 0.98 else -1 for v in range(1, n)], np.int32)
    if shape == "star":
        return np.full(n, -1, np.int32)
    if shape == "chain":
        return np.arange(-1, n - 1, dtype=np.int32)
    if shape == "caterpillar":                   # a spine of n / 2 nodes, a leaf on each
        return np.array([-1] + [v - 1 if v % 2 else max(v - 2, 0) for v in range(1, n)], np.int32)
    return wl._mixed_tree(rng, n)                # chains under a bushy prefix


def _check(pp, oracle_lib, parent, weight, profits, budgets, by_rows):
    n, B = len(parent), len(profits)
    inst = wl.Instance("t", n, 1, parent, weight, np.ones((1, n), np.int64), np.ones((1, n), np.int64),
                       np.ones((1, n), np.int64), 0, np.array([1], np.int32), 1, 1)
    maxb = int(max(budgets))
    with pp.Instance.from_workload(inst) as ppi:
        prof = torch.from_numpy(np.ascontiguousarray(profits, np.int64)).cuda()
        bud = torch.from_numpy(np.asarray(budgets, np.int32)).cuda()
        best = torch.zeros(B, dtype=torch.int64, device="cuda")
        bits = torch.randint(0, 1 << 30, (pp.pp_dp_bits_size(ppi, B, maxb) // 4,), dtype=torch.int32, device="cuda")
        chosen = torch.zeros((B, n), dtype=torch.uint8, device="cuda")
        for _ in range(2):                       # the workspace holds anything, then the last call's
            pp.pp_tree_dp(ppi, prof, bud, maxb, best, bits)
            pp.pp_traceback(ppi, bits, bud, maxb, chosen)
            ppi.sync()
            for b in range(B):
                ob, oc = oracle_lib.rooted_dp(parent, weight, profits[b], int(budgets[b]))
                assert int(best[b]) == ob, b
                np.testing.assert_array_equal(chosen[b].cpu().numpy(), oc, err_msg=str(b))
        by_rows(pp.pp_dp_rows_swept(ppi, B, maxb, bits))
    return chosen.cpu().numpy()


@pytest.mark.parametrize("shape", ["random", "star", "caterpillar", "mixed"])
@pytest.mark.parametrize("n,wmax", [(1024, 1), (1055, 3), (6144, 1), (6145, 2), (12289, 9), (24577, 1)])
def test_reduced_optimum_and_set(pp, oracle_lib, shape, n, wmax):
    """Layouts of one bin, six and sixteen, weights on and above the wavefront kernel's limit;
    per batch: profits over several decades, few values (ties), mostly zero,
    negative ones, a budget of one slot and one that does not bind."""
    rng = np.random.default_rng(n + wmax)
    parent = _tree(rng, shape, n)
    weight = rng.integers(1, wmax + 1, size=n).astype(np.int32)
    wide = np.exp(rng.uniform(0, 18, size=(6, n))).astype(np.int64)
    wide[1] = rng.integers(0, 4, size=n)
    wide[2][rng.random(n) < 0.9] = 0
    wide[3] -= int(np.quantile(wide[3], 0.6))
    tw = int(weight.sum())
    budgets = [n // 9 + 1, n // 20, n // 7, n // 11 + 3, 1, min(tw + 5, 8192)]

    def rows(r):
        if tw <= 8192 and (shape != "caterpillar" or n < 2048):     # (a spine of n / 2 rows is too long from there on)
            assert r[5] == 0                     # nothing is undecided without a limit
        if shape == "mixed":
            assert r[0] <= n // 4                # few rows are left undecided
    _check(pp, oracle_lib, parent, weight, wide, budgets, rows)


@pytest.mark.parametrize("n", [128, 501, 1537, 12289])
@pytest.mark.parametrize("batch", [1, 9, 17, 33, 65])
def test_cluster_sizes(pp, oracle_lib, n, batch):
    """The items of a launch decide how many CTAs share one, and so how many
    bins a CTA walks."""
    rng = np.random.default_rng(n + batch)
    parent = _tree(rng, "mixed", n)
    profits = np.exp(rng.uniform(0, 18, size=(batch, n))).astype(np.int64)
    profits[:, rng.random(n) < 0.3] = 0
    budgets = rng.integers(1, 90, size=batch)
    _check(pp, oracle_lib, parent, np.ones(n, np.int32), profits, budgets, lambda r: None)


def test_ties_and_zero_budget_and_long_paths(pp, oracle_lib):
    """Equal profits on a star leave every row undecided (the pruned sweep
    takes over), a budget of 0 takes nothing, profits near 2^61 are beyond the
    price's range, and a path above 1,024 rows is not reduced at all."""
    rng = np.random.default_rng(5)
    n = 3000
    one = np.ones(n, np.int32)
    profits = np.stack([np.full(n, 7), rng.integers(1, 99, n), np.where(np.arange(n) == 5, 1 << 61, 3)]).astype(np.int64)

    def rows(r):
        assert r[0] == n and r[1] == 0 and r[2] > 1024
    _check(pp, oracle_lib, np.full(n, -1, np.int32), one, profits, [100, 0, 50], rows)
    for m, want in ((1024, False), (1025, True)):
        p = rng.integers(1, 99, size=(1, m)).astype(np.int64)

        def swept(r, want=want, m=m):
            assert (r[0] == m) == want
        _check(pp, oracle_lib, _tree(rng, "chain", m), np.ones(m, np.int32), p, [m], swept)


@pytest.mark.parametrize("n,batch", [(60000, 40), (66000, 40), (72001, 40), (72001, 17), (140000, 20)])
def test_many_tiles_in_few_ctas(pp, oracle_lib, n, batch):
    """More than 2,048 tiles before the last bin, whose rows have no profit, on
    two CTAs an item (and four), accumulators in shared memory and beyond."""
    rng = np.random.default_rng(n)
    parent = np.array([-1] + [int(rng.integers(max(0, v - 60), v)) if rng.random() < 0.95 else int(rng.integers(min(v, 40)))
                              for v in range(1, n)], np.int32)
    profits = np.exp(rng.uniform(0, 18, size=(2, n))).astype(np.int64)
    profits[:, rng.random(n) < 0.5] = 0
    size = np.ones(n, np.int64)
    for v in range(n - 1, 0, -1):
        size[parent[v]] += size[v]
    profits[:, size > 200] = 0
    profits[1] -= 3
    _check(pp, oracle_lib, parent, np.ones(n, np.int32), np.tile(profits, (batch // 2 + 1, 1))[:batch],
           np.resize([400, 60, 7, 150], batch), lambda r: None)


@pytest.mark.parametrize("wmax", [1, 9])
@pytest.mark.parametrize("top", [10 ** 9, (1 << 55) - 1, 1 << 56, 1 << 57, 279496122328932600, 558992244657865200, 1 << 59, 1 << 60])
def test_profits_up_to_the_bound(pp, oracle_lib, top, wmax):
    """Few profits with ties between them (absolute sum below 2^62) and chains
    without any: a price of that size times a tile's 32 rows leaves int64."""
    rng = np.random.default_rng(wmax)
    parent = [-1] * 32 + [19, 4, 8, 4, 35, 2, 12, 37, 0, 30, 3, 32, 13, 17, 10, 34, 35, 12, 25, 13, 35, 30, 22, 29, 31,
                          18, 36, 22, 19, 33, 22, 35, 53, 26, 5, 22]
    for above, length in ((16, 31), (67, 31), (35, 41), (68, 2), (5, 58)):
        parent += [above] + list(range(len(parent), len(parent) + length - 1))
    n = len(parent)
    profits = np.zeros((3, n), np.int64)
    profits[0, [14, 55, 155, 197][: 4 if top < 1 << 60 else 3]] = top
    profits[1, [14, 55, 197]] = top
    profits[2, [14, 55]] = top
    profits[2, :14] = -1
    weight = rng.integers(1, wmax + 1, size=n).astype(np.int32)
    _check(pp, oracle_lib, np.array(parent, np.int32), weight, np.tile(profits, (5, 1)),
           np.repeat([1, 2, 3, 5, 40], 3) * wmax, lambda r: None)


@pytest.mark.parametrize("n", [31, 257, 1030])
@pytest.mark.parametrize("W", [1, 8, 9, 16, 17, 32])
def test_kept_marginals_of_every_lane_group(pp, oracle_lib, n, W):
    """Plans from top-2 tables at the widths where 8, 16 and 32 lanes share a
    chunk, over orders that do not fill their four quarters: many chunks change
    per update, so several are done at once, in one lane group and the next."""
    rng = np.random.default_rng(n * 40 + W)
    inst = wl.random_small(rng, n, W, 1, k_max=max(2, n // 4), w_max=2, demand_max=20)
    o = oracle_lib.plan(oracle_lib.Problem.from_instance(inst), 2, 2)
    with pp.Instance.from_workload(inst) as ppi:
        g = pp.pp_plan_run(ppi, 2, None, 2, marginals=2)
    assert g.used_top2 and g.objective == o.objective
    np.testing.assert_array_equal(g.placement, o.placement)


@pytest.mark.parametrize("starts,schedule", [(1, 0), (3, 0), (3, 1), (9, 2)])
def test_safeguards_beside_the_starts(pp, oracle_lib, starts, schedule):
    """Candidates computed on their own stream while the starts run are those
    computed after them (a plan whose phases are timed), call after call."""
    inst = wl.random_small(np.random.default_rng(starts), 900, 5, 0, k_max=200, w_max=2, demand_max=50)
    o = oracle_lib.plan(oracle_lib.Problem.from_instance(inst), starts, 2)
    with pp.Instance.from_workload(inst) as ppi:
        for timed in (False, True, False, False):
            g = pp.pp_plan_run(ppi, starts, None, 2, schedule=schedule, time_phases=timed)
            assert list(g.safeguard_objective) == o.safeguard_objective.tolist()
            assert g.objective == o.objective and g.best_start == o.best_start
            np.testing.assert_array_equal(g.placement, o.placement)


def _down(x):
    """Sums of two float32 values (exact in float64) rounded down to float32."""
    y = x.astype(np.float32)
    return np.where(y.astype(np.float64) > x, np.nextafter(y, np.float32(-np.inf)), y).astype(np.float64)


def _doubling_sums(a):
    """Sums from each row of a path to its top ([trials][rows], bottom first)
    by a doubling scan of float32 values in tiles of 32, top tile first."""
    out, carry = np.empty_like(a), None
    for t0 in range((a.shape[1] - 1) // 32 * 32, -1, -32):
        x = _down(a[:, t0:t0 + 32])
        m = x.shape[1]
        for o in (1, 2, 4, 8, 16):
            y = x.copy()
            if o < m:
                y[:, :m - o] = _down(x[:, :m - o] + x[:, o:])
            x = y
        if carry is not None:
            x = _down(x + carry[:, None])
        carry = x[:, 0]
        out[:, t0:t0 + 32] = x
    return out


def _rounded_apart(rng, m, tail, wmax, extra):
    """A path of m rows that lose value at the price 2^40, above a row that
    gains; `tail` rows below that one.  Losses of the m rows are such that the
    gaining row's and its parent's, equal by themselves, lie on two sides of a
    key's edge, the first threshold's, if they are sums of a doubling scan.  The
    gaining row without its parent would fill the budget that is left."""
    lam, g = 1 << 40, 1 << 34
    wt = rng.integers(1, wmax + 1, size=m)               # from the gaining row's parent up
    slots = int(wt[1:].sum()) + 1
    k = max(200, 21 * slots * slots)                     # |S| = k - slots is near enough to k
    big, pairs = k - slots, slots - 1
    n = m + 1 + tail + 2 * pairs + big + extra
    t = np.float32(0.1) * np.float32(lam) * (np.float32(n - m + int(wt.sum())) / np.float32(n))
    e = int(np.floor(np.log2(t)))
    edge = int((int(t / 2.0 ** e * 32) + 1) * 2.0 ** (e - 5))          # 32 keys an octave
    hit = []
    while len(hit) == 0:
        cut = np.sort(rng.integers(1, edge, size=(4000, m - 1)), axis=1)
        a = np.diff(np.concatenate([np.zeros((4000, 1), np.int64), cut, np.full((4000, 1), edge)], axis=1), axis=1)
        a = a >> 12 << 12
        a[:, 0] += edge - a.sum(1)
        s = _doubling_sums(np.concatenate([np.full((4000, tail), lam - 5.0), np.zeros((4000, 1)), a], axis=1))
        hit = np.flatnonzero((s[:, tail + 1] >= edge) & (s[:, tail] < edge))
    a = a[hit[0]]
    parent, profit, weight = [], [], []

    def add(above, value, w=1):
        parent.append(above)
        profit.append(int(value))
        weight.append(int(w))
        return len(parent) - 1
    at = -1
    for i in range(m - 1, -1, -1):
        at = add(at, lam * int(wt[i]) - int(a[i]) - (g if i == 0 else 0), wt[i])
    at = add(at, lam + g)
    for _ in range(tail):
        at = add(at, 5)
    for _ in range(pairs):
        add(add(-1, 0), lam + g)
    for i in range(big):
        add(-1, (2 << 40) + 12345 * i)
    while len(parent) < n:
        add(-1, 5 + len(parent) % 97)
    return np.array(parent, np.int32), np.array(weight, np.int32), np.array(profit, np.int64), k


def _assert_closed(parent, chosen):
    below = parent >= 0
    assert not np.any(chosen[:, below] > chosen[:, parent[below]])


@pytest.mark.parametrize("m,tail,wmax,extra", [
    (3, 0, 1, 60), (3, 28, 1, 60), (4, 10, 1, 60), (5, 27, 1, 60), (8, 28, 1, 60), (8, 60, 1, 2000), (14, 25, 1, 9000),
    (4, 0, 3, 60), (5, 28, 3, 60), (8, 28, 2, 60)])
def test_rounded_losses_keep_rows_together(pp, oracle_lib, m, tail, wmax, extra):
    """Losses above 2^24 are rounded: a row is never undecided below one that is
    decided out, in a tile and across its edge, on one CTA and on several."""
    for seed in range(3):
        parent, weight, profit, k = _rounded_apart(np.random.default_rng(seed), m, tail, wmax, extra)
        chosen = _check(pp, oracle_lib, parent, weight, profit[None], [k], lambda r: None)
        _assert_closed(parent, chosen)


def test_three_losses_in_two_orders(pp, oracle_lib):
    """The same with the numbers written out: 13 * 2^33 = a + a + c, budget 200."""
    lam, g, a = 1 << 40, 1 << 34, (1 << 35) + (1 << 12)
    c = 13 * (1 << 33) - 2 * a
    parent = np.array([-1, 0, 1, 2, -1, 4, -1, 6] + [-1] * 257, np.int32)
    profit = np.array([lam - c, lam - a, lam - a - g, lam + g, 0, lam + g, 0, lam + g] +
                      [(2 << 40) + 12345 * i for i in range(197)] + [5 + i for i in range(60)], np.int64)
    chosen = _check(pp, oracle_lib, parent, np.ones(265, np.int32), profit[None], [200], lambda r: None)
    _assert_closed(parent, chosen)


def _few_profits(rng, n, B):
    profits = np.exp(rng.uniform(0, 18, size=(B, n))).astype(np.int64)
    profits[rng.random((B, n)) < 0.9] = 0
    return profits


@pytest.mark.parametrize("n,k", [(1600, 80), (1900, 95)])
def test_rows_left_to_the_sweep_are_pruned(pp, oracle_lib, n, k):
    """A tenth of the profits: whatever the reduction leaves undecided, no row
    is swept that pruning alone would drop."""
    rng = np.random.default_rng(n)
    parent = _tree(rng, "caterpillar", n)
    profits = _few_profits(rng, n, 12)
    positive = profits > 0                       # at or below a row
    for v in range(n - 1, 0, -1):
        if parent[v] >= 0:
            positive[:, parent[v]] |= positive[:, v]

    def rows(r):
        swept = r > 1024                         # more than the DP on chip takes
        assert (r[swept] <= positive.sum(axis=1)[swept]).all()
    chosen = _check(pp, oracle_lib, parent, np.ones(n, np.int32), profits, [k] * 12, rows)
    _assert_closed(parent, chosen)


@pytest.mark.parametrize("shape,n,k", [("random", 1600, 80), ("random", 12000, 600), ("mixed", 4000, 200)])
def test_price_far_above_the_first_guess(pp, oracle_lib, shape, n, k):
    """Few chunks with a profit, whole paths taken for one: the price is a
    hundred times the k-th largest profit, and is found all the same."""
    rng = np.random.default_rng(n + 1)
    parent = _tree(rng, shape, n)

    def rows(r):
        assert (r <= 1024).all() and np.median(r) <= 256
    _check(pp, oracle_lib, parent, np.ones(n, np.int32), _few_profits(rng, n, 6), [k] * 6, rows)


@pytest.mark.parametrize("shape,n,k", [("mixed", 1600, 80), ("random", 800, 40)])
def test_price_just_below_the_first_guess(pp, oracle_lib, shape, n, k):
    """Profits within a tenth of one another: the price lies within that tenth,
    and the search does not go through zero and use up its prices."""
    rng = np.random.default_rng(n + 2)
    parent = _tree(rng, shape, n)
    profits = rng.integers(10 ** 6, 10 ** 6 + 10 ** 5, size=(4, n))

    def rows(r):
        assert (r <= 640).all(), r
    _check(pp, oracle_lib, parent, np.ones(n, np.int32), profits, [k] * 4, rows)


@pytest.mark.parametrize("k,most", [(40, 2.0), (160, 2.8)])
def test_items_that_do_not_reduce_stop_early(pp, oracle_lib, k, most):
    """Nothing to gain on a chain that pays all at its end, and a price takes
    its 25 tiles in turn: up to 128 columns the sweep is left to it at once,
    with more the call may take about twice the sweep of all rows (which is
    what the pruned sweep takes here).  It took 3.4 to 3.8 times."""
    rng = np.random.default_rng(k)
    n = 800
    parent = _tree(rng, "chain", n)
    profit = np.zeros((1, n), np.int64)
    profit[0, -1] = 10 ** 6
    profit[0, ::7] = rng.integers(1, 10 ** 4, size=len(profit[0, ::7]))
    _check(pp, oracle_lib, parent, np.ones(n, np.int32), profit, [k], lambda r: None)
    inst = wl.Instance("t", n, 1, parent, np.ones(n, np.int32), np.ones((1, n), np.int64), np.ones((1, n), np.int64),
                       np.ones((1, n), np.int64), 0, np.array([1], np.int32), 1, 1)
    took = []
    with pp.Instance.from_workload(inst) as ppi:
        prof = torch.from_numpy(profit).cuda()
        bud = torch.full((1,), k, dtype=torch.int32, device="cuda")
        best = torch.zeros(1, dtype=torch.int64, device="cuda")
        bits = torch.zeros(pp.pp_dp_bits_size(ppi, 1, k) // 4, dtype=torch.int32, device="cuda")
        chosen = torch.zeros((1, n), dtype=torch.uint8, device="cuda")
        for noprune in (True, False):
            pp.pp_tune_dp(ppi, 0, 0, False, noprune)
            times = []
            for _ in range(25):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                pp.pp_tree_dp(ppi, prof, bud, k, best, bits)
                pp.pp_traceback(ppi, bits, bud, k, chosen)
                b.record()
                b.synchronize()
                times.append(a.elapsed_time(b))
            took.append(float(np.median(times[5:])))
    assert took[1] <= most * took[0], took


@pytest.mark.parametrize("solved_by_reduction", [True, False])
def test_workspace_is_read_as_it_was_written(pp, oracle_lib, solved_by_reduction):
    """Switching the reduction off or on between the DP and its traceback does
    not change what the workspace holds."""
    rng = np.random.default_rng(8)
    n, k = 900, 120
    parent = _tree(rng, "mixed", n)
    weight = rng.integers(1, 3, size=n).astype(np.int32)
    profit = np.exp(rng.uniform(0, 18, size=(2, n))).astype(np.int64)
    inst = wl.Instance("t", n, 1, parent, weight, np.ones((1, n), np.int64), np.ones((1, n), np.int64),
                       np.ones((1, n), np.int64), 0, np.array([1], np.int32), 1, 1)
    with pp.Instance.from_workload(inst) as ppi:
        prof = torch.from_numpy(profit).cuda()
        bud = torch.full((2,), k, dtype=torch.int32, device="cuda")
        best = torch.zeros(2, dtype=torch.int64, device="cuda")
        bits = torch.zeros(pp.pp_dp_bits_size(ppi, 2, k) // 4, dtype=torch.int32, device="cuda")
        chosen = torch.zeros((2, n), dtype=torch.uint8, device="cuda")
        pp.pp_tune_dp(ppi, 0, 0, False, not solved_by_reduction)
        pp.pp_tree_dp(ppi, prof, bud, k, best, bits)
        pp.pp_tune_dp(ppi, 0, 0, False, solved_by_reduction)
        pp.pp_traceback(ppi, bits, bud, k, chosen)
        ppi.sync()
        assert (pp.pp_dp_rows_swept(ppi, 2, k, bits) < n).all() == solved_by_reduction
        for b in range(2):
            ob, oc = oracle_lib.rooted_dp(parent, weight, profit[b], k)
            assert int(best[b]) == ob
            np.testing.assert_array_equal(chosen[b].cpu().numpy(), oc)


@pytest.mark.parametrize("shape,n,wmax", [("mixed", 6000, 1), ("random", 12000, 3), ("star", 6000, 9)])
def test_some_rows_decided_and_the_rest_swept(pp, oracle_lib, shape, n, wmax):
    """Ten profits close to one another: more rows stay undecided than the DP on
    chip takes and fewer than pruning alone leaves, so the sweep joins the
    decided rows, on the wavefront kernel and the one-CTA kernel."""
    rng = np.random.default_rng(n + wmax)
    parent = _tree(rng, shape, n)
    weight = rng.integers(1, wmax + 1, size=n).astype(np.int32)
    profits = np.stack([rng.integers(10 ** 6, 10 ** 6 + 10 ** 5, n), rng.integers(1000, 1010, n)]).astype(np.int64)

    def rows(r):
        assert 1024 < r[1] < n
    chosen = _check(pp, oracle_lib, parent, weight, profits, [n // 20 * wmax] * 2, rows)
    _assert_closed(parent, chosen)


@pytest.mark.parametrize("shape,n,k", [("random", 100, 20), ("mixed", 2000, 256), ("mixed", 20000, 1000), ("star", 3000, 300)])
def test_update_chain_in_a_graph(pp, oracle_lib, shape, n, k):
    """The allocation-free DP and its traceback, chained by programmatic
    dependent launch, captured in a CUDA graph and replayed on new profits:
    trees with and without the reduction, items that it solves and leaves."""
    rng = np.random.default_rng(n)
    parent = _tree(rng, shape, n)
    inst = wl.Instance("t", n, 1, parent, np.ones(n, np.int32), np.ones((1, n), np.int64), np.ones((1, n), np.int64),
                       np.ones((1, n), np.int64), 0, np.array([1], np.int32), 1, 1)
    with pp.Instance.from_workload(inst) as ppi:
        prof = torch.zeros((3, n), dtype=torch.int64, device="cuda")
        bud = torch.tensor([k, k // 2, 0], dtype=torch.int32, device="cuda")
        best = torch.zeros(3, dtype=torch.int64, device="cuda")
        bits = torch.zeros(pp.pp_dp_bits_size(ppi, 3, k) // 4, dtype=torch.int32, device="cuda")
        chosen = torch.zeros((3, n), dtype=torch.uint8, device="cuda")

        def chain():
            for _ in range(2):                   # a chain, not one call: the second follows the first's last kernel
                pp.pp_tree_dp_noalloc(ppi, prof, bud, k, best, bits)
                pp.pp_traceback(ppi, bits, bud, k, chosen)
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            chain()
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            chain()
        for _ in range(2):
            p = np.exp(rng.uniform(0, 18, size=(3, n))).astype(np.int64)
            p[1] = rng.integers(1, 3, size=n)
            prof.copy_(torch.from_numpy(p))
            chosen.fill_(7)
            graph.replay()
            torch.cuda.synchronize()
            ppi.sync()
            for b, kb in enumerate((k, k // 2, 0)):
                ob, oc = oracle_lib.rooted_dp(parent, np.ones(n, np.int32), p[b], kb)
                assert int(best[b]) == ob
                np.testing.assert_array_equal(chosen[b].cpu().numpy(), oc)


def test_two_instances_on_two_threads(pp, oracle_lib):
    """Launches of instances whose kernels take different amounts of shared
    memory (the sweep's, for weights on both sides of the wavefront kernel's
    limit, and the reduction's) do not disturb one another."""
    errors = []

    def work(n, wmax, k, seed, noprune):
        parent = _tree(np.random.default_rng(seed), "random", n)
        weight = np.random.default_rng(seed).integers(1, wmax + 1, size=n).astype(np.int32)
        profit = np.exp(np.random.default_rng(seed + 1).uniform(0, 18, n)).astype(np.int64)
        best0, set0 = oracle_lib.rooted_dp(parent, weight, profit, k)
        inst = wl.Instance("t", n, 1, parent, weight, np.ones((1, n), np.int64), np.ones((1, n), np.int64),
                           np.ones((1, n), np.int64), 0, np.array([1], np.int32), 1, 1)

        def go():
            try:
                stream = torch.cuda.Stream()
                with pp.Instance.from_workload(inst) as ppi, torch.cuda.stream(stream):
                    pp.pp_tune_dp(ppi, 0, 0, False, noprune)
                    prof = torch.from_numpy(profit[None].copy()).cuda()
                    bud = torch.full((1,), k, dtype=torch.int32, device="cuda")
                    best = torch.zeros(1, dtype=torch.int64, device="cuda")
                    bits = torch.zeros(pp.pp_dp_bits_size(ppi, 1, k) // 4, dtype=torch.int32, device="cuda")
                    chosen = torch.zeros((1, n), dtype=torch.uint8, device="cuda")
                    for _ in range(400):
                        pp.pp_tree_dp(ppi, prof, bud, k, best, bits, stream=stream)
                        pp.pp_traceback(ppi, bits, bud, k, chosen, stream=stream)
                    ppi.sync()
                    stream.synchronize()
                    assert int(best[0]) == best0
                    np.testing.assert_array_equal(chosen[0].cpu().numpy(), set0)
            except Exception as e:                        # noqa: BLE001
                errors.append(repr(e))
        return threading.Thread(target=go)
    threads = [work(300, 9, 500, 1, True), work(301, 9, 1000, 2, True), work(700, 1, 60, 3, True), work(701, 1, 600, 4, True),
               work(1500, 1, 50, 5, False), work(12000, 1, 50, 6, False)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
