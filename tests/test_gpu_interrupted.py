"""What a caller reads after a reduction that stopped part-way: at the time bound or for want of memory.

Every such stop leaves the reduction after some whole number of passes, so the reads are compared with
a pass-by-pass run (a context with per-pass counters) capped there, and with each other. From 3,000,000
columns on columns run ahead of the pass; 270 points have 3,280,455, 200 points 1,333,500.
"""
import numpy as np
import pytest

import pointclouds as pc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ph():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1708_04710_gb300 import build

    build.build()
    import paper_1708_04710_gb300 as ph

    return ph


def _cloud(n):
    return pc.to_grid(pc.sphere(n, np.random.Generator(np.random.PCG64(3)), noise=0.05))


def _built(ph, n, **opts):
    import torch

    ctx = ph.Context(**opts)
    ctx.build_filtration(torch.from_numpy(_cloud(n)).cuda(), None, 2)
    return ctx


class PassByPass:
    """The states of a reduction first capped at pass `first` (a cap takes the pass's marks, and the
    next call goes on behind them) and then at pass k, for any k."""

    def __init__(self, ph, n, first):
        self.ctx, self.first, self.lows = _built(ph, n, collect_stats=True), first, {}
        self.passes = self.state(-1)["passes"]

    def state(self, k):
        self.ctx.reset_reduction()
        st = self.ctx.reduce(max_passes=self.first)
        return st if k == self.first else self.ctx.reduce(max_passes=k)

    def low(self, k):
        if k not in self.lows:
            self.state(k)
            self.lows[k] = self.ctx.filtration(0)["low"]
        return self.lows[k]

    def columns(self, k):
        self.state(k)
        return self.ctx.columns(0)

    def passes_of(self, low):
        """At which cap the lows are these (those that its marks zero may still be there)."""
        for k in range(self.first, self.passes + 1):
            r = self.low(k)
            if np.all((low == r) | (r < 0)):
                return k
        pytest.fail("the lows are those of no pass")


_refs = {}


def _ref(ph, n, first):
    if (n, first) not in _refs:
        _refs[n, first] = PassByPass(ph, n, first)
    return _refs[n, first]


def _check_pairs(ctx):
    """pairs() and essential() are those of the lows."""
    f = ctx.filtration(0)
    order = np.argsort(f["dim"], kind="stable")  # (dimension, index)
    death = order[f["low"][order] >= 0]
    birth = f["low"][death]
    is_low = np.zeros(len(order), bool)
    is_low[birth] = True
    ess = order[(f["low"][order] < 0) & ~is_low[order]]
    for cloud in (-1, 0):
        pr, es = ctx.pairs(cloud, on_device=cloud < 0), ctx.essential(cloud)
        assert np.array_equal(pr["death"].cpu().numpy(), death)
        assert np.array_equal(pr["birth"].cpu().numpy(), birth)
        assert np.array_equal(pr["birth_diam2"].cpu().numpy(), f["diam2"][birth])
        assert np.array_equal(es["idx"].cpu().numpy(), ess)


def _check_columns(ctx, ref):
    """columns() and the lows are those after some pass; returns its number."""
    low = ctx.filtration(0)["low"]
    ptr, rows = ctx.columns(0)
    last = np.full(len(low), -1, np.int64)
    some = np.diff(ptr) > 0
    last[some] = rows[ptr[1:][some] - 1]
    assert np.array_equal(last, low)
    k = ref.passes_of(low)
    rptr, rrows = ref.columns(k)
    kept = ref.low(k) >= 0  # (the others' columns are empty there already)
    assert np.array_equal(np.diff(ptr)[kept], np.diff(rptr)[kept])
    assert np.array_equal(rows[np.repeat(kept, np.diff(ptr))], rrows)
    return k


def _finish(ctx, ref):
    st = ctx.reduce()
    assert st["converged"] and st["passes"] == ref.passes
    assert np.array_equal(ctx.filtration(0)["low"], ref.low(ref.passes))
    _check_pairs(ctx)


def _until_done(ph, ctx, each):
    """Calls reduce until it ends, `each` after every call that the time bound stopped."""
    for stops in range(200):
        try:
            ctx.reduce()
            return stops
        except ph.PHError as err:
            assert err.code == -5
            each()
    pytest.fail("the reduction did not finish")


@pytest.mark.parametrize("n,use_graph", [(200, True), (270, True), (270, False)])
def test_pairs_after_the_time_bound(ph, n, use_graph):
    ctx = _built(ph, n, use_graph=use_graph, timeout_ms=1)
    ctx.reduce(max_passes=0)
    _check_pairs(ctx)
    assert _until_done(ph, ctx, lambda: _check_pairs(ctx)) >= 1
    _finish(ctx, _ref(ph, n, 0))


@pytest.mark.parametrize("n,use_graph", [(200, True), (270, True), (270, False)])
def test_columns_after_the_time_bound(ph, n, use_graph):
    ref = _ref(ph, n, 0)
    ctx = _built(ph, n, use_graph=use_graph, timeout_ms=1)
    ctx.reduce(max_passes=0)
    seen = []
    _until_done(ph, ctx, lambda: seen.append(_check_columns(ctx, ref)))
    assert seen and seen == sorted(set(seen))  # every call runs at least one more pass
    _finish(ctx, ref)


class Allocator:
    """torch's allocator with a number of blocks left to give, or a number of bytes in all."""

    def __init__(self, blocks=None, budget=None):
        self.blocks, self.budget = blocks, budget
        self.size, self.used, self.peak, self.log = {}, 0, 0, []

    def alloc(self, nbytes, stream):
        import torch

        if self.blocks is not None:
            if self.blocks == 0:
                return 0
            self.blocks -= 1
        if self.budget is not None and self.used + nbytes > self.budget:
            return 0
        p = torch.cuda.caching_allocator_alloc(nbytes, stream=stream)
        self.size[p] = nbytes
        self.used += nbytes
        self.peak = max(self.peak, self.used)
        self.log.append(self.used)
        return p

    def free(self, p):
        import torch

        self.used -= self.size.pop(p)
        torch.cuda.caching_allocator_delete(p)

    def opts(self):
        return dict(device_alloc=self.alloc, device_free=self.free)


# one-word arenas, which the passes grow as they need: the call fails at the first to the eighth block
# or, with look-ahead, starts again and gets by with the memory it has
@pytest.mark.parametrize("n,use_graph", [(200, True), (270, True), (270, False)])
def test_reads_after_a_refused_allocation(ph, n, use_graph):
    ref = _ref(ph, n, 3)
    failed = []
    for blocks in range(8):
        mem = Allocator()
        ctx = _built(ph, n, use_graph=use_graph, arena_words=1, **mem.opts())
        ctx.reduce(max_passes=3)
        _check_pairs(ctx)
        mem.blocks = blocks
        try:
            ctx.reduce()
        except ph.PHError as err:
            assert err.code == -2
            mem.blocks = None
            _check_pairs(ctx)
            failed.append(_check_columns(ctx, ref))
        mem.blocks = None
        _finish(ctx, ref)
        ctx.close()
        assert mem.used == 0
    assert failed or n == 270


# budgets from the pass-by-pass run's need to look-ahead's, at every block that its call takes
def test_what_fits_pass_by_pass_fits(ph):
    n = 270
    ref = _ref(ph, n, 5)

    def run(mem, passes, **opts):
        ctx = _built(ph, n, **mem.opts(), **opts)
        built = len(mem.log)
        ctx.reduce(max_passes=5)
        _check_pairs(ctx)
        assert _check_columns(ctx, ref) == 5
        if passes < 0:
            _finish(ctx, ref)
        used = mem.log[built:]
        ctx.close()
        assert mem.used == 0
        return used

    for passes in (5, -1):
        least, most = Allocator(), Allocator()
        run(least, passes, collect_stats=True)
        used = run(most, passes)
        assert most.peak > least.peak
        for budget in sorted({least.peak, (least.peak + most.peak) // 2}
                             | {u for u in used if u > least.peak}):
            run(Allocator(budget=budget), passes)


# 3,126,250 edges of 2500 points: look-ahead is for triangles, edges keep to the memory (and the two to
# three times shorter time) of a pass-by-pass run
def test_edges_alone_take_no_look_ahead(ph):
    import torch

    x = torch.from_numpy(pc.random_cloud(2500, 3, 41)).cuda()
    out = []
    for opts in ({"collect_stats": True}, {}):
        mem = Allocator()
        ctx = ph.Context(**mem.opts(), **opts)
        ctx.build_filtration(x, None, 1)
        built = len(mem.log)
        assert ctx.reduce()["converged"]
        out.append((max(mem.log[built:]), ctx.filtration(0)["low"]))
        ctx.close()
    assert abs(out[0][0] - out[1][0]) < 1 << 20  # (the counters)
    assert np.array_equal(out[0][1], out[1][1])


# a first and a second call of up to two passes take no look-ahead (and its memory), a longer one or the
# third begins it; every state on the way is that of a pass-by-pass run with the same caps
@pytest.mark.parametrize("caps,ahead", [((0,), False), ((2,), False), ((3,), True), ((1, 3), False),
                                        ((0, 1), False), ((0, 4), True), ((1, 2, 3), True),
                                        ((2, -1), True)], ids=str)
@pytest.mark.parametrize("opts", [{}, {"use_graph": False}, {"dense_threshold": 1},
                                  {"predict_pairs": True}], ids=str)
def test_look_ahead_begins_with_a_long_call(ph, caps, ahead, opts):
    n, mem = 270, Allocator()
    got = _built(ph, n, **mem.opts(), **opts)
    ref = _built(ph, n, **{**opts, "collect_stats": True, "use_graph": False})
    built = len(mem.log)
    for i, cap in enumerate(caps):
        st = got.reduce(max_passes=cap)
        want = ref.reduce(max_passes=cap)
        assert st["passes"] == want["passes"] and st["converged"] == want["converged"]
        assert (max(mem.log[built:]) > 400 * got.m) == (ahead and i == len(caps) - 1)
        assert np.array_equal(got.filtration(0)["low"], ref.filtration(0)["low"])
        for a, b in zip(got.columns(0), ref.columns(0)):
            assert np.array_equal(a, b)
        assert np.array_equal(got.essential_estimate(0), ref.essential_estimate(0))
    _check_pairs(got)
    assert got.reduce()["passes"] == ref.reduce()["passes"]
    assert np.array_equal(got.filtration(0)["low"], ref.filtration(0)["low"])
    if "predict_pairs" in opts:
        assert np.array_equal(got.predicted_lows(0), ref.predicted_lows(0))


# the pairs that Corollary 10 predicts, of columns ahead of the pass and in the loop kernel
@pytest.mark.parametrize("n", [17, 40, 86, 270])
def test_predictions_equal_pass_by_pass(ph, n):
    ref = _built(ph, n, collect_stats=True, predict_pairs=True, use_graph=False)
    got = _built(ph, n, predict_pairs=True)
    for caps in ((0,), (1,), (4,), (8,), (9,), (-1,), (2, 3, 9, 10, -1)):
        for ctx in (ref, got):
            ctx.reset_reduction()
            for cap in caps:
                ctx.reduce(max_passes=cap)
        assert np.array_equal(ref.predicted_lows(0), got.predicted_lows(0)), caps
