"""The size- and content-dependent paths of the device code, each against another path or the oracle.

All of it is integer work, so every comparison is exact.
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


@pytest.fixture(scope="module")
def orc():
    import oracle

    oracle.build_lib()
    return oracle


def _build(ctx, clouds, max_dim, cut=-1):
    import torch

    x = torch.from_numpy(np.ascontiguousarray(np.concatenate(clouds), np.int32)).cuda()
    off = np.concatenate([[0], np.cumsum([len(c) for c in clouds])]).astype(np.int64)
    ctx.build_filtration(x, off if len(clouds) > 1 else None, max_dim, cut)
    return ctx


def _r0(ctx, cloud):
    ctx.reduce(max_passes=0)
    return ctx.columns(cloud)


TIED = np.array([[0, 0], [1, 0], [2, 0], [3, 0]], np.int32)  # equal edges: sorted candidates


# clouds without two edges of one length list triangles and tetrahedra per edge, without a sort;
# a batch with a tie in any cloud sorts all candidates. 64 and 65 points have 2016 and 2080 edges,
# around one 2048-element sort and scan tile; 33 and 65 points take a second and third word of an
# edge's vertex mask; 200 points have 19900 edges, listed by warps of two
@pytest.mark.parametrize("n,max_dim,cut", [
    (3, 2, -1), (4, 3, -1), (33, 2, -1), (64, 2, -1), (65, 2, -1), (65, 1, -1), (130, 2, 2.0),
    (200, 2, -1), (5, 3, -1), (32, 3, -1), (33, 3, -1), (65, 3, 1.5), (33, 3, 0.2),
])
def test_direct_listing_equals_sorted_listing(ph, orc, n, max_dim, cut):
    x = pc.random_cloud(n, 2 if n < 200 else 3, 500 + n)  # (the 200 points tie in the plane)
    cut2 = -1 if cut < 0 else int((cut * 65536) ** 2)
    K = orc.vr_build(x, max_dim, cut2)
    edges = K["diam2"][K["dim"] == 1]
    assert len(np.unique(edges)) == len(edges)  # no tie: the direct path
    alone = _build(ph.Context(), [x], max_dim, cut2)
    tied = np.pad(TIED, ((0, 0), (0, x.shape[1] - 2)))
    mixed = _build(ph.Context(), [tied, x, x[: n // 2 + 1]], max_dim, cut2)  # sorted
    batch = _build(ph.Context(), [x[: n // 2 + 1], x], max_dim, cut2)  # direct, several clouds
    fa, fm, fb = alone.filtration(0), mixed.filtration(1), batch.filtration(1)
    assert np.array_equal(fa["beta"], orc.beta(K))
    for k in ("dim", "diam2", "verts", "beta", "low"):
        assert np.array_equal(fa[k], fm[k]) and np.array_equal(fa[k], fb[k]), k
    for k in ("dim", "diam2", "verts"):
        assert np.array_equal(fa[k], K[k]), k
    ca, cm, cb = _r0(alone, 0), _r0(mixed, 1), _r0(batch, 1)
    for i in (0, 1):
        assert np.array_equal(ca[i], cm[i]) and np.array_equal(ca[i], cb[i])


# one block sorts up to 2048, 4096 or 8192 edges of a cloud (64, 91 and 128 points have 2016, 4095 and
# 8128); above, and with several truncated clouds, all edges are sorted over the whole device
@pytest.mark.parametrize("sizes", [[64], [65], [91], [92], [128], [129], [3, 1, 128, 2, 64],
                                   [129, 1, 2]])
@pytest.mark.parametrize("cut", [-1, 65536 ** 2])
def test_edge_sort_sizes(ph, orc, sizes, cut):
    clouds = [pc.lattice_cloud(n, 2, 700 + n, side=40) for n in sizes]  # with ties: stable
    ctx = _build(ph.Context(), clouds, 1, cut)
    for c, x in enumerate(clouds):
        K, f = orc.vr_build(x, 1, cut), ctx.filtration(c)
        assert np.array_equal(f["diam2"], K["diam2"]) and np.array_equal(f["verts"], K["verts"])


def test_long_sort_clears_its_states(ph):
    """12,259,940 triangles by three digits: one digit's tile states at a time."""
    n = 420
    x = pc.random_cloud(n, 3, 77).astype(np.int64)
    x[1] = 2 * x[0] - x[2]  # x0 halfway between x1 and x2: a tie, so candidates are sorted
    ctx = _build(ph.Context(), [x], 2)
    f = ctx.filtration(0)
    tri = f["dim"] == 2
    d2 = ((x[:, None] - x[None]) ** 2).sum(-1)
    i, j, k = f["verts"][tri, :3].T.astype(np.int64)
    want = np.maximum(np.maximum(d2[i, j], d2[i, k]), d2[j, k])
    assert len(want) == 12_259_940 and (i < j).all() and (j < k).all()
    assert np.array_equal(f["diam2"][tri], want) and (np.diff(want) >= 0).all()
    code = (i * n + j) * n + k  # ties in lexicographic order, so no triangle twice
    assert (np.diff(code)[np.diff(want) == 0] > 0).all()


# 1024 and 4096 ids are a writer's round and a scan's tile; 235 points have more than 2^21 ids (long
# rounds); three hundred clouds put many segments, some empty, into one tile
@pytest.mark.parametrize("sizes,max_dim,passes", [
    ([1], 2, -1), ([2, 1, 1], 2, -1), ([18, 1], 2, -1), ([25], 3, -1), ([29, 30], 2, 1),
    ([1 + i % 6 for i in range(300)], 2, -1), ([235], 2, 2),
])
def test_extraction_routes(ph, sizes, max_dim, passes):
    import ctypes

    import torch

    clouds = [pc.random_cloud(n, 3, 900 + i) for i, n in enumerate(sizes)]
    ctx = _build(ph.Context(), clouds, max_dim)
    ctx.reduce(max_passes=passes)
    pr, es = ctx.pairs(-1), ctx.essential(-1)  # written straight into the tensors
    pr = {k: v.cpu().numpy() for k, v in pr.items()}
    es = {k: v.cpu().numpy() for k, v in es.items()}
    want_p = {k: [] for k in pr}
    want_e = {k: [] for k in es}
    for c in range(len(sizes)):
        f = ctx.filtration(c)
        order = np.argsort(f["dim"], kind="stable")  # (dimension, index)
        death = order[f["low"][order] >= 0]
        birth = f["low"][death]
        is_low = np.zeros(len(order), bool)
        is_low[birth] = True
        e = order[(f["low"][order] < 0) & ~is_low[order]]
        one = dict(birth=birth, death=death, dim=f["dim"][birth], birth_diam2=f["diam2"][birth],
                   death_diam2=f["diam2"][death])
        onee = dict(idx=e, dim=f["dim"][e], diam2=f["diam2"][e])
        for w, o in ((want_p, one), (want_e, onee)):
            for k, v in o.items():
                w[k].append(v)
        if c in (0, len(sizes) - 1):  # internal arrays and copies
            for host in (False, True):
                got = {**{"p" + k: v for k, v in ctx.pairs(c, not host).items()},
                       **{"e" + k: v for k, v in ctx.essential(c, not host).items()}}
                for k, v in [("p" + k, v) for k, v in one.items()] + [
                        ("e" + k, v) for k, v in onee.items()]:
                    assert np.array_equal(got[k].cpu().numpy(), v), k
    for w, o in ((want_p, pr), (want_e, es)):
        for k in o:
            assert np.array_equal(o[k], np.concatenate(w[k])), k
    # an array off its type's alignment, and one left out, in a fresh extraction
    ctx2 = _build(ph.Context(), clouds, max_dim)
    ctx2.reduce(max_passes=passes)
    n = ctypes.c_int64(len(pr["death"]))
    for shift in (0, 1):
        raw = torch.zeros(2 * n.value + 1, dtype=torch.int32, device="cuda")
        rc = ctx2.lib.ph_get_pairs(ctx2._h, -1, None, ctypes.c_void_p(raw.data_ptr() + 4 * shift),
                                   None, None, None, n.value, ctypes.byref(n), 1)
        assert rc == 0
        got = raw[shift:2 * n.value + shift].cpu().numpy().view(np.int64)
        assert np.array_equal(got, pr["death"])


# pairs are listed 2048 columns at a time and taken 256 at a time: 65 points have 2080 edges, 30 points
# 4060 triangles and 406 pairs; points on the grid, so the 64-bit lengths come from the pairs
@pytest.mark.parametrize("sizes,dim", [([65], 0), ([2, 65, 3, 30], 0), ([30, 3, 5], 1), ([3], 1),
                                       ([40, 12], 1)])
def test_diagram_loss_rounds(ph, sizes, dim):
    import torch

    clouds = [pc.random_cloud(n, 3, 1300 + n) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    x = torch.from_numpy((np.concatenate(clouds) / 65536).astype(np.float32)).cuda()
    ctx = ph.Context()
    ctx.build_filtration_f32(x, off if len(sizes) > 1 else None, dim + 1)
    ctx.reduce()
    loss = ctx.diagram_loss(x, dim).cpu().numpy()
    w = torch.arange(1, len(sizes) + 1, dtype=torch.float32, device="cuda")
    grad = ctx.diagram_backward(x, w, dim).cpu().numpy()
    n_pairs = 0
    for c in range(len(sizes)):
        pr = ctx.pairs(c, on_device=False)
        sel = pr["dim"].numpy() == dim
        b, d = (np.sqrt(pr[k].numpy()[sel].astype(np.float64)) / 65536
                for k in ("birth_diam2", "death_diam2"))
        n_pairs += len(d)
        want = ((d - b) ** 2).sum()
        # a length is off by 4 roundings at most, a sum of positive terms by one per addition
        bound = 2 ** -24 * (8 * (np.abs(d - b) * (d + b)).sum() + (len(d) / 256 + 16) * want)
        assert abs(loss[c] - want) <= bound
        # the gradient moves points along edges: it sums to zero, up to one rounding per addition
        g = grad[off[c]:off[c + 1]]
        size = 4 * (c + 1) * np.abs(d - b).sum()
        assert np.abs(g.sum(0)).max() <= 2 ** -24 * (len(d) + 8) * max(size, 1e-30)
    assert ctx.last_pairs == n_pairs


def _state(ctx, cloud=0):
    ptr, rows = ctx.columns(cloud)
    return ctx.filtration(cloud)["low"], ptr, rows, ctx.essential_estimate(cloud)


def _same_reduction(ph, build, opts, caps, cloud=0):
    """A context with per-pass counters takes every pass of every column, in k_add."""
    ref = ph.Context(**{**opts, "collect_stats": True, "use_graph": False})
    got = ph.Context(**opts)
    for ctx in (ref, got):
        build(ctx)
    for cap in caps:
        st = []
        for ctx in (ref, got):
            ctx.reset_reduction()
            st.append(ctx.reduce(max_passes=cap))
        assert st[0]["passes"] == st[1]["passes"] and st[0]["converged"] == st[1]["converged"]
        for r, g in zip(_state(ref, cloud), _state(got, cloud)):
            assert np.array_equal(r, g), (opts, cap)
    for ctx in (ref, got):  # in steps: a call resumes where the last one stopped
        ctx.reset_reduction()
        for cap in (2, 3, 9, 10):
            ctx.reduce(max_passes=cap)
        ctx.reduce()
    for r, g in zip(_state(ref, cloud), _state(got, cloud)):
        assert np.array_equal(r, g), opts


# from 3,000,000 columns of at most three rows a visit runs up to eight passes of a column; a cap,
# a horizon of eight passes, zeroing rules, bit-packed columns and space stops cut through that
@pytest.mark.parametrize("opts", [
    {}, {"strict_phase2": True}, {"use_cor10": False}, {"dense_threshold": 1}, {"arena_words": 1},
    {"use_graph": False}, {"predict_pairs": True},
], ids=str)
def test_look_ahead_equals_pass_by_pass(ph, opts):
    x = pc.to_grid(pc.sphere(270, np.random.Generator(np.random.PCG64(3)), noise=0.05))
    _same_reduction(ph, lambda c: _build(c, [x], 2), opts, (1, 7, 8, 9, -1))


def test_look_ahead_of_a_batch(ph):
    clouds = [pc.random_cloud(60 + i % 17, 3, 1500 + i) for i in range(64)]
    assert sum(len(c) * (len(c) - 1) * (len(c) - 2) // 6 for c in clouds) > 3_000_000
    _same_reduction(ph, lambda c: _build(c, clouds, 2), {}, (4, -1), cloud=37)


# the loop kernel: 1, 4, 8 or 32 columns per warp (8, 32, 64 columns, then 8 per warp of up to 64
# blocks), one block up to 64 columns, several tiles per block above 77,824 (86 points, 106,081), and 93
# points (134,230 columns) that begin in the pass graph; a lack of space stops it within a pass
@pytest.mark.parametrize("n", [3, 4, 5, 7, 8, 12, 17, 40, 86, 93])
@pytest.mark.parametrize("opts", [{}, {"arena_words": 1}, {"predict_pairs": True}], ids=str)
def test_loop_kernel_equals_host_loop(ph, n, opts):
    x = pc.random_cloud(n, 2, 1700 + n)
    _same_reduction(ph, lambda c: _build(c, [x], 2), opts, (0, 1, 3, -1))


def test_rebuilt_contexts(ph):
    """Blocks, graphs and pinned memory that a context keeps hold nothing of an earlier build."""
    ctx = ph.Context()
    for i, (n, max_dim) in enumerate([(93, 2), (93, 2), (40, 2), (93, 2), (30, 3), (95, 2), (93, 2)]):
        x = pc.random_cloud(n, 3, 1900 + i)
        fresh = _build(ph.Context(), [x], max_dim)
        _build(ctx, [x], max_dim)
        assert ctx.reduce()["passes"] == fresh.reduce()["passes"]
        for r, g in zip(_state(fresh), _state(ctx)):
            assert np.array_equal(r, g)
        for a, b in ((fresh.pairs(), ctx.pairs()), (fresh.essential(), ctx.essential())):
            assert all(np.array_equal(a[k].cpu(), b[k].cpu()) for k in a)


def test_look_ahead_without_room_runs_pass_by_pass(ph):
    """Its arrays take 360 bytes per column: a refused one (96 bytes per column) leaves the rest."""
    import torch

    refused = []

    def alloc(nbytes, stream):
        if nbytes > 250 << 20:
            refused.append(nbytes)
            return 0
        return torch.cuda.caching_allocator_alloc(nbytes, stream=stream)

    x = pc.to_grid(pc.sphere(270, np.random.Generator(np.random.PCG64(3)), noise=0.05))
    ref = _build(ph.Context(), [x], 2)
    got = _build(ph.Context(device_alloc=alloc, device_free=torch.cuda.caching_allocator_delete),
                 [x], 2)
    assert not refused
    assert got.reduce(max_passes=5)["passes"] == ref.reduce(max_passes=5)["passes"] == 5
    assert refused
    for r, g in zip(_state(ref), _state(got)):
        assert np.array_equal(r, g)


# read-out of columns: up to eight rows by a lane, longer ones and bitmaps by the warp, 32 columns at a time
@pytest.mark.parametrize("n", [1, 31, 32, 33, 97])
def test_columns_of_all_lengths(ph, n):
    rng = np.random.default_rng(n)
    rows0 = 400
    length = rng.choice([0, 1, 7, 8, 9, 31, 32, 33, 64, 200], n)
    cols = [np.sort(rng.choice(rows0, k, replace=False)) for k in length]
    dims = np.repeat(np.array([0, 1], np.int32), [rows0, n])
    colptr = np.concatenate([np.zeros(rows0, np.int64), [0], np.cumsum(length)])
    rows = np.concatenate(cols + [[]]).astype(np.int32)
    ctx = ph.Context(use_cor10=False)
    ctx.load_boundary(dims, colptr, rows)
    ctx.reduce(max_passes=0)  # no addition: the columns as they were loaded
    ptr, got = ctx.columns(0)
    assert np.array_equal(ptr, colptr) and np.array_equal(got, rows)
    full = []
    for threshold in (-1, 1):  # reduced, as rows and as bitmaps
        c = ph.Context(dense_threshold=threshold)
        c.load_boundary(dims, colptr, rows)
        c.reduce()
        full.append(c.columns(0))
    assert all(np.array_equal(a, b) for a, b in zip(*full))


# a pass of more than 2^20 arena words goes back to the pass graph, one of half as many on to the loop kernel:
# random columns of three rows fill in, and thin out at the end
@pytest.mark.parametrize("opts", [{}, {"dense_threshold": -1}, {"arena_words": 1}], ids=str)
def test_loop_kernel_hands_long_columns_back(ph, opts):
    rows0, n = 6000, 10000
    rng = np.random.default_rng(5)
    cols = np.sort(rng.integers(0, rows0, (n, 3)), axis=1)
    cols = cols[(np.diff(cols, axis=1) > 0).all(1)]
    dims = np.repeat(np.array([0, 1], np.int32), [rows0, len(cols)])
    colptr = np.concatenate([np.zeros(rows0, np.int64), 3 * np.arange(len(cols) + 1)])

    def load(ctx):
        ctx.load_boundary(dims, colptr, cols.reshape(-1).astype(np.int32))

    _same_reduction(ph, load, opts, (200, -1))
    ctx = ph.Context(**opts)
    load(ctx)
    before = ctx.kernel_launches()
    ctx.reduce()
    assert ctx.kernel_launches() - before > 300  # three kernels for each of the graph's passes
