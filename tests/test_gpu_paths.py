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
# edge's vertex mask
@pytest.mark.parametrize("n,max_dim,cut", [
    (3, 2, -1), (4, 3, -1), (33, 2, -1), (64, 2, -1), (65, 2, -1), (65, 1, -1), (130, 2, 2.0),
    (5, 3, -1), (32, 3, -1), (33, 3, -1), (65, 3, 1.5), (33, 3, 0.2),
])
def test_direct_listing_equals_sorted_listing(ph, orc, n, max_dim, cut):
    x = pc.random_cloud(n, 2, 500 + n)
    cut2 = -1 if cut < 0 else int((cut * 65536) ** 2)
    K = orc.vr_build(x, max_dim, cut2)
    edges = K["diam2"][K["dim"] == 1]
    assert len(np.unique(edges)) == len(edges)  # no tie: the direct path
    alone = _build(ph.Context(), [x], max_dim, cut2)
    mixed = _build(ph.Context(), [TIED, x, x[: n // 2 + 1]], max_dim, cut2)  # sorted
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
