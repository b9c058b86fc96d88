"""The search over the dictionary's search order: its routes."""
import numpy as np
import pytest

import synth_inputs as S
from tests.test_gpu_prune import _build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _equal(a, b):
    return torch.equal(a["nbr"], b["nbr"]) and torch.equal(a["dist"], b["dist"])


@pytest.mark.parametrize("prec", [0, 1])
def test_search_2_takes_the_dense_filter_in_both_forms(prec):
    # seen in the search's workspace, the call's largest allocation: the
    # query lists of the search order are several times the dense search's
    import paper_1004_3980_gb300 as Z
    ctx, ix = _build(70001)
    lr = torch.from_numpy(S.make_image(1, 151, 163)).cuda()
    got, size = [], []
    for search in (0, 2):
        ctx.test_allocator.sizes = []
        got.append(Z.query(ix, lr, Z.UpscaleParams(K=8, precision=prec, search=search)))
        size.append(max(ctx.test_allocator.sizes))
    assert size[1] < size[0] / 2
    assert _equal(*got)


@pytest.mark.parametrize("h,w", [(60, 71), (230, 201)])   # fewer than 152 x 256 queries, and a round and a part
@pytest.mark.parametrize("prm", [dict(search=2), dict(search=3), dict(precision=1, search=2)], ids=str)
def test_a_refused_dense_search_runs_in_two_parts(h, w, prm):
    import paper_1004_3980_gb300 as Z
    ctx, ix = _build(30001)
    A = ctx.test_allocator
    lr = torch.from_numpy(S.make_image(3, h, w)).cuda()
    A.sizes = []
    ref = Z.query(ix, lr, Z.UpscaleParams(K=8, **prm))
    A.limit, A.refused = max(A.sizes) - 1, 0
    got = Z.query(ix, lr, Z.UpscaleParams(K=8, **prm))
    torch.cuda.synchronize()
    assert A.refused == 1 and _equal(got, ref)
    A.limit = 1000   # no room at all
    with pytest.raises(Exception, match="OOM"):
        Z.query(ix, lr, Z.UpscaleParams(K=8, **prm))


@pytest.mark.parametrize("feature", [1, 2])
def test_features_of_50_values_are_searched_densely(feature):
    import paper_1004_3980_gb300 as Z
    ctx, ix = _build(70001, feature=feature, w=8.0)
    lr = torch.from_numpy(S.make_image(1, 151, 163)).cuda()
    got, sizes = [], []
    for search in (0, 2):
        ctx.test_allocator.sizes = []
        got.append(Z.query(ix, lr, Z.UpscaleParams(K=8, search=search)))
        sizes.append(ctx.test_allocator.sizes)
    assert sizes[0] == sizes[1]
    assert _equal(*got)


def _ramps(n, h, w, g):
    """n horizontal ramps of slope g (LR values, h x w) -> HR images of scale 2."""
    x = np.arange(2 * w, dtype=np.float64) / 2 * g
    return [np.ascontiguousarray(np.broadcast_to(x + 0.01 * i, (2 * h, 2 * w))).astype(np.float32) for i in range(n)]


def test_pieces_of_a_list_keep_the_chunks_one_piece_would():
    # A few queries (vertical ramps) are left to the dense filter, their lists
    # made in pieces.  Their nearest entries are thousands of patches of
    # horizontal ramps, equal but for the rounding of their features: hundreds
    # of chunks whose filter values d~ - ||q||^2 = ||c||^2 differ in the last
    # bits, and of which some are equal once ||q||^2 is added (the sum lies in
    # the next binade: 0.014 and 0.018 to 0.022 around 1/64).  All other
    # entries are farther (norms above 0.06).
    import paper_1004_3980_gb300 as Z
    from oracle import zoom_oracle as O
    P, n_ramp = 5, 4
    train = _ramps(n_ramp, 64, 64, (0.014 / 50) ** 0.5) + [3 * S.make_image(300 + i, 512, 512) for i in range(4)]
    pos, ramp = [], 0
    for m, im in enumerate(train):
        lr = O.degrade(im, 2, 0.8)
        f = np.lib.stride_tricks.sliding_window_view(np.asarray(lr), (P, P)).reshape(lr.shape[0] - P + 1, -1, P * P)
        n2 = ((f - f.mean(-1, keepdims=True)) ** 2).sum(-1)
        i, j = np.nonzero(n2 > 0.06) if m >= n_ramp else np.nonzero(n2 > 0)
        if m < n_ramp:   # away from the clamped edges
            keep = (j > 2) & (j < 56)
            i, j = i[keep], j[keep]
            ramp += len(i)
        pos.append(np.stack([np.full(len(i), m), i, j], 1))
    pos = np.concatenate(pos).astype(np.int32)
    assert len(pos) >= 70000
    ctx = Z.Context(0)
    d = Z.Dictionary(ctx, [torch.from_numpy(x).cuda() for x in train], pos, 2, P)
    a, b = S.lsh_draws(6, 8, 12, P * P, 4.0)
    ix = Z.Index(d, 8, 12, 4.0, a, b)
    img = 3 * S.make_image(1, 200, 200)
    for k in range(100):   # 100 patches, slopes of ||q||^2 from 0.004 to 0.008
        g = ((0.004 + 0.00004 * k) / 50) ** 0.5
        r, c = 20 * (k // 10) + 3, 20 * (k % 10) + 3
        img[r:r + P, c:c + P] = (0.5 + g * (np.arange(P) - 2))[:, None]
    lr = torch.from_numpy(np.ascontiguousarray(img)).cuda()
    got = Z.query(ix, lr, Z.UpscaleParams(K=8, precision=1, rerank_mult=2))
    left = ctx.stats()["n_filter_fallback"]
    ref = Z.query(ix, lr, Z.UpscaleParams(K=8, precision=1, rerank_mult=2, search=2))
    rows = [(20 * (k // 10) + 3) * 196 + 20 * (k % 10) + 3 for k in range(100)]
    assert int(got["nbr"][rows].max()) < ramp and left >= 100, left
    assert _equal(got, ref)


def _index_on(ctx, n_pairs, n_train=10, L=8, k=12, **kw):
    import paper_1004_3980_gb300 as Z
    train = [S.make_image(300 + i, 256, 256) for i in range(n_train)]
    pos = S.sample_positions(5, n_train, 128, 128, 5, n_pairs)
    a, b = S.lsh_draws(6, L, k, 25, 4.0)
    dic = Z.Dictionary(ctx, [torch.from_numpy(x).cuda() for x in train], pos, 2, 5)
    return Z.Index(dic, L, k, 4.0, a, b, **kw)


@pytest.mark.parametrize("memory", ["ordinary", "random bytes"])
@pytest.mark.parametrize("prec", [0, 1])
def test_waits_that_run_out_in_the_list_filter(prec, memory):
    # Every filter of the call withholds its accumulators' releases, so its
    # waits run out after 20 ms: reported, nothing followed outside the
    # dictionary (with random bytes in place of what was never written), and
    # the next call is the ordinary one's again.
    import paper_1004_3980_gb300 as Z
    from paper_1004_3980_gb300.capi import ZoomError
    from tests.test_gpu_faults import GarbageAllocator
    n = 65536
    ctx = Z.Context(0, allocator=GarbageAllocator()) if memory == "random bytes" else Z.Context(0)
    ix = _index_on(ctx, n)
    lr = torch.from_numpy(S.make_image(1, 150, 152)).cuda()
    p = Z.UpscaleParams(K=8, precision=prec)
    ref = Z.query(ix, lr, Z.UpscaleParams(K=8, precision=prec, search=2))
    ctx.sync_status()
    ctx.set_fault_injection(1, 20_000_000)
    try:
        r = Z.query(ix, lr, p)
        with pytest.raises(ZoomError, match="TIMEOUT"):
            ctx.sync_status()
    finally:
        ctx.set_fault_injection(0, 0)
    ctx.sync_status()
    assert int(r["nbr"].min()) >= 0 and int(r["nbr"].max()) < n
    assert _equal(Z.query(ix, lr, p), ref)
    ctx.sync_status()


@pytest.mark.parametrize("n_pairs,L,hits", [(150001, 16, 1), (300007, 12, 3)])
@pytest.mark.parametrize("prec", [0, 1])
def test_many_super_tiles(n_pairs, L, hits, prec):
    # more than 32 super tiles (131,072 entries): the visits' parts, the
    # seeds' second key a lane, ragged last tiles of both kinds
    import paper_1004_3980_gb300 as Z
    ctx = Z.Context(0)
    ix = _index_on(ctx, n_pairs, n_train=21, L=L, k=14, min_table_hits=hits)
    lr = torch.from_numpy(S.make_image(7, 260, 271)).cuda()
    a = Z.query(ix, lr, Z.UpscaleParams(K=7, precision=prec))
    b = Z.query(ix, lr, Z.UpscaleParams(K=7, precision=prec, search=2 if prec else 1))
    ctx.sync_status()
    assert _equal(a, b)


@pytest.mark.parametrize("prec", [0, 1])
def test_pixels_that_are_no_numbers(prec):
    # NaN, infinite and very large pixels: their queries find what the scan
    # finds, and the others beside them too
    import paper_1004_3980_gb300 as Z
    ctx = Z.Context(0)
    ix = _index_on(ctx, 70001)
    img = S.make_image(1, 180, 170)
    img[20, 30], img[21, 90], img[100, 5], img[150, 150] = np.nan, np.inf, -np.inf, 1e30
    img[60, 60], img[120:124, 40:44] = 300.0, 1e6
    lr = torch.from_numpy(img).cuda()
    a = Z.query(ix, lr, Z.UpscaleParams(K=8, precision=prec))
    b = Z.query(ix, lr, Z.UpscaleParams(K=8, precision=prec, search=2 if prec else 1))
    ctx.sync_status()
    assert torch.equal(a["nbr"], b["nbr"])
    assert torch.equal(a["dist"].view(torch.int32), b["dist"].view(torch.int32))


@pytest.mark.parametrize("prec,n_pairs,h,w", [(0, 200_003, 280, 281), (1, 120_001, 260, 281)])
def test_noise_is_given_up_for_the_dense_filters(prec, n_pairs, h, w):
    # Uniform noise: a query's radius reaches nearly every tile's box.  Every
    # round is given up (all its queries counted as left), and the dense
    # filters find the scan's and the dense search's neighbours.
    import paper_1004_3980_gb300 as Z
    g = np.random.default_rng(8)
    n_train = n_pairs // 15000 + 1
    train = [torch.from_numpy(g.random((256, 256), dtype=np.float32)).cuda() for _ in range(n_train)]
    ctx = Z.Context(0)
    dic = Z.Dictionary(ctx, train, S.sample_positions(5, n_train, 128, 128, 5, n_pairs), 2, 5)
    a, b = S.lsh_draws(6, 8, 12, 25, 64.0)
    ix = Z.Index(dic, 8, 12, 64.0, a, b)
    lr = torch.from_numpy(g.random((h, w), dtype=np.float32)).cuda()
    got = Z.query(ix, lr, Z.UpscaleParams(K=8, precision=prec))
    st = ctx.stats()
    ref = Z.query(ix, lr, Z.UpscaleParams(K=8, precision=prec, search=2 if prec else 1))
    ctx.sync_status()
    assert st["n_filter_fallback"] == st["n_queries"] == (h - 4) * (w - 4)
    assert _equal(got, ref)


@pytest.mark.parametrize("L,k,n_pairs", [(1, 1, 65_536), (2, 3, 150_001), (16, 16, 65_537)])
def test_a_hash_shorter_than_the_trees_first_levels(L, k, n_pairs):
    # the index build launches the two beside each other
    import paper_1004_3980_gb300 as Z
    ctx, ix = _build(n_pairs, L=L, k=k)
    lr = torch.from_numpy(S.make_image(5, 163, 151)).cuda()
    got = [Z.query(ix, lr, Z.UpscaleParams(K=8, search=search)) for search in (0, 2)]
    assert _equal(*got)
