"""The search over the dictionary's search order (dictionaries of 65,536
entries or more, 20,000 queries or more): its neighbours and distances must be
the SIMT scan's, bit for bit, in the automatic form and the dense filter's in
the precision form, over the features, K, ragged sizes, several rounds of
queries and data whose duplicates overflow the candidate lists."""
import numpy as np
import pytest

import synth_inputs as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


class Limited:
    """An allocator that refuses requests above `limit` bytes."""

    def __init__(self):
        self.limit, self.refused, self.sizes = None, 0, []

    def alloc(self, nbytes, stream, user):
        self.sizes.append(int(nbytes))
        if self.limit is not None and nbytes > self.limit:
            self.refused += 1
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))

    def free(self, ptr, nbytes, stream, user):
        torch.cuda.caching_allocator_delete(ptr)


def _build(n_pairs, scale=2, patch=5, feature=0, w=4.0, n_train=10, L=8, k=12, flat=False, **kw):
    import paper_1004_3980_gb300 as Z
    train = [S.make_image(300 + i, 256, 256) for i in range(n_train)]
    if flat:   # half of every training image is one grey level: thousands of equal entries
        for im in train:
            im[:, :128] = 0.5
    lr = 256 // scale
    pos = S.sample_positions(5, n_train, lr, lr, patch, n_pairs)
    d = patch * patch * (2 if feature else 1)
    a, b = S.lsh_draws(6, L, k, d, w)
    A = Limited()
    ctx = Z.Context(0, allocator=A)
    ctx.test_allocator = A
    dic = Z.Dictionary(ctx, [torch.from_numpy(x).cuda() for x in train], pos, scale, patch, feature=feature)
    return ctx, Z.Index(dic, L, k, w, a, b, **kw)


def _check(ctx, ix, lr, K, **kw):
    import paper_1004_3980_gb300 as Z
    lr = torch.from_numpy(np.ascontiguousarray(lr)).cuda()
    A = ctx.test_allocator
    A.sizes = []
    got = Z.query(ix, lr, Z.UpscaleParams(K=K, **kw))
    st = ctx.stats()
    ctx.sync_status()
    if kw.get("precision"):   # its workspace refused, the search is the dense one
        A.limit, A.refused = max(A.sizes) - 1, 0
        ref = Z.query(ix, lr, Z.UpscaleParams(K=K, **kw))
        assert A.refused == 1
        A.limit = None
    else:
        ref = Z.query(ix, lr, Z.UpscaleParams(K=K, search=1))
    assert torch.equal(got["nbr"], ref["nbr"])
    assert torch.equal(got["dist"], ref["dist"])
    return st


@pytest.mark.parametrize("n_pairs", [65536, 70001, 100000])
@pytest.mark.parametrize("prec", [0, 1])
def test_sizes_of_the_dictionary(n_pairs, prec):
    ctx, ix = _build(n_pairs)
    st = _check(ctx, ix, S.make_image(1, 151, 163), 8, precision=prec)
    assert st["n_filter_fallback"] < 0.2 * st["n_queries"], st


@pytest.mark.parametrize("K", [1, 5, 12, 13, 16])
@pytest.mark.parametrize("prec", [0, 1])
def test_neighbour_counts(K, prec):
    ctx, ix = _build(66666)
    # one and two list sizes of the precision form (rerank_mult * K up to 16, to 32)
    for mult in (1, 2):
        _check(ctx, ix, S.make_image(2, 150, 152), K, precision=prec, rerank_mult=mult)


@pytest.mark.parametrize("patch,feature,w", [(3, 0, 4.0), (3, 1, 4.0), (5, 1, 8.0), (3, 2, 8.0), (5, 2, 8.0)])
@pytest.mark.parametrize("prec", [0, 1])
def test_features(patch, feature, w, prec):
    ctx, ix = _build(81234, patch=patch, feature=feature, w=w)
    _check(ctx, ix, S.make_image(3, 148, 160), 8, precision=prec)


@pytest.mark.parametrize("prec", [0, 1])
def test_several_rounds_of_queries_and_t_of_L(prec):
    # 300 x 290 image: 84,656 queries, two rounds of at most 65,280
    ctx, ix = _build(90001, min_table_hits=2)
    _check(ctx, ix, S.make_image(4, 300, 290), 8, precision=prec)


@pytest.mark.parametrize("prec", [0, 1])
def test_duplicates_overflow_the_candidate_lists(prec):
    ctx, ix = _build(70000, flat=True)
    lr = S.make_image(5, 150, 160)
    lr[:, :70] = 0.5
    st = _check(ctx, ix, lr, 8, precision=prec)
    assert st["n_filter_fallback"] > 0   # the flat queries have thousands of entries at distance 0


def test_refused_query_lists_fall_back_to_the_dense_search():
    import paper_1004_3980_gb300 as Z
    A = Limited()
    train = [S.make_image(300 + i, 256, 256) for i in range(10)]
    pos = S.sample_positions(5, 10, 128, 128, 5, 70000)
    a, b = S.lsh_draws(6, 8, 12, 25, 4.0)
    ctx = Z.Context(0, allocator=A)
    dic = Z.Dictionary(ctx, [torch.from_numpy(x).cuda() for x in train], pos, 2, 5)
    ix = Z.Index(dic, 8, 12, 4.0, a, b)
    lr = torch.from_numpy(S.make_image(1, 151, 163)).cuda()
    ref = Z.query(ix, lr, Z.UpscaleParams(K=8, search=1))
    A.sizes = []
    Z.query(ix, lr, Z.UpscaleParams(K=8))
    A.limit = max(A.sizes) - 1   # the search's workspace
    got = Z.query(ix, lr, Z.UpscaleParams(K=8))
    torch.cuda.synchronize()
    assert A.refused == 1
    assert torch.equal(got["nbr"], ref["nbr"]) and torch.equal(got["dist"], ref["dist"])


def test_index_without_room_for_the_search_order():
    import paper_1004_3980_gb300 as Z
    A = Limited()
    train = [S.make_image(300 + i, 256, 256) for i in range(10)]
    pos = S.sample_positions(5, 10, 128, 128, 5, 70000)
    a, b = S.lsh_draws(6, 8, 12, 25, 4.0)
    ctx = Z.Context(0, allocator=A)
    dic = Z.Dictionary(ctx, [torch.from_numpy(x).cuda() for x in train], pos, 2, 5)
    A.sizes = []
    ref = Z.Index(dic, 8, 12, 4.0, a, b)
    A.limit = max(A.sizes) - 1   # the index arrays with the order
    ix = Z.Index(dic, 8, 12, 4.0, a, b)
    assert A.refused == 1
    A.limit = None
    lr = torch.from_numpy(S.make_image(1, 151, 163)).cuda()
    for prec in (0, 1):
        p = Z.UpscaleParams(K=8, precision=prec)
        got, want = Z.query(ix, lr, p), Z.query(ref, lr, p)
        assert torch.equal(got["nbr"], want["nbr"]) and torch.equal(got["dist"], want["dist"])


def test_batch_equals_single_images():
    import paper_1004_3980_gb300 as Z
    ctx, ix = _build(70001)
    lrs = [torch.from_numpy(S.make_image(20 + i, h, w)).cuda() for i, (h, w) in enumerate([(64, 190), (33, 41), (180, 171)])]
    p = Z.UpscaleParams(K=8, bp_iters=2)
    ref = [Z.upscale(ix, x, p) for x in lrs]
    outs, _ = Z.upscale_batch([ix], lrs, p)
    outs, _ = Z.upscale_batch([ix], lrs, p, outs=outs)
    Z.batch_release(ctx)
    # the small image alone is searched densely, in the batch with the others
    for a, b in zip(outs, ref):
        assert torch.equal(a, b)
