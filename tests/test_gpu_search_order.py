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
