"""Sums over patches: the one-pass overlap average against the two-pass form
(the same bits) at the edges of its tiles, and the dictionary gradient of
entries with few and with thousands of uses against FP64."""
import numpy as np
import pytest

import synth_inputs as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _index(scale, patch, n):
    import paper_1004_3980_gb300 as Z
    train = [torch.from_numpy(S.make_image(300, 48 * scale, 48 * scale)).cuda()]
    ctx = Z.Context(0)
    d = Z.Dictionary(ctx, train, S.sample_positions(5, 1, 48, 48, patch, n), scale, patch)
    a, b = S.lsh_draws(6, 2, 4, patch * patch, 4.0)
    return Z.Index(d, 2, 4, 4.0, a, b)


def _uses(h, w, patch, n, K, seed):
    g = np.random.default_rng(seed)
    nq = (h - patch + 1) * (w - patch + 1)
    nbr = g.integers(0, n, (nq, K))
    nbr[g.random((nq, K)) < 0.5] = 3           # half of the uses are one entry's
    wgt = g.standard_normal((nq, K)).astype(np.float32)
    mu = g.random(nq).astype(np.float32)
    return (torch.from_numpy(nbr.astype(np.int32)).cuda(), torch.from_numpy(wgt).cuda(), torch.from_numpy(mu).cuda())


@pytest.mark.parametrize("scale,patch,h,w,K", [(1, 3, 3, 3, 1), (2, 5, 5, 33, 8), (3, 5, 40, 31, 9), (4, 5, 7, 65, 16),
                                               (2, 3, 64, 37, 64), (4, 5, 6, 32, 64)])
def test_one_pass_overlap_average_is_the_two_pass_one(scale, patch, h, w, K):
    import paper_1004_3980_gb300 as Z
    ix = _index(scale, patch, 300)
    nbr, wgt, mu = _uses(h, w, patch, 300, K, 1)
    two = Z.reconstruct(ix, nbr, wgt, mu, h, w)
    one = Z.reconstruct_with(ix, Z.dictionary_hr(ix.dictionary), nbr, wgt, mu, h, w)
    assert torch.equal(one, two)


@pytest.mark.parametrize("scale,patch,h,w,K", [(1, 3, 3, 3, 1), (1, 3, 20, 21, 2), (2, 5, 30, 31, 3), (3, 5, 47, 52, 8),
                                               (4, 5, 40, 45, 16)])
def test_dictionary_gradient_of_entries_with_many_uses(scale, patch, h, w, K):
    import paper_1004_3980_gb300 as Z
    n = 300
    ix = _index(scale, patch, n)
    nbr, wgt, mu = _uses(h, w, patch, n, K, 2)
    R = Z.dictionary_hr(ix.dictionary).requires_grad_(True)
    x = Z.ReconstructFunction.apply(R, ix, nbr, wgt, mu, h, w)
    g = torch.from_numpy(np.random.default_rng(3).standard_normal(tuple(x.shape)).astype(np.float32)).cuda()
    (got,) = torch.autograd.grad(x, R, g)
    PH = scale * patch
    unf = lambda t: torch.nn.functional.unfold(t[None, None], PH, stride=scale)[0].T   # [nq][PH^2]
    ones = torch.ones_like(g, dtype=torch.float64)
    cov = torch.nn.functional.fold(unf(ones).T[None], x.shape, PH, stride=scale)[0, 0]
    gP = unf(g.double() / cov)
    terms = wgt.double()[:, :, None] * gP[:, None, :]                                  # [nq][K][PH^2]
    flat = nbr.long().reshape(-1)
    ref = torch.zeros((n, PH * PH), dtype=torch.float64, device="cuda").index_add_(0, flat, terms.reshape(-1, PH * PH))
    size = torch.zeros_like(ref).index_add_(0, flat, terms.abs().reshape(-1, PH * PH))
    uses = torch.bincount(flat, minlength=n).double()[:, None]
    # each of a sum's operations rounds to half an ulp of at most the terms' sizes
    bound = (uses + 20) * 2.0 ** -24 * size + 1e-30
    assert ((got.double() - ref).abs() <= bound).all()
    assert torch.equal(got, torch.autograd.grad(Z.ReconstructFunction.apply(R, ix, nbr, wgt, mu, h, w), R, g)[0])
