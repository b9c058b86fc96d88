"""The overlap term of the MAP energy alone against FP64 of the same FP32
patches: one neighbour a patch with a fixed weight, so that the patches are
mu + w R rounded once.  65,536 threads sum 3.8M values (three groups of
sixteen a thread and more); a sum of n non-negative FP64 terms in any order
is within n 2^-53 of itself, and no chain here is longer than 600 terms: 1e-12
with room."""
import numpy as np
import pytest

import synth_inputs as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# weights whose differences' squares lie inside FP32's range, below and above it
@pytest.mark.parametrize("weight", [1.0, 1e-22, 1e21])
def test_overlap_term_in_fp64(weight):
    import paper_1004_3980_gb300 as Z
    h, w, s, P, n = 201, 199, 2, 5, 500
    ctx = Z.Context(0)
    train = [torch.from_numpy(S.make_image(300, 96, 96)).cuda()]
    d = Z.Dictionary(ctx, train, S.sample_positions(5, 1, 48, 48, P, n), s, P)
    ix = Z.Index(d, 2, 4, 4.0, *S.lsh_draws(6, 2, 4, 25, 4.0))
    img = S.make_image(301, h, w) if weight == 1.0 else np.zeros((h, w), np.float32)
    lr = torch.from_numpy(img).cuda()
    nh, nw, PH = h - P + 1, w - P + 1, s * P
    nbr = np.random.default_rng(3).integers(0, n, (nh * nw, 1)).astype(np.int32)
    wgt = torch.full((nh * nw, 1), weight, dtype=torch.float32, device="cuda")
    mu = Z.query(ix, lr, Z.UpscaleParams(K=1))["mu"].cpu().numpy()
    tn = torch.from_numpy(nbr).cuda()
    lam = float(1 << 20)
    e = [Z.map_energy_grads(ix, lr, tn, wgt, lam=v)["energy"] for v in (0.0, lam)]
    got = (e[1] - e[0]) / lam
    R = Z.dictionary_hr(d).cpu().numpy()[nbr[:, 0]]
    # (weight 1: one rounding; else mu = 0: one rounding)
    p = (R + mu[:, None] if weight == 1.0 else R * np.float32(weight)).astype(np.float32)
    p = p.reshape(nh, nw, PH, PH).astype(np.float64)
    ref = ((p[:, :-1, :, s:] - p[:, 1:, :, :-s]) ** 2).sum() + ((p[:-1, :, s:, :] - p[1:, :, :-s, :]) ** 2).sum()
    assert ref > 0 and abs(got - ref) <= 1e-12 * ref, (got, ref, got / ref - 1)
