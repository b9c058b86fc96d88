"""The work that a user of this package has it do, as cases that can be timed.

A case is a dict of plain values.  Its "kind" names the public call:

  zoom      upscale: the whole zoom of one LR image
  query     query: the per-patch steps alone (neighbours, weights)
  batch     upscale_batch: many LR images of mixed sizes and scales in one call
  backproj  backproject: the error back-projection of an HR estimate
  energy    map_energy_grads: MAP energy and its gradients, neighbours fixed
  train     one autograd step of the HR dictionary through the reconstruction
            and the degradation (neighbours fixed)
  build     a dictionary and its index from training images, then the first
            zoom with them

Images follow the recipe of synth_inputs.py (oriented sinusoids, ellipses,
noise, quantised to 8 bits), made on the GPU from the seed.  `exact` restates
the method in plain torch at 64 bits; it uses nothing of the package.
"""
import math

import numpy as np
import torch

import paper_1004_3980_gb300 as Z

BLUR = 0.8
REG = 1e-3
SIGMA_SP, SIGMA_R, RADIUS = 1.5, 0.1, 3


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _zoom(name, h, w, scale, n_pairs, **kw):
    c = {"name": name, "kind": "zoom", "h": h, "w": w, "scale": scale, "patch": 5, "n_pairs": n_pairs, "L": 16,
         "k": 16, "K": 8, "bin": 4.0, "feature": 0, "bp": 5, "precision": 0, "mult": 2, "cap": 0}
    c.update(kw)
    return c


def listed():
    return [
        # a thumbnail against a small dictionary of 3x3 patches: the smallest
        # call, all launches and latency
        _zoom("zoom2x_64_dict20k", 64, 64, 2, 20_000, patch=3, L=8, k=12, K=5, bp=3),
        # the method's ordinary size: a 512 x 512 image, a million pairs,
        # exact neighbours
        _zoom("zoom2x_512_dict1m", 512, 512, 2, 1_000_000),
        # the benchmark's workload: full HD to 6K, four million pairs, the
        # BF16 form with the best 32 chunks -- the largest call
        _zoom("zoom3x_1920x1080_dict4m_bf16", 1080, 1920, 3, 4_000_000, k=18, precision=1, mult=4),
        # a small photograph zoomed by 4 against 300,000 pairs, the training-set
        # size of the paper's 4x example
        _zoom("zoom4x_280_dict300k", 280, 280, 4, 300_000),
        # odd sizes everywhere: image sides, dictionary, BF16 with 16 chunks
        _zoom("zoom3x_637x419_dict777k_bf16", 419, 637, 3, 777_777, precision=1),
        # the paper's early stop at 3L candidates on the largest image
        _zoom("zoom3x_1920x1080_dict4m_cap48", 1080, 1920, 3, 4_000_000, k=18, cap=48),
        # first-order gradient features (50 values a patch): neighbours and
        # weights for a caller that does its own blending
        _zoom("query2x_gradient_523x307_dict500k", 307, 523, 2, 500_000, kind="query", feature=1, bin=8.0),
        # a queue of images of mixed sizes and two scales in one call, one
        # dictionary per scale
        {"name": "batch16_mixed_dict250k", "kind": "batch", "n_images": 16, "min_side": 96, "max_side": 768,
         "patch": 5, "n_pairs": 250_000, "L": 16, "k": 16, "K": 8, "bin": 4.0, "feature": 0, "bp": 5,
         "precision": 1, "mult": 2, "cap": 0},
        # refinement of an HR estimate that came from elsewhere
        {"name": "backproj3x_1920x1080", "kind": "backproj", "h": 1080, "w": 1920, "scale": 3, "bp": 5},
        # MAP energy and its gradients over every dictionary entry
        {"name": "energy2x_256_dict64k", "kind": "energy", "h": 256, "w": 256, "scale": 2, "patch": 5,
         "n_pairs": 65_536, "K": 8},
        # one training step of the HR dictionary, ragged sizes
        {"name": "train3x_301x407_dict150k", "kind": "train", "h": 407, "w": 301, "scale": 3, "patch": 5,
         "n_pairs": 150_000, "K": 8},
        # new training images: dictionary, index and the first small zoom
        _zoom("build2x_dict1m", 96, 128, 2, 1_000_000, kind="build"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["zoom", "zoom", "zoom", "query", "batch", "backproj", "energy", "train", "build"])
    if kind == "batch":
        return {"kind": "batch", "n_images": rng.randint(2, 20), "min_side": rng.randint(24, 128),
                "max_side": rng.randint(256, 768), "patch": rng.choice([3, 5, 5]),
                "n_pairs": _log_int(rng, 8_000, 400_000), "L": 16, "k": 16, "K": rng.randint(3, 8), "bin": 4.0,
                "feature": 0, "bp": rng.randint(1, 6), "precision": rng.choice([0, 1]), "mult": 2, "cap": 0}
    scale = rng.choice([2, 2, 3, 4])
    if kind == "backproj":
        return {"kind": kind, "h": _log_int(rng, 17, 1080), "w": _log_int(rng, 17, 1920), "scale": scale,
                "bp": rng.randint(1, 8)}
    if kind in ("energy", "train"):
        return {"kind": kind, "h": _log_int(rng, 24, 512), "w": _log_int(rng, 24, 512), "scale": scale,
                "patch": rng.choice([3, 5]), "n_pairs": _log_int(rng, 8_000, 200_000), "K": rng.randint(3, 12)}
    feature = rng.choice([0, 0, 0, 1, 2]) if kind != "build" else 0
    K = rng.randint(3, 12)
    cap = rng.choice([0, 0, 0, 48, 96])
    precision = rng.choice([0, 1])
    c = {"kind": kind, "scale": scale, "patch": rng.choice([3, 5, 5]), "n_pairs": _log_int(rng, 8_000, 2_000_000),
         "L": rng.choice([8, 16]), "k": rng.randint(12, 18), "K": K, "bin": 4.0 if feature == 0 else 8.0,
         "feature": feature, "bp": rng.randint(1, 6), "precision": precision,
         "mult": rng.choice([m for m in (1, 2, 4) if m * K <= 32]), "cap": cap}
    if kind == "build":
        c.update(h=_log_int(rng, 24, 200), w=_log_int(rng, 24, 200), cap=0)
    else:
        c.update(h=_log_int(rng, 17, 900), w=_log_int(rng, 17, 1200))
    if cap or kind == "query":
        c["precision"] = 0   # a caller of query wants the exact neighbours; the early stop has one form
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _images(seed, n, h, w):
    """n images float32 [n][h][w] on the GPU (the recipe of synth_inputs.make_image)."""
    rng = np.random.Generator(np.random.PCG64([int(seed) & 0xFFFFFFFF, n, h, w]))
    dev = torch.device("cuda")

    def par(lo, hi):
        return torch.from_numpy(rng.uniform(lo, hi, size=n)).to(dev).view(n, 1, 1)

    yy = torch.arange(h, device=dev, dtype=torch.float64).view(1, h, 1)
    xx = torch.arange(w, device=dev, dtype=torch.float64).view(1, 1, w)
    img = torch.full((n, h, w), 128.0, device=dev, dtype=torch.float64)
    for _ in range(6):
        period, ang, phase, amp = par(4, 32), par(0, math.pi), par(0, 2 * math.pi), par(8, 24)
        img += amp * torch.sin(2 * math.pi * (xx * torch.cos(ang) + yy * torch.sin(ang)) / period + phase)
    m = min(h, w)
    for _ in range(8):
        level, cy, cx = par(-48, 48), par(0, h), par(0, w)
        ay, ax, ang = par(m / 16, m / 4), par(m / 16, m / 4), par(0, math.pi)
        u = (xx - cx) * torch.cos(ang) + (yy - cy) * torch.sin(ang)
        v = -(xx - cx) * torch.sin(ang) + (yy - cy) * torch.cos(ang)
        img += level * ((u / ax) ** 2 + (v / ay) ** 2 <= 1.0)
    g = torch.Generator(device=dev)
    g.manual_seed(int(rng.integers(0, 2**62)))
    img += 2.0 * torch.randn((n, h, w), generator=g, device=dev, dtype=torch.float64)
    img = torch.round(img.clamp_(0, 255))
    return (img.float() / 255.0).contiguous()


def _training(case, seed, scale):
    """Training images, positions (image, row, col) in row order, projections."""
    P, n = case["patch"], case["n_pairs"]
    side = 768 if scale == 3 else 512
    lr = side // scale
    per = (lr - P + 1) ** 2
    n_img = max(4, -(-n * 4 // (3 * per)))
    hr = _images(seed * 7 + 1, n_img, side, side)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7 + 2)
    flat = torch.randperm(n_img * per, generator=g, device="cuda")[:n].sort().values
    nw = lr - P + 1
    pos = torch.stack([flat // per, flat % per // nw, flat % nw], 1).int().cpu().numpy()
    return hr, pos


def _projections(case, seed):
    d = case["patch"] ** 2 * (2 if case["feature"] else 1)
    rng = np.random.Generator(np.random.PCG64([seed & 0xFFFFFFFF, 11]))
    alpha = rng.standard_normal((case["L"] * case["k"], d)).astype(np.float32)
    beta = (rng.uniform(0, 0.999, size=case["L"] * case["k"]) * case["bin"]).astype(np.float32)
    return alpha, beta


def _params(case):
    return Z.UpscaleParams(K=case["K"], reg_rel=REG, bp_iters=case["bp"], sigma_spatial=SIGMA_SP,
                           sigma_range=SIGMA_R, bp_radius=RADIUS, precision=case["precision"],
                           rerank_mult=case["mult"])


def _batch_shapes(case):
    """Sides and scales of a batch's images, half of them 3x (a function of the case alone)."""
    rng = np.random.Generator(np.random.PCG64([case["n_images"], case["min_side"], case["max_side"]]))
    lo, hi = case["min_side"], case["max_side"]
    return [(2 + i % 2, int(rng.integers(lo, hi + 1)), int(rng.integers(lo, hi * 4 // 3 + 1)))
            for i in range(case["n_images"])]


def _fixed_neighbours(case, seed):
    """Inputs of the calls that take neighbours: features, the K nearest of
    every query and its weights, found with plain torch."""
    hr, pos = _training(case, seed, case["scale"])
    lr = _images(seed * 7 + 3, 1, case["h"], case["w"])[0]
    f = _lr_patches(lr.double(), case["patch"])
    mu = f.mean(1)
    q = f - mu[:, None]
    dfeat = _dictionary(hr, pos, case["scale"], case["patch"], 0)[0]
    nbr, dist = _nearest(q, dfeat, case["K"])
    wgt = _lle(q, dfeat, nbr)
    return hr, pos, lr, nbr, wgt, mu


def prepare(case, seed):
    kind = case["kind"]
    seed = int(seed)
    ctx = Z.Context(0)
    if kind == "backproj":
        s = case["scale"]
        lr, hr = _backproj_inputs(case, seed)
        return {"case": case, "ctx": ctx, "lr": lr, "hr0": hr, "hr": torch.empty_like(hr), "p": Z.UpscaleParams(
            bp_iters=case["bp"], sigma_spatial=SIGMA_SP, sigma_range=SIGMA_R, bp_radius=RADIUS), "s": s}
    if kind in ("energy", "train"):
        hr, pos, lr, nbr, wgt, mu = _fixed_neighbours(case, seed)
        d = Z.Dictionary(ctx, list(hr), pos, case["scale"], case["patch"], BLUR)
        a, b = _projections(dict(case, L=4, k=8, bin=4.0, feature=0), seed)
        ix = Z.Index(d, 4, 8, 4.0, a, b)
        st = {"case": case, "ix": ix, "lr": lr, "nbr": nbr.int().contiguous(), "wgt": wgt.float().contiguous(),
              "mu": mu.float().contiguous()}
        if kind == "train":
            st["R"] = Z.dictionary_hr(d).requires_grad_(True)
        return st
    p = _params(case)
    if kind == "batch":
        ixs = []
        for s in (2, 3):
            hr, pos = _training(case, seed * 3 + s, s)
            d = Z.Dictionary(ctx, list(hr), pos, s, case["patch"], BLUR)
            ixs.append(Z.Index(d, case["L"], case["k"], case["bin"], *_projections(case, seed * 3 + s)))
        lrs = [(s, _images(seed * 1000 + i, 1, h, w)[0]) for i, (s, h, w) in enumerate(_batch_shapes(case))]
        outs = [torch.empty((s * x.shape[0], s * x.shape[1]), device="cuda") for s, x in lrs]
        return {"case": case, "ixs": ixs, "lrs": lrs, "outs": outs, "p": p}
    hr, pos = _training(case, seed, case["scale"])
    a, b = _projections(case, seed)
    lr = _images(seed * 7 + 3, 1, case["h"], case["w"])[0]
    if kind == "build":
        return {"case": case, "ctx": ctx, "hr": list(hr), "pos": pos, "a": a, "b": b, "lr": lr, "p": p}
    d = Z.Dictionary(ctx, list(hr), pos, case["scale"], case["patch"], BLUR, feature=case["feature"])
    ix = Z.Index(d, case["L"], case["k"], case["bin"], a, b, max_candidates=case["cap"])
    return {"case": case, "ix": ix, "lr": lr, "p": p}


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "zoom":
        return Z.upscale(state["ix"], state["lr"], state["p"])
    if kind == "query":
        r = Z.query(state["ix"], state["lr"], state["p"])
        return {k: r[k] for k in ("nbr", "dist", "wgt", "mu", "bucket_sum")}
    if kind == "batch":
        outs, _ = Z.upscale_batch(state["ixs"], state["lrs"], state["p"], outs=state["outs"])
        return outs
    if kind == "backproj":
        state["hr"].copy_(state["hr0"])
        return Z.backproject(state["ctx"], state["lr"], state["hr"], state["s"], state["p"], BLUR)
    if kind == "energy":
        return Z.map_energy_grads(state["ix"], state["lr"], state["nbr"], state["wgt"])
    if kind == "train":
        h, w = state["lr"].shape
        ix, R = state["ix"], state["R"]
        x = Z.ReconstructFunction.apply(R, ix, state["nbr"], state["wgt"], state["mu"], h, w)
        y = Z.DegradeFunction.apply(x, ix.dictionary.ctx, c["scale"], BLUR)
        loss = ((y - state["lr"]) ** 2).sum()
        (g,) = torch.autograd.grad(loss, R)
        return {"loss": loss.detach(), "hr": x.detach(), "grad": g}
    d = Z.Dictionary(state["ctx"], state["hr"], state["pos"], c["scale"], c["patch"], BLUR, feature=c["feature"])
    ix = Z.Index(d, c["L"], c["k"], c["bin"], state["a"], state["b"])
    return Z.upscale(ix, state["lr"], state["p"])


# ---------------------------------------------------------------------------
# the least work of a pass
# ---------------------------------------------------------------------------

def _image_work(h, w, s, P, K, L, k, d, bp, n_pairs, cap):
    """One image's zoom: queries' hashing, a distance to every kept neighbour,
    the weights, the blend, the overlap average and the back-projection; the
    images, every dictionary feature and the HR rows of the kept neighbours
    (no more than the dictionary has) read once."""
    nq, ph2 = (h - P + 1) * (w - P + 1), (s * P) ** 2
    flops = nq * (2 * L * k * d + 3 * d * max(K, cap) + K * K * d + K ** 3 / 3 + 2 * K * ph2 + ph2)
    flops += bp * (s * s * h * w * (4 * (2 * RADIUS + 1) + 20) + 10 * h * w)
    rows = min(n_pairs, nq * K)
    return 4 * (h * w + s * s * h * w * (1 + 2 * bp) + rows * ph2), flops


def work(case):
    kind = case["kind"]
    if kind == "backproj":
        px, lp = case["scale"] ** 2 * case["h"] * case["w"], case["h"] * case["w"]
        # the estimate read and written by every iteration, each of which
        # needs the whole image of the one before
        return {"bytes": 4 * case["bp"] * (2 * px + lp), "flops": case["bp"] * px * (4 * (2 * RADIUS + 1) + 20)}
    P, n, K = case["patch"], case["n_pairs"], case["K"]
    if kind in ("energy", "train"):
        s, h, w = case["scale"], case["h"], case["w"]
        nq, ph2 = (h - P + 1) * (w - P + 1), (s * P) ** 2
        rows = min(n, nq * K)
        return {"bytes": 4 * (rows * ph2 + n * ph2 + 3 * s * s * h * w + 2 * nq * K),
                "flops": nq * ph2 * (4 * K + (10 if kind == "energy" else 2))}
    d = P * P * (2 if case["feature"] else 1)
    hashed = (case["L"], case["k"], d)
    if kind == "batch":
        tot_b = sum(4 * n * d for _ in (2, 3))
        tot_f = 0
        for s, h, w in _batch_shapes(case):
            b, f = _image_work(h, w, s, P, K, *hashed, case["bp"], 0, 0)
            tot_b, tot_f = tot_b + b, tot_f + f
        return {"bytes": tot_b, "flops": tot_f}
    s, h, w = case["scale"], case["h"], case["w"]
    b, f = _image_work(h, w, s, P, K, *hashed, case["bp"] if kind != "query" else 0, n if kind != "query" else 0,
                       case["cap"])
    b += 4 * n * d
    if kind == "build":
        # training pixels read, features, HR rows, keys and bins written
        b += 4 * n * (d + (s * P) ** 2) * 2 + 12 * n * case["L"]
        f += 2 * n * case["L"] * case["k"] * d
    if kind == "query":
        nq = (h - P + 1) * (w - P + 1)
        b += nq * (12 * K + 8 + 8 * case["L"])
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------

def _clamped(x, r):
    """x [.., h, w] with its edge repeated r pixels on every side."""
    h, w = x.shape[-2:]
    i = torch.arange(-r, h + r, device=x.device).clamp(0, h - 1)
    j = torch.arange(-r, w + r, device=x.device).clamp(0, w - 1)
    return x[..., i, :][..., j]


def _degrade(x, s):
    g = math.exp(-1 / (2 * BLUR ** 2))
    t = [g / (1 + 2 * g), 1 / (1 + 2 * g), g / (1 + 2 * g)]
    h, w = x.shape[-2:]
    p = _clamped(x, 1)
    p = sum(t[u] * p[..., u:u + h, :] for u in range(3))
    p = sum(t[u] * p[..., :, u:u + w] for u in range(3))
    p = p[..., :h // s * s, :w // s * s]
    return p.reshape(*p.shape[:-2], h // s, s, w // s, s).mean((-3, -1))


def _lr_patches(img, P):
    """[origins][P*P] patches of img [h][w]."""
    return img.unfold(0, P, 1).unfold(1, P, 1).reshape(-1, P * P)


def _gradients(x, feature):
    r = 1 if feature == 1 else 2
    h, w = x.shape[-2:]
    p = _clamped(x, r)
    c = p[..., r:r + h, r:r + w]
    left, right = p[..., r:r + h, :w], p[..., r:r + h, 2 * r:]
    up, down = p[..., :h, r:r + w], p[..., 2 * r:, r:r + w]
    if feature == 1:
        return right - left, down - up
    return 2 * c - left - right, 2 * c - up - down


def _query_features(lr, P, feature):
    f = _lr_patches(lr, P)
    mu = f.mean(1)
    if feature == 0:
        return f - mu[:, None], mu
    gx, gy = _gradients(lr, feature)
    return torch.cat([_lr_patches(gx, P), _lr_patches(gy, P)], 1), mu


def _gather(imgs, pos, P, step):
    i, r, c = (torch.from_numpy(pos[:, j].astype(np.int64)).to(imgs.device) for j in range(3))
    o = torch.arange(P, device=imgs.device)
    return imgs[i[:, None, None], (r * step)[:, None, None] + o[:, None], (c * step)[:, None, None] + o].reshape(
        len(pos), P * P)


def _dictionary(hr, pos, s, P, feature, want_hr=False):
    """Features (and HR residuals) of the pairs; LR training images are kept in 32 bits."""
    lr = torch.stack([_degrade(x.double(), s).float() for x in hr]).double()
    pix = _gather(lr, pos, P, 1)
    mu = pix.mean(1, keepdim=True)
    if feature == 0:
        f = pix - mu
    else:
        gx, gy = _gradients(lr, feature)
        f = torch.cat([_gather(gx, pos, P, 1), _gather(gy, pos, P, 1)], 1)
    return f, (_gather(hr, pos, s * P, s).double() - mu) if want_hr else None


def _keys(f, alpha, beta, case):
    """One 64-bit word per table for the tuple of its k hash values."""
    L, k = case["L"], case["k"]
    g = np.random.Generator(np.random.PCG64(5))
    m = torch.from_numpy(g.integers(-2**62, 2**62, size=k) * 2 + 1).to(f.device)
    a = torch.from_numpy(alpha).to(f.device).double()
    b = torch.from_numpy(beta).to(f.device).double()
    out = []
    for part in f.split(1 << 18):
        hsh = torch.floor((part @ a.T + b) / float(np.float32(case["bin"]))).long().view(-1, L, k)
        out.append((hsh * m).sum(2))
    return torch.cat(out)


def _nearest(q, dfeat, K, qkeys=None, dkeys=None):
    """The K nearest entries of every query in 64 bits, among those that share
    a key with it in some table where keys are given.  A 32-bit distance
    preselects 64 of them."""
    df32 = dfeat.float()
    n2 = (dfeat ** 2).sum(1).float()
    m = min(len(dfeat), 64)
    rows = max(1, (1 << 30) // len(dfeat))
    nbrs, dists = [], []
    for i in range(0, len(q), rows):
        p = q[i:i + rows]
        pre = torch.addmm(n2[None], p.float(), df32.T, alpha=-2.0).topk(m, largest=False).indices
        d = ((p[:, None] - dfeat[pre]) ** 2).sum(2)
        if qkeys is not None:
            member = torch.zeros_like(pre, dtype=torch.bool)
            for t in range(qkeys.shape[1]):
                member |= dkeys[:, t][pre] == qkeys[i:i + rows, t, None]
            d = torch.where(member, d, d + 1e6)
        v, o = d.topk(K, largest=False)
        v, o2 = v.sort(1)
        nbrs.append(pre.gather(1, o.gather(1, o2)))
        dists.append(torch.where(v >= 1e6, v - 1e6, v))
    return torch.cat(nbrs), torch.cat(dists)


def _capped(q, dfeat, K, cap, qkeys, dkeys):
    """The K nearest among the first cap distinct entries of a query's bins,
    tables in order, entries in order within a bin."""
    L, n = qkeys.shape[1], len(dfeat)
    tabs = []
    for t in range(L):
        o = torch.sort(dkeys[:, t], stable=True)
        tabs.append((o.values.contiguous(), o.indices))
    ar = torch.arange(cap, device=q.device)
    nbrs, dists = [], []
    for i in range(0, len(q), 1 << 16):
        p = q[i:i + (1 << 16)]
        got = torch.full((len(p), cap), n, device=q.device)
        cnt = torch.zeros(len(p), dtype=torch.long, device=q.device)
        for t in range(L):
            if int(cnt.min()) >= cap:
                break
            kt = qkeys[i:i + (1 << 16), t].contiguous()
            lo = torch.searchsorted(tabs[t][0], kt)
            hi = torch.searchsorted(tabs[t][0], kt, right=True)
            at = lo[:, None] + ar
            ids = tabs[t][1][at.clamp(max=n - 1)]
            new = (at < hi[:, None]) & ~(ids[:, :, None] == got[:, None, :]).any(2)
            rank = cnt[:, None] + torch.cumsum(new, 1) - 1
            new &= rank < cap
            r, c = new.nonzero(as_tuple=True)
            got[r, rank[r, c]] = ids[r, c]
            cnt += new.sum(1)
        d = ((p[:, None] - dfeat[got.clamp(max=n - 1)]) ** 2).sum(2)
        d = torch.where(got < n, d, float("inf"))
        v, o = d.topk(K, largest=False)
        v, o2 = v.sort(1)
        nbrs.append(got.gather(1, o.gather(1, o2)).clamp(max=n - 1))
        dists.append(v)
    return torch.cat(nbrs), torch.cat(dists)


def _lle(q, dfeat, nbr):
    K = nbr.shape[1]
    out = []
    for p, nb in zip(q.split(1 << 18), nbr.split(1 << 18)):
        e = p[:, None] - dfeat[nb]
        G = e @ e.transpose(1, 2)
        tr = G.diagonal(dim1=1, dim2=2).sum(1)
        G = G + (REG * tr).clamp_min(1e-300)[:, None, None] * torch.eye(K, device=q.device, dtype=q.dtype)
        z = torch.linalg.solve(G, torch.ones(len(G), K, 1, device=q.device, dtype=q.dtype))[:, :, 0]
        w = z / z.sum(1, keepdim=True)
        hit = (e[:, 0] ** 2).sum(1) == 0
        w[hit] = torch.eye(K, device=q.device, dtype=q.dtype)[0]
        out.append(w)
    return torch.cat(out)


def _overlap(patch_rows, h, w, s, P):
    """Overlap average of the HR patches; patch_rows(i) gives those of patch row i, [nw][PH][PH]."""
    PH, nh, nw = s * P, h - P + 1, w - P + 1
    acc = None
    for i in range(nh):
        pt = patch_rows(i)
        if acc is None:
            acc = pt.new_zeros(s * h, s * w)
        band = pt.new_zeros(PH, s * w)
        for p in range(P):   # the patches whose columns lie p apart do not overlap
            part = pt[p::P].permute(1, 0, 2).reshape(PH, -1)
            band[:, s * p:s * p + part.shape[1]] += part
        acc[s * i:s * i + PH] += band
    cy = torch.zeros(h, device=acc.device, dtype=acc.dtype)
    cx = torch.zeros(w, device=acc.device, dtype=acc.dtype)
    for p in range(P):
        cy[p:p + nh] += 1
        cx[p:p + nw] += 1
    return acc / (cy.repeat_interleave(s)[:, None] * cx.repeat_interleave(s)[None])


def _blend(hres, nbr, wgt, mu, h, w, s, P):
    nw, PH = w - P + 1, s * P

    def rows(i):
        a = slice(i * nw, (i + 1) * nw)
        return (mu[a, None] + (wgt[a, :, None] * hres[nbr[a]]).sum(1)).view(nw, PH, PH)

    return _overlap(rows, h, w, s, P)


def _backproject(x, y, s, iters):
    r = RADIUS
    o = torch.arange(-r, r + 1, device=x.device, dtype=x.dtype)
    g1 = torch.exp(-o ** 2 / (2 * SIGMA_SP ** 2))
    g1 = g1 / g1.sum()
    b1 = torch.full_like(g1, 1.0 / (2 * r + 1))
    h, w = x.shape

    def window(z, k1):
        p = _clamped(z, r)
        p = sum(k1[u] * p[u:u + h] for u in range(2 * r + 1))
        return sum(k1[u] * p[:, u:u + w] for u in range(2 * r + 1))

    for _ in range(iters):
        e = (_degrade(x, s) - y).repeat_interleave(s, 0).repeat_interleave(s, 1)
        x = x - torch.exp(-(x - window(x, b1)) ** 2 / (2 * SIGMA_R * SIGMA_R)) * window(e, g1)
    return x


def _backproj_inputs(case, seed):
    """An LR image and an HR estimate of the same scene: the degraded HR image
    and a blurred, noisy copy of it."""
    s = case["scale"]
    true = _images(seed * 7 + 5, 1, s * case["h"], s * case["w"])[0]
    lr = _degrade(true.double(), s).float().contiguous()
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7 + 6)
    est = lr.repeat_interleave(s, 0).repeat_interleave(s, 1)
    est = 0.5 * (est + true) + 0.01 * torch.randn(est.shape, generator=g, device="cuda")
    return lr, est.contiguous()


def _exact_queries(case, seed, lr, scale):
    hr, pos = _training(case, seed, scale)
    dfeat, hres = _dictionary(hr, pos, scale, case["patch"], case["feature"], want_hr=case["kind"] != "query")
    a, b = _projections(case, seed)
    dkeys = _keys(dfeat, a, b, case)
    out = []
    for x in lr:
        q, mu = _query_features(x.double(), case["patch"], case["feature"])
        qkeys = _keys(q, a, b, case)
        if case["cap"]:
            nbr, dist = _capped(q, dfeat, case["K"], case["cap"], qkeys, dkeys)
        else:
            nbr, dist = _nearest(q, dfeat, case["K"], qkeys, dkeys)
        wgt = _lle(q, dfeat, nbr)
        if case["kind"] == "query":
            return dist, wgt, mu
        h, w = x.shape
        x0 = _blend(hres, nbr, wgt, mu, h, w, scale, case["patch"])
        out.append(_backproject(x0, x.double(), scale, case["bp"]))
    return out


def exact(case, seed):
    kind, seed = case["kind"], int(seed)
    if kind == "backproj":
        lr, hr = _backproj_inputs(case, seed)
        return _backproject(hr.double(), lr.double(), case["scale"], case["bp"])
    s, P = case.get("scale"), case["patch"]
    if kind in ("energy", "train"):
        h, w = case["h"], case["w"]
        hr, pos, lr, nbr, wgt, mu = _fixed_neighbours(case, seed)
        # what the call takes: indices, 32-bit weights and (autograd) means
        wgt = wgt.float().double()
        R = _dictionary(hr, pos, s, P, 0, want_hr=True)[1].requires_grad_(True)
        y = lr.double()
        if kind == "train":
            R = R.detach().float().double().requires_grad_(True)   # the call's own 32-bit rows
            x = _blend(R, nbr, wgt, mu.float().double(), h, w, s, P)
            loss = ((_degrade(x, s) - y) ** 2).sum()
            return {"loss": loss.detach(), "hr": x.detach(), "grad": torch.autograd.grad(loss, R)[0]}
        nh, nw, PH, ov = h - P + 1, w - P + 1, s * P, s * P - s
        pt = (mu[:, None] + torch.einsum("qk,qkp->qp", wgt, R[nbr])).view(nh, nw, PH, PH)
        x = _overlap(lambda i: pt[i], h, w, s, P)
        xd = x.detach().requires_grad_(True)
        (gx,) = torch.autograd.grad(((_degrade(xd, s) - y) ** 2).sum(), xd)
        prior = ((pt[:, :-1, :, s:] - pt[:, 1:, :, :ov]) ** 2).sum() + ((pt[:-1, :, s:, :] - pt[1:, :, :ov, :]) ** 2).sum()
        e = ((_degrade(x, s) - y) ** 2).sum() + 0.1 * prior
        (gd,) = torch.autograd.grad(e, R)
        return {"energy": float(e), "grad_x": gx, "grad_dict": gd, "hr": x.detach()}
    if kind == "batch":
        shapes = _batch_shapes(case)
        if sum(h * w for _, h, w in shapes) * case["n_pairs"] > 1.5e12:
            return None
        lrs = [_images(seed * 1000 + i, 1, h, w)[0] for i, (_, h, w) in enumerate(shapes)]
        by = {}
        for sc in (2, 3):
            at = [i for i, x in enumerate(shapes) if x[0] == sc]
            if at:
                by.update(zip(at, _exact_queries(case, seed * 3 + sc, [lrs[i] for i in at], sc)))
        return [by[i] for i in range(len(lrs))]
    if not case["cap"] and case["h"] * case["w"] * case["n_pairs"] > 6e11:
        return None   # the distances of every query to every entry would take minutes
    lr = _images(seed * 7 + 3, 1, case["h"], case["w"])[0]
    got = _exact_queries(case, seed, [lr], s)
    if kind == "query":
        dist, wgt, mu = got
        return {"nbr": None, "dist": dist, "wgt": wgt, "mu": mu, "bucket_sum": None}
    return got[0]
