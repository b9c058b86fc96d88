"""The recorded batch of a context (zoom_upscale_batch) and its tuned search
choices: a record is replayed only for the call it was made from, and neither
outlives what it refers to."""
import numpy as np
import pytest

import synth_inputs as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


class LiveAllocator:
    """PyTorch's caching allocator with the live allocations recorded."""

    def __init__(self):
        self.live = {}

    def alloc(self, nbytes, stream, user):
        p = torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))
        self.live[p] = int(nbytes)
        return p

    def free(self, ptr, nbytes, stream, user):
        assert self.live.pop(ptr) == nbytes
        torch.cuda.caching_allocator_delete(ptr)


def _context():
    import paper_1004_3980_gb300 as Z
    A = LiveAllocator()
    return Z.Context(0, allocator=A), A


def _index(ctx, n_pairs=5000, n_train=3, hr=96):
    import paper_1004_3980_gb300 as Z
    train = [S.make_image(3000 + i, hr, hr) for i in range(n_train)]
    pos = S.sample_positions(7, n_train, hr // 2, hr // 2, 5, n_pairs)
    alpha, beta = S.lsh_draws(11, 8, 10, 25, 4.0)
    d = Z.Dictionary(ctx, [torch.from_numpy(x).cuda() for x in train], pos, 2, 5)
    return Z.Index(d, 8, 10, 4.0, alpha, beta)


def _images(*shapes):
    return [(2, torch.from_numpy(S.make_image(3100 + i, h, w)).cuda()) for i, (h, w) in enumerate(shapes)]


def test_destroying_an_index_frees_the_batch_recorded_from_it():
    # (seen in the allocator: the graph of a destroyed index is never run)
    import paper_1004_3980_gb300 as Z
    ctx, A = _context()
    ix = _index(ctx)
    other = _index(ctx)
    torch.cuda.synchronize()
    held = dict(A.live)
    p = Z.UpscaleParams(K=8, bp_iters=1)
    lrs = _images((20, 24), (31, 17))
    outs, _ = Z.upscale_batch([ix], lrs, p)
    torch.cuda.synchronize()
    record = {a: n for a, n in A.live.items() if a not in held}
    assert record
    other.close()                                  # not the record's: it stays
    assert all(A.live.get(a) == n for a, n in record.items())
    ix.close()
    assert not any(a in A.live for a in record)
    ix = _index(ctx)                               # the same sizes: the handle's address may come back
    got, _ = Z.upscale_batch([ix], lrs, p, outs=outs)
    for (_, x), o in zip(lrs, got):
        assert torch.equal(o, Z.upscale(ix, x, p))
    Z.batch_release(ctx)


@pytest.mark.parametrize("change", [dict(fp64_cond_threshold=1.0), dict(reg_rel=9e-10), dict(sigma_spatial=1.5000005)],
                         ids=lambda c: next(iter(c)))
def test_a_changed_parameter_is_not_a_replay(change):
    # each call's images must be those of single calls with its parameters
    import dataclasses
    import paper_1004_3980_gb300 as Z
    ctx, _ = _context()
    ix = _index(ctx)
    p = Z.UpscaleParams(K=8, bp_iters=2, reg_rel=2e-10 if "reg_rel" in change else 1e-3)
    lrs = _images((40, 44), (31, 17))
    outs, _ = Z.upscale_batch([ix], lrs, p)
    first = [o.clone() for o in outs]
    q = dataclasses.replace(p, **change)
    outs, _ = Z.upscale_batch([ix], lrs, q, outs=outs)
    second = [o.clone() for o in outs]
    n_fp64 = ctx.stats()["n_fp64_solves"]
    for (_, x), a, b in zip(lrs, first, second):
        assert torch.equal(a, Z.upscale(ix, x, p))
        assert torch.equal(b, Z.upscale(ix, x, q))
    assert not all(torch.equal(a, b) for a, b in zip(first, second))
    if "fp64_cond_threshold" in change:
        assert n_fp64 > 0
    Z.batch_release(ctx)


@pytest.mark.parametrize("n_pairs, first, second", [(256, (20, 24), (21, 24)),            # dense both times
                                                    (65536, (120, 160), (150, 160))],      # then over the search order
                         ids=["dense", "search order"])
def test_list_sizes_follow_the_calls_own_rerank_mult(n_pairs, first, second):
    # A precision-form batch with rerank_mult 2 (16 chunks a query) tunes the
    # searches of its query count; one with rerank_mult 4 (32 chunks) and as
    # many queries, to a power of two, must not search 16.  The list size is
    # seen in the search workspace, the batch's largest allocations (a
    # dictionary of 256 entries is one step, so the tuned splits are 1).
    import paper_1004_3980_gb300 as Z

    def sizes(calls):
        ctx, A = _context()
        ix = _index(ctx, n_pairs, *((3, 96) if n_pairs < 5000 else (10, 256)))
        torch.cuda.synchronize()
        held = dict(A.live)
        for shape, mult in calls:
            lrs = _images(shape)
            p = Z.UpscaleParams(K=8, bp_iters=1, precision=1, rerank_mult=mult)
            outs, _ = Z.upscale_batch([ix], lrs, p)
        torch.cuda.synchronize()
        single = Z.upscale(ix, lrs[0][1], p)
        assert torch.equal(outs[0], single)
        got = sorted(n for a, n in A.live.items() if a not in held)
        Z.batch_release(ctx)
        return got

    assert sizes([(first, 2), (second, 4)]) == sizes([(second, 4)])
