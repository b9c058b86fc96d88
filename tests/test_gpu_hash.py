"""Hash keys of many rows (two rows a thread) and of few (tables split over
blocks): a query's keys depend on its patch alone, so the keys of a large
image equal those of the strips it is cut into, bit for bit -- odd and even
table counts, bin widths that are no power of two, and a key buffer that
starts 8 bytes past a 16-byte boundary."""
import numpy as np
import pytest

import synth_inputs as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("L,k,w,patch,feature", [(16, 16, 4.0, 5, 0), (7, 12, 0.37, 5, 0), (1, 3, 1e-3, 3, 0),
                                                 (6, 9, 2.9, 5, 1), (8, 12, 1e30, 3, 1)])
def test_keys_of_an_image_are_its_strips(L, k, w, patch, feature):
    import paper_1004_3980_gb300 as Z
    d = patch * patch * (2 if feature else 1)
    a, b = S.lsh_draws(6, L, k, d, w)
    train = [torch.from_numpy(S.make_image(300, 128, 128)).cuda()]
    pos = S.sample_positions(5, 1, 64, 64, patch, 500)
    ctx = Z.Context(0)
    ix = Z.Index(Z.Dictionary(ctx, train, pos, 2, patch, feature=feature), L, k, w, a, b)
    h, wd = 283, 301   # more than 77,824 queries, not a multiple of 256
    img = torch.from_numpy(np.ascontiguousarray(S.make_image(1, h, wd))).cuda()
    p = Z.UpscaleParams(K=3, search=1)
    whole = Z.query(ix, img, p)["keys"].cpu().numpy().reshape(h - patch + 1, wd - patch + 1, L)
    got = []
    for i in range(0, h - patch + 1, 100):
        n = min(100, h - patch + 1 - i)
        # gradients clamp at the image's edge: rows beside the strip are kept
        lo, hi = max(0, i - 2), min(h, i + n + patch + 1)
        r = Z.query(ix, img[lo:hi].contiguous(), p)["keys"].cpu().numpy()
        got.append(r.reshape(hi - lo - patch + 1, wd - patch + 1, L)[i - lo:i - lo + n])
    assert np.array_equal(whole, np.concatenate(got))


@pytest.mark.parametrize("h,wd", [(61, 60), (283, 301)])   # one row a thread, two
def test_keys_into_a_buffer_8_bytes_past_a_16_byte_boundary(h, wd):
    import ctypes as C
    import paper_1004_3980_gb300 as Z
    from paper_1004_3980_gb300 import capi
    L, k = 6, 9
    a, b = S.lsh_draws(6, L, k, 25, 2.9)
    train = [torch.from_numpy(S.make_image(300, 128, 128)).cuda()]
    ix = Z.Index(Z.Dictionary(Z.Context(0), train, S.sample_positions(5, 1, 64, 64, 5, 500), 2, 5), L, k, 2.9, a, b)
    img = torch.from_numpy(np.ascontiguousarray(S.make_image(1, h, wd))).cuda()
    p = Z.UpscaleParams(K=3, search=1)
    want = Z.query(ix, img, p)
    nq = (h - 4) * (wd - 4)
    keys = torch.full((nq * L + 2,), -1, dtype=torch.int64, device="cuda")
    assert keys.data_ptr() % 16 == 0
    nbr = torch.empty((nq, 3), dtype=torch.int32, device="cuda")
    cp = p.c()
    ptr = lambda t, off=0: C.c_void_p(t.data_ptr() + off)
    capi.call("zoom_query", ix.handle, ptr(img), h, wd, C.byref(cp), ptr(keys, 8), ptr(nbr), None, None, None, None,
              C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert torch.equal(keys[1:-1].reshape(nq, L), want["keys"].reshape(nq, L).view(torch.int64))
    assert keys[0] == -1 and keys[-1] == -1
    assert torch.equal(nbr, want["nbr"])
