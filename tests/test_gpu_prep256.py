"""256 x 256 pre-processing at the edges of its loads and stores: crops whose
rows are or are not 16-byte aligned, images and outputs off a 16-byte
boundary, more images than resident clusters, degenerate images among them.
Bound: 2e-6 absolute on unit-norm data (FP32 transforms of N^2 points)."""
import ctypes as C

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def px():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_11313_gb300 as px
    px.load()
    return px


def _call(px, ctx, img, P, g, spec, spat, deg):
    """xcf_prep on raw device addresses."""
    lib = px.load()
    rc = lib.xcf_prep(ctx.handle, C.c_void_p(img), P, C.byref(g), C.c_void_p(spec), C.c_void_p(spat), C.c_void_p(deg),
                      C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()


@pytest.mark.parametrize("W,H", [(256, 256), (259, 257), (260, 278), (511, 256), (264, 400)])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("window", [0, 1])
def test_alignments_match_oracle(px, orc, W, H, shift, window):
    P, n = 3, 256
    rng = np.random.default_rng(W + H)
    imgs = (rng.standard_normal((P, H, W)) * 5 + 60).astype(np.float32)
    imgs[1] = 4.0
    ctx = px.Context(window=window)
    g = px.geometry(W, H)
    _, ox, oy, _ = px.xcf_crop(g)
    store = torch.zeros(P * H * W + 4, device="cuda")
    store[shift:shift + P * H * W] = torch.from_numpy(imgs).cuda().reshape(-1)
    spec = torch.zeros((P, n, n // 2 + 1, 2), device="cuda")
    spat = torch.full((P * n * n + 8,), 7.0, device="cuda")
    deg = torch.zeros(P, dtype=torch.int32, device="cuda")
    _call(px, ctx, store.data_ptr() + 4 * shift, P, g, spec.data_ptr(), spat.data_ptr() + 4 * shift, deg.data_ptr())
    opts = orc.default_opts(n)
    opts.window = window
    S, y, odeg = orc.prep_many(imgs[:, oy:oy + n, ox:ox + n], opts, want_spatial=True)
    assert deg.cpu().numpy().tolist() == odeg.tolist() == [0, 1, 0]
    got = spec.cpu().numpy()
    np.testing.assert_allclose(got[..., 0] + 1j * got[..., 1], S[:, :, : n // 2 + 1], rtol=0, atol=2e-6)
    out = spat.cpu().numpy()
    np.testing.assert_allclose(out[shift:shift + P * n * n].reshape(P, n, n), y, rtol=0, atol=2e-6)
    assert (out[:shift] == 7).all() and (out[shift + P * n * n:] == 7).all()
    ctx.close()


@pytest.mark.parametrize("P", [1, 2, 75, 76, 77, 160])
def test_many_images_equal_single_images(px, P):
    """Each image's outputs do not depend on its place in the batch."""
    n = 256
    g = px.geometry(n, n)
    ctx = px.Context()
    base = torch.rand((5, n, n), generator=torch.Generator().manual_seed(1)).cuda() * 40
    base[2] = 1.5
    which = torch.arange(P, device="cuda") % 5
    S, y, d = px.xcf_prep(ctx, base[which].contiguous(), g, want_spatial=True)
    S1, y1, d1 = zip(*(px.xcf_prep(ctx, base[i:i + 1].contiguous(), g, want_spatial=True) for i in range(5)))
    S1, y1, d1 = torch.cat(S1), torch.cat(y1), torch.cat(d1)
    assert d1.tolist() == [0, 0, 1, 0, 0]
    assert torch.equal(torch.view_as_real(S), torch.view_as_real(S1[which])) and torch.equal(y, y1[which])
    assert torch.equal(d, d1[which])
    S2, _, _ = px.xcf_prep(ctx, base[which].contiguous(), g)      # without the filtered images
    assert torch.equal(torch.view_as_real(S2), torch.view_as_real(S))
    ctx.close()
