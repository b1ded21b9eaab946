"""Images with a NaN or infinite pixel in their crop have no statistics: they are
flagged degenerate, with zero spectra and filtered images, and the images beside
them keep their bits; the dictionary search gives them no template."""
import math

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


def _images(n, P=6):
    clean = torch.rand((P, n, n), generator=torch.Generator().manual_seed(n)).cuda() * 50 + 10
    bad = clean.clone()
    bad[0, 0, 0] = math.nan        # the pixel that the statistics are taken about
    bad[2, n - 1, n // 3] = math.nan
    bad[3, n // 2, n - 1] = math.inf
    bad[5] = -math.inf
    return clean, bad, torch.tensor([1, 0, 1, 1, 0, 1], device="cuda")


@pytest.mark.parametrize("n", [16, 32, 64, 96, 128, 160, 200, 256])
@pytest.mark.parametrize("spatial", [False, True])
def test_preprocessing(px, n, spatial):
    ctx = px.Context(native_sizes=1)
    g = px.geometry(n, n)
    clean, bad, flag = _images(n)
    S, y, d = px.xcf_prep(ctx, bad, g, want_spatial=spatial)
    assert torch.equal(d, flag.int())
    assert (torch.view_as_real(S)[flag == 1] == 0).all()
    good = flag == 0
    # native 96 and 160 transform two images at once: the partner's place holds zeros in both calls
    ref = clean.clone()
    ref[flag == 1] = 4.0
    S0, y0, _ = px.xcf_prep(ctx, ref, g, want_spatial=spatial)
    assert torch.equal(torch.view_as_real(S)[good], torch.view_as_real(S0)[good])
    if spatial:
        assert (y[flag == 1] == 0).all() and torch.equal(y[good], y0[good])
    ctx.close()


@pytest.mark.parametrize("n", [16, 32, 64, 128, 256])
def test_dictionary_search(px, n):
    ctx = px.Context()
    g = px.geometry(n, n)
    clean, bad, flag = _images(n)
    q = torch.zeros((6, 4), dtype=torch.float64, device="cuda")
    q[:, 0] = 1
    lib = px.xcf_build_library_ex(ctx, q, g, images=clean, flags=px.XCF_LIB_NDP)
    best = px.xcf_index_ndp(ctx, lib, bad, k=2)[0]
    assert best.tolist() == [-1, 1, -1, -1, 4, -1]
    lib.close()
    ctx.close()
