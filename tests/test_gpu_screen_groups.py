"""The two-CTA screen over more pattern tiles than one group of its tile order (four
pairs): a last group of one, two and four pairs, and a ring of 256 turns (K = 16,384),
against float64 products of the same BF16 operands.  Bound: partial sums of unit
vectors stay within 1, and each of the K / 16 accumulations rounds once in FP32, at
most 2^-23."""
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


@pytest.mark.parametrize("n,P,T", [(64, 1200, 7937), (64, 1500, 6600), (64, 2000, 2561), (128, 512, 9729)])
def test_pairs_of_several_groups(px, n, P, T):
    g = px.geometry(n, n)
    ctx = px.Context()
    gen = torch.Generator().manual_seed(P + T)
    timg = torch.randn((T, n, n), generator=gen).cuda()
    pimg = torch.randn((P, n, n), generator=gen).cuda()
    q = torch.zeros((T, 4), dtype=torch.float64, device="cuda")
    q[:, 0] = 1
    lib = px.xcf.xcf_build_library_ex(ctx, q, g, images=timg, flags=px.xcf.XCF_LIB_SCREEN)
    cand, score = px.xcf.xcf_screen_topk(ctx, lib, pimg, 64)
    yt, yp = (px.xcf_prep(ctx, im, g, want_spatial=True)[1].flatten(1).bfloat16().double() for im in (timg, pimg))
    ref = yp @ yt.T
    atol = n * n / 16 * 2.0 ** -23 + 1e-6
    torch.testing.assert_close(score.double(), ref.gather(1, cand.long()), rtol=0, atol=atol)
    torch.testing.assert_close(score.double(), ref.topk(64, dim=1).values, rtol=0, atol=atol)
    lib.close()
    ctx.close()
