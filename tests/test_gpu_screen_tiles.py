"""The zero-shift screen at the edges of its tiles: one and two CTAs per tile (two
with an even number of 128-pattern tiles, more tiles than SMs and K >= 4,096), last
tiles of patterns and templates that are nearly empty, K of less than one to many
turns of the ring, against float64 products of the same BF16 operands.  Bound:
partial sums of unit vectors stay within 1, and each of the K / 16 accumulations
rounds once in FP32, at most 2^-23."""
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


def check(px, n, P, T):
    k = min(T, 64)
    g = px.geometry(n, n)
    ctx = px.Context()
    gen = torch.Generator().manual_seed(P * 1000 + T)
    timg = torch.randn((T, n, n), generator=gen).cuda()
    pimg = torch.randn((P, n, n), generator=gen).cuda()
    q = torch.zeros((T, 4), dtype=torch.float64, device="cuda")
    q[:, 0] = 1
    lib = px.xcf.xcf_build_library_ex(ctx, q, g, images=timg, flags=px.xcf.XCF_LIB_SCREEN)
    cand, score = px.xcf.xcf_screen_topk(ctx, lib, pimg, k)
    yt, yp = (px.xcf_prep(ctx, im, g, want_spatial=True)[1].flatten(1).bfloat16().double() for im in (timg, pimg))
    ref = yp @ yt.T
    atol = n * n / 16 * 2.0 ** -23 + 1e-6
    torch.testing.assert_close(score.double(), ref.gather(1, cand.long()), rtol=0, atol=atol)
    torch.testing.assert_close(score.double(), ref.topk(k, dim=1).values, rtol=0, atol=atol)
    lib.close()
    ctx.close()


@pytest.mark.parametrize("P", [1, 128, 129, 256, 257, 385, 1000])
@pytest.mark.parametrize("T", [1, 33, 256, 257, 2050, 9729])
def test_tiles(px, P, T):
    check(px, 16, P, T)


@pytest.mark.parametrize("n", [32, 64, 128])
def test_ring(px, n):
    check(px, n, 200, 300)
    check(px, n, 100, 300)


@pytest.mark.parametrize("P,T", [(256, 19457), (129, 19712), (200, 20000), (1000, 5100), (385, 10001), (512, 9729)])
def test_pairs(px, P, T):
    check(px, 64, P, T)
