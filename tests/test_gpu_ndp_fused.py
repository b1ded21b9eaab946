"""Background correction and normalisation in one kernel (2^k sides up to 128 at the
default blur): crops of uneven detectors, images off a 16-byte boundary, constant
images, against Eq. 1 in float64 on the same crops.  Bound: 2e-6 on the dot
products, as the FP32 rescore's."""
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


def _operands(crops, n):
    """Crop minus its Gaussian blur (sigma n / 8, radius 3 n / 8, edges repeated), unit contrast."""
    R, x = 3 * n // 8, crops.double()
    w = torch.exp(-torch.arange(-R, R + 1, dtype=torch.float64, device=x.device) ** 2 / (2 * (n / 8) ** 2))
    w /= w.sum()
    pad = lambda a: torch.nn.functional.pad(a[:, None], (R, R, R, R), mode="replicate")
    blur = torch.nn.functional.conv2d(torch.nn.functional.conv2d(pad(x), w[None, None, None, :]), w[None, None, :, None])
    y = (x - blur[:, 0]).flatten(1)
    y = y - y.mean(1, keepdim=True)
    return y / y.norm(dim=1, keepdim=True)


@pytest.mark.parametrize("n", [16, 32, 64, 128])
@pytest.mark.parametrize("dw,dh", [(0, 0), (3, 1), (4, 5)])
def test_matches_float64(px, n, dw, dh):
    P, T, W, H = 5, 4, n + dw, n + dh
    ctx = px.Context()
    g = px.geometry(W, H)
    _, ox, oy, _ = px.xcf_crop(g)
    gen = torch.Generator().manual_seed(n + dw)
    timg = (torch.randn((T, H, W), generator=gen) * 3 + 40).cuda()
    store = torch.empty(P * H * W + 1, device="cuda")
    pats = store[1:].view(P, H, W)   # one float off
    pats.copy_(timg[[0, 1, 2, 3, 0]] + torch.randn((P, H, W), generator=gen).cuda())
    pats[3] = 7.0
    q = torch.zeros((T, 4), dtype=torch.float64, device="cuda")
    q[:, 0] = 1
    lib = px.xcf.xcf_build_library_ex(ctx, q, g, images=timg, flags=px.XCF_LIB_NDP | px.XCF_LIB_NO_SPECTRA)
    best, ndp = px.xcf_index_ndp(ctx, lib, pats, k=T)[:2]
    crop = lambda a: a[:, oy:oy + n, ox:ox + n]
    ok = torch.tensor([0, 1, 2, 4])
    S = _operands(crop(pats)[ok.cuda()], n) @ _operands(crop(timg), n).T
    assert best.tolist() == [0, 1, 2, -1, 0] and ndp[3] == 0
    torch.testing.assert_close(ndp[ok.cuda()].double(), S.amax(1), rtol=0, atol=2e-6)
    lib.close()
    ctx.close()
