"""Peak of one 256 x 256 surface: circular shifts at every wrap and at the
borders of the lines a CTA holds (32) and of the packed halves (128), ties, more
surfaces than resident clusters."""
import pytest
import torch

pytestmark = pytest.mark.gpu
N = 256


@pytest.fixture(scope="module")
def px():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_11313_gb300 as px
    px.load()
    return px


def _image(seed, P=1):
    x = torch.randn((P, N + 4, N + 4), generator=torch.Generator().manual_seed(seed), dtype=torch.float64)
    return torch.nn.functional.avg_pool2d(x[:, None], 5, 1)[:, 0].float().cuda().contiguous()


def _library(px, ctx, img):
    q = torch.tensor([[1.0, 0, 0, 0]], dtype=torch.float64, device="cuda")
    return px.xcf_build_library_images(ctx, img, q, px.geometry(N, N))


SHIFTS = [(dy, dx) for dy in (0, 1, 31, 32, 127, 128, 129, 160, 255) for dx in (0, 1, 15, 16, 127, 128, 255)]


def test_every_wrap(px):
    """An unwindowed pattern shifted circularly peaks at exactly that shift, wrapped
    into [-128, 128); the parabola of a symmetric peak adds nothing (1e-3 px: FP32
    differences of neighbouring values near 1)."""
    ctx = px.Context(window=0)
    img = _image(7)
    lib = _library(px, ctx, img)
    pats = torch.cat([torch.roll(img, s, (1, 2)) for s in SHIFTS] * 3).contiguous()   # more than the resident clusters
    best, peak, shift = px.xcf_index(ctx, lib, pats)
    want = torch.tensor([[float(d if d < N // 2 else d - N) for d in (dx, dy)] for dy, dx in SHIFTS] * 3)
    assert (best == 0).all() and ((peak - 1).abs() < 1e-5).all()
    torch.testing.assert_close(shift.cpu(), want, rtol=0, atol=1e-3)
    lib.close()
    ctx.close()


def test_tie_takes_the_lowest_shift(px):
    """A template without signal gives a surface of equal values: index 0."""
    ctx = px.Context()
    lib = _library(px, ctx, torch.full((1, N, N), 2.0, device="cuda"))
    best, peak, shift = px.xcf_index(ctx, lib, _image(9, 3))
    assert best.tolist() == [0] * 3 and peak.tolist() == [0] * 3 and (shift == 0).all()
    lib.close()
    ctx.close()
