"""Row top-k of the screen at its edges: counts around the register tiers, k up
to 64 and above the library size, rows of equal scores (longer than the short
list), exact against a stable sort of the kernel's own scores."""
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


def _library(px, ctx, imgs):
    q = torch.zeros((imgs.shape[0], 4), dtype=torch.float64, device="cuda")
    q[:, 0] = 1
    return px.xcf_build_library_ex(ctx, q, px.geometry(16, 16), images=imgs, flags=px.XCF_LIB_SCREEN)


@pytest.mark.parametrize("T", [1, 2, 63, 64, 65, 511, 513, 2047, 2049, 5121, 20481, 40961, 51200])
def test_topk_is_the_stable_sort(px, T):
    """All scores through k = 64 lists of library slices would hide the order, so
    the reference sorts scores of a one-template-at-a-time screen: every
    template repeated with a few distinct images, ties in index order."""
    ctx = px.Context()
    g = torch.Generator().manual_seed(T)
    base = torch.randn((7, 16, 16), generator=g).cuda()
    which = torch.randint(0, 7, (T,), generator=g)
    lib = _library(px, ctx, base[which.cuda()].contiguous())
    pats = torch.cat([base[:3], torch.randn((2, 16, 16), generator=g).cuda()])
    small = _library(px, ctx, base)
    cand7, score7 = px.xcf_screen_topk(ctx, small, pats, 7)
    by_image = torch.empty((5, 7))
    by_image.scatter_(1, cand7.cpu().long(), score7.cpu())
    full = by_image[:, which].numpy()                              # [5, T]: many equal scores
    for k in (1, 4, 32, 64):
        cand, score = (t.cpu().numpy() for t in px.xcf_screen_topk(ctx, lib, pats, k))
        order = np.argsort(-full, axis=1, kind="stable")[:, :min(k, T)]
        assert (cand[:, :min(k, T)] == order).all()
        assert (score[:, :min(k, T)] == np.take_along_axis(full, order, 1)).all()
        assert (cand[:, T:] == -1).all() and np.isneginf(score[:, T:]).all()
    small.close()
    lib.close()
    ctx.close()


@pytest.mark.parametrize("T", [40000])
def test_topk_of_distinct_scores(px, T):
    ctx = px.Context()
    imgs = torch.randn((T, 16, 16), generator=torch.Generator().manual_seed(3)).cuda()
    lib = _library(px, ctx, imgs)
    pats = imgs[::4000].contiguous() + 0.5 * torch.randn((10, 16, 16), generator=torch.Generator().manual_seed(4)).cuda()
    full, _ = px.xcf_screen_topk(ctx, lib, pats, 64)
    cand, score = px.xcf_screen_topk(ctx, lib, pats, 32)
    assert torch.equal(cand, full[:, :32]) and (score[:, :-1] >= score[:, 1:]).all()
    assert (cand[:, 0].cpu() == torch.arange(0, T, 4000, dtype=torch.int32)).all()
    lib.close()
    ctx.close()
