"""The 256 x 256 kernels on thread-block clusters give the same bits on every
run: pre-processing with and without filtered images and with images that have
no signal between the others (they take fewer barriers), search, every peak, and
the single-surface peaks, on more work than clusters are resident together."""
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


@pytest.mark.parametrize("flat", [2, 3, 7])
def test_runs_agree(px, flat):
    gen = torch.Generator().manual_seed(flat)
    g, P, T = px.geometry(N, N), 331, 40
    ctx = px.Context()
    tmpl = torch.randn((T, N, N), generator=gen).cuda()
    pats = torch.randn((P, N, N), generator=gen).cuda()
    pats[::flat] = 3.0
    q = torch.zeros((T, 4), dtype=torch.float64, device="cuda")
    q[:, 0] = 1
    lib = px.xcf_build_library_images(ctx, tmpl, q, g)
    runs = []
    for _ in range(6):
        S, y, d = px.xcf_prep(ctx, pats, g, want_spatial=True)
        S0, _, d0 = px.xcf_prep(ctx, pats, g)
        best, peak, shift = px.xcf_index(ctx, lib, pats)
        runs.append([torch.view_as_real(S), y, d, torch.view_as_real(S0), d0, best, peak, shift])
    assert d.sum() == len(range(0, P, flat)) and (best[d == 0] >= 0).all()
    assert torch.equal(runs[0][0], runs[0][3])
    for r in runs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(r, runs[0]))
    lib.close()
    ctx.close()
