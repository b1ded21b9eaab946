"""All-pairs search at library sizes where its work split ends unevenly (odd
counts, one template, fewer templates than a part), against float64 inverse
transforms of the same FP32 spectra.  Bound: 1e-4 relative + 1e-6 on the peaks
(FP32 transforms of unit-norm spectra), the best template exact."""
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


def _images(n, P, seed):
    x = torch.randn((P, n + 4, n + 4), generator=torch.Generator().manual_seed(seed), dtype=torch.float64)
    x = torch.nn.functional.avg_pool2d(x[:, None], 5, 1)[:, 0]   # correlated pixels, as a pattern's
    return x.float().cuda().contiguous()


def _reference(St, Sp):
    n = Sp.shape[1]
    out = torch.stack([torch.fft.irfft2(St.to(torch.complex128).conj() * s.to(torch.complex128), s=(n, n), norm="forward")
                       .flatten(1).amax(1) for s in Sp])
    return out


def check_search(px, n, T, P, native=0):
    ctx = px.Context(native_sizes=native)
    g = px.geometry(n, n)
    q = torch.zeros((T, 4), dtype=torch.float64, device="cuda")
    q[:, 0] = 1
    lib = px.xcf_build_library_images(ctx, _images(n, T, T), q, g)
    pats = _images(n, P, 1000 + P)
    if P > 2:
        pats[1] = 3.0   # degenerate: skipped
    Sp, _, deg = px.xcf_prep(ctx, pats, g)
    ref = _reference(lib.spectra(), Sp)
    ok = deg == 0
    peaks = px.xcf_correlate_all(ctx, lib, pats)
    torch.testing.assert_close(peaks[ok].double(), ref[ok], rtol=1e-4, atol=1e-6)
    assert (peaks[~ok] == 0).all()
    best, peak, _ = px.xcf_index(ctx, lib, pats)
    assert (best[~ok] == -1).all()
    assert torch.equal(best[ok].long(), ref[ok].argmax(1))
    torch.testing.assert_close(peak[ok].double(), ref[ok].amax(1), rtol=1e-4, atol=1e-6)
    lib.close()
    ctx.close()


@pytest.mark.parametrize("T", [1, 2, 3, 15, 16, 17, 33, 130])
@pytest.mark.parametrize("P", [1, 3, 153])
def test_search_128(px, T, P):
    check_search(px, 128, T, P)


@pytest.mark.parametrize("dy", [0, 1, 63, 64, 65, 127])
@pytest.mark.parametrize("dx", [0, 1, 63, 64, 127])
def test_peak_128_at_every_wrap(px, dy, dx):
    """A circularly shifted, unwindowed pattern peaks at exactly that shift,
    wrapped into [-64, 64); the parabola of a symmetric peak adds nothing
    (1e-3 px: FP32 differences of neighbouring values near 1)."""
    n = 128
    ctx = px.Context(window=0)
    g = px.geometry(n, n)
    img = _images(n, 1, 7)
    q = torch.tensor([[1.0, 0, 0, 0]], dtype=torch.float64, device="cuda")
    lib = px.xcf_build_library_images(ctx, img, q, g)
    best, peak, shift = px.xcf_index(ctx, lib, torch.roll(img, (dy, dx), (1, 2)).contiguous())
    want = [float(d if d < n // 2 else d - n) for d in (dx, dy)]
    assert best.tolist() == [0] and abs(peak.item() - 1) < 1e-5
    torch.testing.assert_close(shift[0].cpu(), torch.tensor(want), rtol=0, atol=1e-3)
    lib.close()
    ctx.close()


def test_peak_128_tie_takes_the_lowest_shift(px):
    """A template without signal gives a surface of equal values: index 0."""
    n = 128
    ctx = px.Context()
    g = px.geometry(n, n)
    q = torch.tensor([[1.0, 0, 0, 0]], dtype=torch.float64, device="cuda")
    lib = px.xcf_build_library_images(ctx, torch.full((1, n, n), 2.0, device="cuda"), q, g)
    best, peak, shift = px.xcf_index(ctx, lib, _images(n, 3, 9))
    assert best.tolist() == [0] * 3 and peak.tolist() == [0] * 3 and (shift == 0).all()
    lib.close()
    ctx.close()


@pytest.mark.parametrize("T", [1, 2, 3, 7, 8, 9, 33, 130])
@pytest.mark.parametrize("P", [1, 3, 40])
@pytest.mark.parametrize("n", [64, 96])
def test_search_64_and_96(px, n, T, P):
    check_search(px, n, T, P, native=1)


@pytest.mark.parametrize("n", [64, 96, 128, 160, 200, 256])
@pytest.mark.parametrize("k", [1, 2, 5, 8])
def test_candidate_lists(px, n, k):
    """Lists with empty entries, repeated templates (ties to the lowest index)
    and descending order against float64."""
    T, P = 20, 5
    ctx = px.Context(native_sizes=1)
    g = px.geometry(n, n)
    q = torch.zeros((T, 4), dtype=torch.float64, device="cuda")
    q[:, 0] = 1
    imgs = _images(n, T, 5)
    imgs[11] = imgs[4]
    lib = px.xcf_build_library_images(ctx, imgs, q, g)
    pats = torch.cat([imgs[11:12], _images(n, P - 1, 6)])
    cand = torch.tensor([[11, 4, -1, 19, 0, 7, -1, 3], [-1] * 8, [0, 1, 2, 3, 4, 5, 6, 7], [19, 18, 17, 16, 15, 14, 13, 12],
                         [4, -1, 11, -1, 4, 9, 9, 9]], dtype=torch.int32, device="cuda")[:, :k].contiguous()
    best, peak, _ = px.xcf_rescore(ctx, lib, pats, cand)
    ref = _reference(lib.spectra(), px.xcf_prep(ctx, pats, g)[0])
    for p in range(P):
        c = sorted({int(t) for t in cand[p] if t >= 0})
        if not c:
            assert best[p] == -1 and peak[p] == 0
            continue
        top = max(c, key=lambda t: (ref[p, t].item(), -t))
        if ref[p, top] - ref[p, 4] < 1e-7 and 4 in c:   # equal templates 4 and 11
            top = 4
        assert int(best[p]) == top
        torch.testing.assert_close(peak[p].double(), ref[p, top], rtol=1e-4, atol=1e-6)
    lib.close()
    ctx.close()


@pytest.mark.parametrize("T", [1, 2, 7, 8, 9, 17])
@pytest.mark.parametrize("P", [1, 3])
@pytest.mark.parametrize("n", [160, 200])
def test_search_160_and_200(px, n, T, P):
    check_search(px, n, T, P, native=1)


@pytest.mark.parametrize("T", [1, 2, 3, 5, 17, 65])
@pytest.mark.parametrize("P", [1, 3, 80])
def test_search_256(px, T, P):
    check_search(px, 256, T, P)


def test_long_candidate_lists_128(px):
    """Lists in several parts, with runs of empty entries longer than a part's step."""
    n, T, P, k = 128, 70, 4, 64
    ctx = px.Context()
    g = px.geometry(n, n)
    q = torch.zeros((T, 4), dtype=torch.float64, device="cuda")
    q[:, 0] = 1
    lib = px.xcf_build_library_images(ctx, _images(n, T, 8), q, g)
    pats = _images(n, P, 9)
    cand = torch.stack([torch.randperm(T, generator=torch.Generator().manual_seed(p))[:k] for p in range(P)]).int()
    cand[1, 5:40] = -1
    cand[2, :63] = -1
    cand[3, 1::2] = -1
    best, peak, _ = px.xcf_rescore(ctx, lib, pats, cand.cuda())
    ref = _reference(lib.spectra(), px.xcf_prep(ctx, pats, g)[0])
    for p in range(P):
        c = cand[p][cand[p] >= 0].cuda().long()
        assert int(best[p]) == int(c[ref[p, c].argmax()])
        torch.testing.assert_close(peak[p].double(), ref[p, c].amax(), rtol=1e-4, atol=1e-6)
    lib.close()
    ctx.close()
