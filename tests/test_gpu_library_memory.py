"""Where a library keeps the master's 2 x 2 cells: behind its spectra, behind its
master, or nowhere (a few templates of a small master, which then take no
device mapping of their own), with the same template spectra in each."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def px():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_11313_gb300 as px
    px.load()
    return px


def _inputs(M, T):
    m = torch.rand((2, M, M), generator=torch.Generator().manual_seed(M), dtype=torch.float32).cuda()
    return m, torch.from_numpy(synth.random_quaternions(T, M)).cuda()


# spectra of 2 MB and less on either side; masters of 2, 3 and 37 clamp at every edge, 513 is above 2 MB, 1,449 has no cells
@pytest.mark.parametrize("n,T", [(64, 120), (64, 130), (128, 31), (128, 32), (256, 9)])
@pytest.mark.parametrize("M", [2, 3, 37, 512, 513, 1449])
def test_same_spectra_wherever_the_cells_lie(px, n, T, M):
    g = px.geometry(n, n, (0.47, 0.55, 0.62))
    m, q = _inputs(M, T)
    c = px.Context()
    lib = px.xcf_build_library(c, m, q, g)
    spec, _, _ = px.xcf_prep(c, px.xcf_project(c, m, q, g), g)
    assert torch.equal(torch.view_as_real(lib.spectra()), torch.view_as_real(spec))
    seeds = q[:2].contiguous()
    pats = px.xcf_project(c, m, seeds, g)
    one = px.xcf_build_library(c, m, seeds[:1].contiguous(), g)   # its cells may lie elsewhere, or be missing
    a, b = px.xcf_refine(c, lib, pats, seeds), px.xcf_refine(c, one, pats, seeds)
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    one.close()
    lib.close()
    c.close()


@pytest.mark.parametrize("M,T,interp,most", [(256, 4, 0, 0.6), (512, 4, 1, 4.2), (1024, 4, 1, 8.5)])
def test_small_and_bicubic_libraries_take_no_cells(px, M, T, interp, most):
    """Ten libraries take what their spectra, orientations and masters take (`most` MB
    each), in mappings of 2 MB: no cells (16 bytes per master pixel more)."""
    g = px.geometry(64, 64)
    m, q = _inputs(M, T)
    c = px.Context(master_interp=interp)
    px.xcf_build_library(c, m, q, g).close()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    libs = [px.xcf_build_library(c, m, q, g) for _ in range(10)]
    torch.cuda.synchronize()
    taken = free - torch.cuda.mem_get_info()[0]
    each = most if most < 2 else 2 * (int(most) // 2 + 1)
    assert taken <= (10 * each + 6) * MB
    for lib in libs:
        lib.close()
    c.close()
