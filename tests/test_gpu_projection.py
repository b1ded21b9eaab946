"""Projection lookups: a library's templates, looked up in the master's 2 x 2
cells (or, for masters above their size limit, in the master itself), equal
xcf_project's four plain loads bit for bit, then xcf_prep's spectra; and both
match the FP64 projector."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def px():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_11313_gb300 as px
    px.load()
    return px


def _quats():
    q = synth.random_quaternions(5, 3)
    # axis-aligned frames look along the square's axes, its diagonals and the poles
    s = np.sqrt(0.5)
    return np.concatenate([q, [[1, 0, 0, 0], [s, s, 0, 0], [s, 0, s, 0], [0, 0, 1, 0], [np.cos(np.pi / 8), 0, 0, np.sin(np.pi / 8)]]])


# 1,448 is the largest master kept as cells; 2 and 3 clamp at every edge
@pytest.mark.parametrize("M", [2, 3, 37, 1448, 1449])
@pytest.mark.parametrize("n,W,H", [(64, 64, 64), (128, 131, 140), (256, 256, 256)])
def test_library_lookup_equals_projection(px, M, n, W, H):
    g = px.geometry(W, H, (0.47, 0.55, 0.62))
    master = torch.rand((2, M, M), generator=torch.Generator().manual_seed(M), dtype=torch.float32).cuda()
    q = torch.from_numpy(_quats()).cuda()
    c = px.Context()
    lib = px.xcf_build_library(c, master, q, g)
    spec, _, _ = px.xcf_prep(c, px.xcf_project(c, master, q, g), g)
    assert torch.equal(torch.view_as_real(lib.spectra()), torch.view_as_real(spec))
    lib.close()
    c.close()


@pytest.mark.parametrize("W,H", [(1, 5), (7, 3), (64, 64), (333, 97)])
def test_projection_matches_oracle_on_any_detector(px, orc, W, H):
    """Row and column stepping for detectors of any width; bound: the FP32
    frame, ray and map against FP64, as for the square detectors (2e-3 of the
    master's range at single pixels, 1e-4 at the 99th percentile)."""
    master = synth.master_pattern("bcc", 256)
    q, pc, side = _quats(), (0.5, 0.5, 0.6), max(W, H)
    c = px.Context()
    got = px.xcf_project(c, torch.from_numpy(master.copy()).cuda(), torch.from_numpy(q).cuda(), px.geometry(W, H, pc)).cpu().numpy()
    # the same rays on the square detector of side max(W, H): pixel offsets from the pattern centre agree
    pcs = (0.5 * W / side, 1 - 0.5 * H / side, 0.6 * W / side)
    ref = orc.project_many(master, q, (pcs[0], 0.5 * H / side, pcs[2]), side)[:, :H, :W]
    d = np.abs(got - ref) / (master.max() - master.min())
    assert d.max() < 2e-3 and np.quantile(d, 0.99) < 1e-4
    c.close()
