"""The product transform's own grid: matrix elements of spheres that need fewer
points than the caller's grid equal the defining sums, at the sizes where the
choice of grid changes."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _box(lo, hi, keep, rng):
    """Points of the box [lo, hi]^3 with its extreme corners, about `keep` of them."""
    ax = np.arange(lo, hi + 1)
    g = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    pick = rng.random(len(g)) < keep / len(g)
    pick[[0, -1]] = True
    return np.ascontiguousarray(g[pick].astype(np.int32))


# wavefunction bound, epsilon bounds, caller's grid: need = 2 wfn + max|eps| + 1
@pytest.mark.parametrize("w,lo,hi,n", [(2, -1, 1, 16), (2, -2, 2, 8), (3, -3, 3, 20), (4, -2, 2, 12), (5, -2, 2, 20),
                                       (10, -8, 7, 40), (10, -8, 8, 40), (10, -8, 7, 30), (11, -8, 7, 32),
                                       (11, -9, 9, 40), (13, -9, 9, 36), (16, -12, 11, 60), (17, -12, 12, 64),
                                       (18, -13, 13, 50)])
@pytest.mark.parametrize("prec,tol", [(0, 1e-12), (1, 1e-5)])
def test_smaller_grid_matches_definition(w, lo, hi, n, prec, tol):
    from paper_1111_4429_gb300 import bgw
    rng = np.random.default_rng(1000 * w + 10 * hi + n)
    gv, gc, ge = _box(-w, w, 60, rng), _box(-w, w, 60, rng), _box(lo, hi, 40, rng)
    cv = rng.standard_normal((3, len(gv))) + 1j * rng.standard_normal((3, len(gv)))
    cc = rng.standard_normal((5, len(gc))) + 1j * rng.standard_normal((5, len(gc)))
    cv /= np.linalg.norm(cv, axis=1, keepdims=True)
    cc /= np.linalg.norm(cc, axis=1, keepdims=True)
    ctx = bgw.Context(0)
    M = torch.zeros((15, len(ge)), dtype=torch.complex128 if prec == 0 else torch.complex64, device="cuda")
    cell = bgw.make_cell(np.eye(3) * 0.3, 8641.0, (0.1, 0.0, 0.0), n)
    ctx.mtxel(cell, gv, torch.from_numpy(cv).cuda(), gc, torch.from_numpy(cc).cuda(), ge, prec, M)
    ctx.sync()
    ref = oracle.mtxel_direct(gv, cv, gc, cc, ge)
    assert np.linalg.norm(M.cpu().numpy().reshape(ref.shape) - ref) <= tol * np.linalg.norm(ref)
