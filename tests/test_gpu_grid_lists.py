"""Matrix elements and Sigma of lists of very different widths (an epsilon list wider than the bands' products, one
sphere far wider than the other): every element is written and equals the defining sum, and runs repeat bit for bit."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _box(lo, hi):
    ax = np.arange(lo, hi + 1)
    return np.ascontiguousarray(np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3).astype(np.int32))


def _bands(rng, nb, g):
    c = rng.standard_normal((nb, len(g))) + 1j * rng.standard_normal((nb, len(g)))
    return c / np.linalg.norm(c, axis=1, keepdims=True)


@pytest.mark.parametrize("v,c,e,n", [((-1, 1), (-1, 1), (-4, 4), 20), ((-6, 6), (-1, 1), (-1, 1), 20),
                                     ((-1, 1), (-7, 7), (-2, 2), 24), ((0, 0), (0, 0), (-5, 4), 16)])
@pytest.mark.parametrize("prec,tol", [(0, 1e-12), (1, 1e-5)])
def test_elements(v, c, e, n, prec, tol):
    from paper_1111_4429_gb300 import bgw
    rng = np.random.default_rng(n + 7 * e[1])
    gv, gc, ge = _box(*v), _box(*c), _box(*e)
    cv, cc = _bands(rng, 3, gv), _bands(rng, 4, gc)
    cell = bgw.make_cell(np.eye(3) * 0.3, 8641.0, (0.1, 0.0, 0.0), n)
    runs = []
    for _ in range(2):
        ctx = bgw.Context(0)
        M = torch.full((12, len(ge)), float("nan"), dtype=torch.complex128 if prec == 0 else torch.complex64,
                       device="cuda")
        ctx.mtxel(cell, gv, torch.from_numpy(cv).cuda(), gc, torch.from_numpy(cc).cuda(), ge, prec, M)
        ctx.sync()
        runs.append(M.cpu().numpy())
    ref = oracle.mtxel_direct(gv, cv, gc, cc, ge)
    assert np.linalg.norm(runs[0].reshape(ref.shape) - ref) <= tol * np.linalg.norm(ref)
    assert np.array_equal(runs[0], runs[1])


# the grids that the next one with low-band lines replaces: 50 by 60 (FP32), 60 by 64
@pytest.mark.parametrize("w,e,n", [(18, 12, 60), (18, 12, 50), (21, 15, 64), (21, 15, 60), (20, 14, 64)])
@pytest.mark.parametrize("prec,tol", [(0, 1e-12), (1, 1e-5)])
def test_low_band_neighbours(w, e, n, prec, tol):
    from paper_1111_4429_gb300 import bgw
    rng = np.random.default_rng(w + e)

    def some(r, keep):
        g = rng.integers(-r, r + 1, (keep, 3))
        return np.unique(np.concatenate([g, [[r, -r, 0], [-r, r, r], [0, 0, -r]]]), axis=0).astype(np.int32)
    gv, gc, ge = some(w, 300), some(w, 300), some(e, 200)
    cv, cc = _bands(rng, 5, gv), _bands(rng, 4, gc)
    ctx = bgw.Context(0)
    M = torch.full((20, len(ge)), float("nan"), dtype=torch.complex128 if prec == 0 else torch.complex64, device="cuda")
    ctx.mtxel(bgw.make_cell(np.eye(3) * 0.3, 8641.0, (0.1, 0.0, 0.0), n), gv, torch.from_numpy(cv).cuda(), gc,
              torch.from_numpy(cc).cuda(), ge, prec, M)
    ctx.sync()
    ref = oracle.mtxel_direct(gv, cv, gc, cc, ge)
    assert np.linalg.norm(M.cpu().numpy().reshape(ref.shape) - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("o,i,e,n", [((-1, 1), (-1, 1), (-4, 4), 20), ((-1, 1), (-6, 6), (-2, 2), 20)])
def test_sigma(o, i, e, n):
    from paper_1111_4429_gb300 import bgw
    rng = np.random.default_rng(n + 3 * e[1])
    go, gi, ge = _box(*o), _box(*i), _box(*e)
    co, ci = _bands(rng, 2, go), _bands(rng, 5, gi)
    q = np.array([0.1, 0.05, 0.0])
    b = np.eye(3) * 0.3
    x = rng.standard_normal((8, len(ge))) + 1j * rng.standard_normal((8, len(ge)))
    inv = 0.7 * np.eye(len(ge)) - 0.5 * (x.conj().T @ x) / np.linalg.norm(x) ** 2
    cell = bgw.make_cell(b, 8641.0, q, n)
    ctx = bgw.Context(0)
    got = ctx.sigma_cohsex(cell, go, torch.from_numpy(co).cuda(), gi, torch.from_numpy(ci).cuda(), 2, ge,
                           torch.from_numpy(inv).cuda())
    ref = oracle.sigma_cohsex(gi, ci, 2, go, co, ge, inv, oracle.coulomb(b, q, ge), 8641.0)
    for k, key in enumerate(("X", "SX", "CH", "CH_exact")):
        r = np.real(ref[key])
        assert np.abs(got[k] - r).max() <= 1e-12 * np.abs(r).max(), key
