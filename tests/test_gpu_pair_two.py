"""Two pairs a warp in the product transform (lines of 36, 40 and 48 points, calls
of many pairs): every pair's matrix elements equal the block kernel's, for odd and
even numbers of pairs and pairs that cross from one valence band to the next.

Bound, pair by pair: each kernel's stages round at most 72 times (two transforms
of three axes, four stages of three roundings), so the two differ by at most
144 u of the norm of the pair's whole product."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _box(lo, hi, keep, rng):
    ax = np.arange(lo, hi + 1)
    g = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    pick = rng.random(len(g)) < keep / len(g)
    pick[[0, -1]] = True
    return np.ascontiguousarray(g[pick].astype(np.int32))


def _density(g, c, n):
    u = np.zeros((len(c), n, n, n), dtype=complex)
    u[:, g[:, 0], g[:, 1], g[:, 2]] = c
    return (np.abs(np.fft.ifftn(u, axes=(1, 2, 3)) * n ** 3) ** 2).reshape(len(c), -1)


@pytest.mark.parametrize("prec,u", [(0, 2.0 ** -53), (1, 2.0 ** -24)])
@pytest.mark.parametrize("nv,nc", [(7, 165), (2, 608)])
@pytest.mark.parametrize("n", [36, 40, 48])
def test_equals_block_kernel(n, nv, nc, prec, u):
    from paper_1111_4429_gb300 import bgw
    rng = np.random.default_rng(n + nv)
    e = n // 4 - 1
    w = (n - 1 - e) // 2
    gv, gc, ge = _box(-w, w, 60, rng), _box(-w, w, 60, rng), _box(-e, e, 200, rng)
    cv = rng.standard_normal((nv, len(gv))) + 1j * rng.standard_normal((nv, len(gv)))
    cc = rng.standard_normal((nc, len(gc))) + 1j * rng.standard_normal((nc, len(gc)))
    ctx = bgw.Context(0)
    cell = bgw.make_cell(np.eye(3) * 0.3, 8641.0, (0.1, 0.0, 0.0), n)
    out = []
    for kernel in (0, 1):
        ctx.set_option(bgw.BGW_OPT_PAIR_KERNEL, kernel)
        M = torch.zeros((nv * nc, len(ge)), dtype=torch.complex128 if prec == 0 else torch.complex64, device="cuda")
        ctx.mtxel(cell, gv, torch.from_numpy(cv).cuda(), gc, torch.from_numpy(cc).cuda(), ge, prec, M)
        ctx.sync()
        out.append(M.cpu().numpy().astype(complex))
    # sum over all G of |M_G|^2 is the mean of |u_v|^2 |u_c|^2 over the grid
    whole = np.sqrt(_density(gv, cv, n) @ _density(gc, cc, n).T / n ** 3).reshape(-1)
    diff = np.linalg.norm(out[1] - out[0], axis=1)
    assert np.linalg.norm(out[0]) > 0.0
    assert (diff <= 144 * u * whole).all()
