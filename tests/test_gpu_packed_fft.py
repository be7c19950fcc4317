"""The FP32 transforms' packed complex arithmetic at every line length: matrix
elements in single precision against those in double precision, on grids that
the spheres fill (whole lines) and whose quarters they fill (the two outer
quarters of each line).

Bound: a transform multiplies the norm by a constant and its stages' roundings
add up in it; two transforms of three axes, at most four stages of at most
three roundings each: 72 u of the norm of the whole product."""
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


def _on_grid(g, c, n):
    u = np.zeros((len(c), n, n, n), dtype=complex)
    u[:, g[:, 0], g[:, 1], g[:, 2]] = c
    return np.fft.ifftn(u, axes=(1, 2, 3)) * n ** 1.5


@pytest.mark.parametrize("whole", [False, True])
@pytest.mark.parametrize("n", [8, 10, 12, 16, 20, 24, 30, 32, 36, 40, 48, 50, 60, 64])
def test_single_against_double(n, whole):
    from paper_1111_4429_gb300 import bgw
    rng = np.random.default_rng(n)
    e = n // 4 if whole else max(1, n // 4 - 1)      # |k| < n / 4: the quarters' form
    w = (n - 1 - e) // 2                             # 2 w + e + 1 points needed: n or n - 1
    gv, gc, ge = _box(-w, w, 60, rng), _box(-w, w, 60, rng), _box(-e, e, 40, rng)
    cv = rng.standard_normal((3, len(gv))) + 1j * rng.standard_normal((3, len(gv)))
    cc = rng.standard_normal((5, len(gc))) + 1j * rng.standard_normal((5, len(gc)))
    ctx = bgw.Context(0)
    cell = bgw.make_cell(np.eye(3) * 0.3, 8641.0, (0.1, 0.0, 0.0), n)
    out = []
    for prec, dt in ((0, torch.complex128), (1, torch.complex64)):
        M = torch.zeros((15, len(ge)), dtype=dt, device="cuda")
        ctx.mtxel(cell, gv, torch.from_numpy(cv).cuda(), gc, torch.from_numpy(cc).cuda(), ge, prec, M)
        ctx.sync()
        out.append(M.cpu().numpy().astype(complex))
    uv, uc = _on_grid(gv, cv, n), _on_grid(gc, cc, n)
    whole_norm = np.sqrt(n ** 3 * sum(np.linalg.norm(a.conj() * b) ** 2 for a in uv for b in uc)) / n ** 1.5
    assert np.linalg.norm(out[1] - out[0]) <= 72 * 2.0 ** -24 * max(whole_norm, np.linalg.norm(out[0]))
