"""FP64 inverses of eps~ whose diagonal is graded (a macroscopic constant of 1e4 to 1e8 in the head, as a metal has at a
small q, or diagonals that vary): the tensor-core update loses no more than the FP64 FMA sweep.

Bound: Gauss-Jordan elimination of a positive definite matrix is as accurate as the matrix scaled to a unit diagonal
allows, c n^1/2 u cond of the scaled matrix with c u = 1e-15; the pivoted elimination is not free of the grading where
it is not in the first row, so it is held to that bound for graded heads only."""
import numpy as np
import pytest

import oracle
from paper_1111_4429_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
Q = (0.1, 0.0, 0.0)


def _exact_inverse(a):
    """Inverse in extended precision: Newton steps from NumPy's."""
    a = a.astype(np.clongdouble)
    x = np.linalg.inv(a.astype(complex)).astype(np.clongdouble)
    for _ in range(3):
        x = x + x @ (np.eye(len(a)) - a @ x)
    return x


@pytest.mark.parametrize("call,grading", [(c, g) for c in ("epsinv", "epsinv_general", "epsinv_rflavor")
                                          for g in (1e2, 1e3, 1e4)] + [("epsinv", "varied"), ("epsinv_rflavor", "varied")])
@pytest.mark.parametrize("n", [40, 90])
def test_graded_diagonal(call, grading, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4429_gb300 import bgw
    rng = np.random.default_rng(n)
    bvec, _ = synth.cubic_cell(30.0)
    g = synth.gsphere(bvec, Q, 12.0)[:n]
    sv = np.sqrt(oracle.coulomb(bvec, Q, g))
    x = rng.standard_normal((2 * n, n)) + (0 if call == "epsinv_rflavor" else 1j * rng.standard_normal((2 * n, n)))
    x /= np.sqrt(2 * n)
    d = 2.0 ** rng.uniform(-10, 10, n) if grading == "varied" else np.r_[grading, np.ones(n - 1)]
    chi = (np.eye(n) - d[:, None] * (np.eye(n) + x.conj().T @ x) * d[None, :]) / (sv[:, None] * sv[None, :])
    chi = 0.5 * (chi + chi.conj().T)
    c = torch.from_numpy(chi).cuda()
    inv, eps = torch.zeros_like(c), torch.zeros_like(c)
    ctx = bgw.Context(0)
    getattr(ctx, call)([bgw.make_cell(bvec, 27000.0, Q, 64)], [g], [c], [eps], [inv])
    ctx.sync()
    e = eps.cpu().numpy()
    u = np.sqrt(np.abs(np.diag(e)))
    scaled = e / np.outer(u, u)
    ref = _exact_inverse(scaled.astype(np.clongdouble))
    err = np.linalg.norm((inv.cpu().numpy() * np.outer(u, u) - ref).astype(complex))
    assert err <= 1e-15 * np.sqrt(n) * np.linalg.cond(scaled) * np.linalg.norm(ref.astype(complex))
