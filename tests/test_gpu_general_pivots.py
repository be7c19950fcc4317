"""Row selection and panel solve of the general (pivoted) inverse where their
splits can go wrong: fewer rows than a block of 32 columns, one row or column
past a block, past a warp's 8 columns of the solve and past a selection slice
of 256 rows, and matrices full of ties (a permutation), where every step has
to interchange rows.

Bound: Gauss-Jordan elimination with pivoting, forward error
<= c n^1/2 u cond(A) with a modest growth factor; c u = 1e-15 as for the
general inverse's other tests.  A permutation's inverse involves products of
zeros and ones only, so its error is that of forming eps~ (1 - v chi, a few
units of the last place of 1 per entry)."""
import numpy as np
import pytest

import oracle
from paper_1111_4429_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4429_gb300 import bgw
    return bgw.Context(0)


def _invert(ctx, eps, mode):
    from paper_1111_4429_gb300 import bgw
    ng = eps.shape[0]
    bvec, _ = synth.cubic_cell(30.0)
    geps = synth.gsphere(bvec, (0.1, 0.0, 0.0), 12.0)[:ng]
    assert geps.shape[0] == ng
    sv = np.sqrt(oracle.coulomb(bvec, (0.1, 0.0, 0.0), geps))
    chi = (np.eye(ng) - eps) / (sv[:, None] * sv[None, :])
    formed = np.eye(ng) - sv[:, None] * chi * sv[None, :]
    inv = torch.zeros((ng, ng), dtype=torch.complex128, device="cuda")
    try:
        ctx.set_option(bgw.BGW_OPT_INVERSE, mode)
        ctx.epsinv_general([bgw.make_cell(bvec, 27000.0, (0.1, 0.0, 0.0), 64)], [geps],
                           [torch.from_numpy(chi.astype(complex)).cuda()], None, [inv])
        ctx.sync()
    finally:
        ctx.set_option(bgw.BGW_OPT_INVERSE, -1)
    return inv.cpu().numpy(), formed


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("ng", [1, 2, 31, 32, 33, 64, 65, 255, 257, 289])
def test_edges(ctx, ng, mode):
    gen = np.random.default_rng(ng)
    eps = (gen.standard_normal((ng, ng)) + 1j * gen.standard_normal((ng, ng))) / np.sqrt(ng)
    got, formed = _invert(ctx, eps, mode)
    ref = np.linalg.inv(formed)
    assert np.linalg.norm(got - ref) <= 1e-15 * np.linalg.cond(formed) * ng ** 0.5 * np.linalg.norm(ref)


@pytest.mark.parametrize("ng", [31, 64, 300, 520])
def test_permutation(ctx, ng):
    perm = np.random.default_rng(ng).permutation(ng)
    eps = np.zeros((ng, ng), dtype=complex)
    eps[np.arange(ng), perm] = 1j
    got, formed = _invert(ctx, eps, 0)
    assert np.abs(got - np.conj(eps).T).max() <= 1e-14
