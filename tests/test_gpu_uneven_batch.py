"""Batches of Hermitian inverses of uneven sizes, where the smaller matrix
finishes while the larger one's bulk update has nothing to do (both inside one
row tile of 128), one step earlier, later, or in a tile of its own; with the FP64
chain and with the double-FP32 one, in both widths of the update's items.

Bound: forward error of Gauss-Jordan elimination on a positive definite matrix,
c n^1/2 u cond with c u = 1e-15 (FP64) or 2^-44 (double FP32: 2^-46 an operation,
four of them a step)."""
import numpy as np
import pytest

import oracle
from paper_1111_4429_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chain,cu", [(0, 1e-15), (1, 2.0 ** -44)])
@pytest.mark.parametrize("items", [-1, 0, 1])
@pytest.mark.parametrize("sizes", [(65, 40), (97, 64), (33, 97), (97, 65), (96, 33), (128, 97, 64, 20), (161, 128, 97),
                                   (300, 129, 40)])
def test_uneven(sizes, items, chain, cu):
    from paper_1111_4429_gb300 import bgw
    rng = np.random.default_rng(sum(sizes))
    ctx = bgw.Context(0)
    bvec, _ = synth.cubic_cell(30.0)
    allg = synth.gsphere(bvec, (0.1, 0.0, 0.0), 12.0)
    cells, lists, chis, eps = [], [], [], []
    for n in sizes:
        g = allg[:n]
        sv = np.sqrt(oracle.coulomb(bvec, (0.1, 0.0, 0.0), g))
        x = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))) / np.sqrt(n)
        chi = -(x.conj().T @ x) / (sv[:, None] * sv[None, :])
        cells.append(bgw.make_cell(bvec, 27000.0, (0.1, 0.0, 0.0), 64))
        lists.append(g)
        chis.append(torch.from_numpy(chi).cuda())
        eps.append(np.eye(n) - sv[:, None] * chi * sv[None, :])
    invs = [torch.zeros_like(c) for c in chis]
    ctx.set_option(bgw.BGW_OPT_INVERSE, 1 if chain else -1)   # FP64 inputs take the double-FP32 chain by request only
    ctx.set_option(bgw.BGW_OPT_DOUBLE_FP32, chain)
    ctx.set_option(bgw.BGW_OPT_UPDATE_ITEMS, items)
    ctx.epsinv(cells, lists, chis, None, invs)
    ctx.sync()
    for e, inv in zip(eps, invs):
        ref = np.linalg.inv(e)
        err = np.linalg.norm(inv.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= cu * np.sqrt(len(e)) * np.linalg.cond(e)
