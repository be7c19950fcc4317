"""A captured graph keeps the kernels of the direct run before it: FP64 calls under memory budgets of every size around
the one at which the inverse's buffers push the polarizability's digit planes out of the pool.  The results of the
direct call and of the calls after it (replays, or direct runs where the capture was given up) are equal bit for bit."""
import numpy as np
import pytest

from paper_1111_4429_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _eps_lists():
    """Two epsilon lists of 128 and 130 vectors with the same (x, y) columns: the product transform's scratch is the
    same for both, the digit planes (padded to 128 rows) are not."""
    cols = sorted(((x, y) for x in range(-3, 4) for y in range(-3, 4)), key=lambda t: t[0] ** 2 + t[1] ** 2)[:19]
    g = [(x, y, z) for z in (0, 1, -1, 2, -2, 3, -3) for x, y in cols]
    return [np.array(g[:k], dtype=np.int32) for k in (128, 130)]


def test_graph_repeats_the_direct_run():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4429_gb300 import bgw
    b, omega = synth.cubic_cell(8.0)
    q = (0.1, 0.0, 0.0)
    gv, gc = synth.gsphere(b, q, 8.0), synth.gsphere(b, (0.0, 0.0, 0.0), 8.0)
    nv, nc = 4, 250
    rng = np.random.default_rng(3)
    cv, cc = (torch.from_numpy(x / np.linalg.norm(x, axis=1, keepdims=True)).cuda() for x in
              (rng.standard_normal((k, len(g))) + 1j * rng.standard_normal((k, len(g))) for k, g in ((nv, gv), (nc, gc))))
    ev, ec = np.sort(rng.uniform(-0.5, 0.0, nv)), np.sort(rng.uniform(0.1, 1.5, nc))
    cell = bgw.make_cell(b, omega, q, 16)
    st = torch.cuda.Stream()
    lists = _eps_lists()
    out = [(torch.empty((1, len(g), len(g)), dtype=torch.complex128, device="cuda"),
            torch.empty((1, len(g), len(g)), dtype=torch.complex128, device="cuda")) for g in lists]
    ran = replayed = 0
    for budget in range(20 << 20, 100 << 20, 256 << 10):
        ctx = bgw.Context(0, budget)
        try:
            with torch.cuda.stream(st):
                def call(k):
                    chi, inv = out[k]
                    ctx.epsilon(cell, gv, cv, ev, gc, cc, ec, lists[k], None, bgw.BGW_PREC_FP64, 0, chi, inv)
                    ctx.sync(st)
                    return chi.clone(), inv.clone()
                call(0)   # its graph keeps the transform's scratch in the pool
                first = call(1)
                again = [call(1) for _ in range(2)]
                replayed += ctx.graph_stats()[1]
        except bgw.BgwError as e:
            assert e.code == bgw.BGW_ENOMEM
            continue
        ran += 1
        for r in again:
            assert torch.equal(r[0], first[0]) and torch.equal(r[1], first[1]), f"budget {budget}"
    assert ran > 10 and replayed > 0
