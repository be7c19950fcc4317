"""Tensor-core inverses under a memory budget: with room for one set of the update's slices only, the sweep runs without
overlap and gives the same bits as with two.  What it needs beyond the FP64 FMA sweep is at most two sets of one row
of slices for each operand, 7 x 64 FP16 values a row."""
import numpy as np
import pytest

import oracle
from paper_1111_4429_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
Q = (0.1, 0.0, 0.0)
KIB = 1 << 10


@pytest.mark.parametrize("chain", [0, 1])
@pytest.mark.parametrize("call", ["epsinv", "epsinv_general"])
def test_one_set_of_slices(call, chain):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4429_gb300 import bgw
    n = 1000
    bvec, _ = synth.cubic_cell(30.0)
    g = synth.gsphere(bvec, Q, 12.0)[:n]
    sv = torch.from_numpy(np.sqrt(oracle.coulomb(bvec, Q, g))).cuda()
    gen = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((n, n), dtype=torch.complex128, device="cuda", generator=gen) / np.sqrt(n)
    chi = -(x.conj().T @ x) / (sv[:, None] * sv[None, :])
    cell = bgw.make_cell(bvec, 27000.0, Q, 64)

    def run(budget, mode):
        ctx = bgw.Context(0, budget)
        ctx.set_option(bgw.BGW_OPT_INVERSE, mode)
        ctx.set_option(bgw.BGW_OPT_DOUBLE_FP32, chain)
        inv = torch.zeros_like(chi)
        st = torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st):
            for _ in range(3):   # direct, and replays of its graph
                getattr(ctx, call)([cell], [g], [chi], None, [inv])
            ctx.sync(st)
        return inv

    def fits(budget, mode):
        try:
            return run(budget, mode) is not None
        except bgw.BgwError as e:
            assert e.code == bgw.BGW_ENOMEM
            return False

    lo, hi = 0, 64 << 20   # the least budget (in 64 KiB) of the FP64 FMA sweep
    while hi - lo > 64 * KIB:
        mid = (lo + hi) // 2 // (64 * KIB) * (64 * KIB)
        lo, hi = (lo, mid) if fits(mid, 0) else (mid, hi)
    rows = (n + 127) // 128 * 128
    slices = 2 * 7 * rows * 64 * 2
    want = run(0, 1)
    got = run(hi + 2 * slices + 3 * 64 * KIB, 1)   # and the exponents and the diagonal block, 64 KiB each
    assert torch.equal(got, want)
    one_set = slices // 2 + slices
    assert torch.equal(run(hi + one_set + 5 * 64 * KIB, 1), want)
