"""FP64 inverses under the default BGW_OPT_INVERSE: the options that trade accuracy for speed in the mixed precisions
(BGW_OPT_UPDATE_SLICES = 5, BGW_OPT_DOUBLE_FP32 = 1) leave them as they are, bit for bit, and within the FP64 bar."""
import numpy as np
import pytest

import oracle
from paper_1111_4429_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("call", ["epsinv", "epsinv_general", "epsinv_rflavor", "epsilon"])
@pytest.mark.parametrize("option", ["BGW_OPT_UPDATE_SLICES", "BGW_OPT_DOUBLE_FP32"])
def test_options_leave_fp64_alone(call, option):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4429_gb300 import bgw
    s = synth.make_system("r", a=17.0, fft=40, ecut_wfn=8.0, ecut_eps=3.5, nv=4, nc=90, seed=89)
    cell, v = bgw.system_cell(s), oracle.coulomb(s.bvec, s.q_frac, s.geps)
    chi = oracle.solve(s)["chi"]
    if call == "epsinv_rflavor":
        chi = np.ascontiguousarray(chi.real)
    sv = np.sqrt(v)
    want = np.linalg.inv(np.eye(s.ng) - sv[:, None] * chi * sv[None, :])

    def run(value):
        ctx = bgw.Context(0)
        if value is not None:
            ctx.set_option(getattr(bgw, option), value)
        x = _dev(chi)
        inv = torch.zeros_like(x)
        if call == "epsilon":
            ctx.epsilon(cell, s.gv, _dev(s.cv), s.ev, s.gc, _dev(s.cc), s.ec, s.geps, None, bgw.BGW_PREC_FP64, 0, None,
                        inv.view(1, s.ng, s.ng))
        else:
            getattr(ctx, call)([cell], [s.geps], [x], None, [inv])
        ctx.sync()
        return inv.cpu().numpy()

    plain, optioned = run(None), run({"BGW_OPT_UPDATE_SLICES": 5, "BGW_OPT_DOUBLE_FP32": 1}[option])
    assert np.linalg.norm(plain - want) <= 1e-12 * np.linalg.norm(want)
    assert np.array_equal(plain, optioned)
