"""The FP64 inverse with tensor-core updates: sizes around the block and tile
edges against a refined inverse, matrices of different sizes in one batch,
values that are not finite, and budgets without room for the slices."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _problem(ng, seed, real=False):
    """A chi whose eps~ has a condition number of a few hundred."""
    from paper_1111_4429_gb300 import bgw, synth
    b, omega = synth.cubic_cell(20.52)
    ge = synth.gsphere(b, (0.1, 0.0, 0.0), 4.0)[:ng]
    r = np.random.default_rng(seed)
    sv = np.sqrt(4 * np.pi / (((ge + np.array([0.1, 0, 0])) @ b) ** 2).sum(1))
    k = max(4, ng // 8)
    x = r.standard_normal((k, ng)) + (0 if real else 1j * r.standard_normal((k, ng)))
    x = x / sv * (8 / np.sqrt(k)) / (1 + 3 * r.random(ng))
    chi = -(x.conj().T @ x)
    chi = 0.5 * (chi + chi.conj().T)
    return bgw.make_cell(b, omega, (0.1, 0.0, 0.0), 40), ge, chi


def _check(eps, inv):
    # forward error of Gauss-Jordan on a positive definite matrix: at most 8 n^(5/2) u cond (Higham, Accuracy and
    # Stability of Numerical Algorithms, section 14.4), held here with n in place of n^(5/2); the reference
    # (LU inverse and one Newton step) is within a few u cond itself
    n = eps.shape[0]
    ref = np.linalg.inv(eps)
    ref = ref + ref @ (np.eye(n) - eps @ ref)
    assert np.linalg.norm(inv - ref) <= 8 * n * 2.0 ** -53 * np.linalg.cond(eps) * np.linalg.norm(ref)


@pytest.mark.parametrize("mode", [-1, 0])
def test_batch_of_edge_sizes(mode):
    from paper_1111_4429_gb300 import bgw
    ctx = bgw.Context(0)
    ctx.set_option(bgw.BGW_OPT_INVERSE, mode)
    sizes = [1, 31, 33, 64, 95, 127, 128, 129, 160, 257, 385]
    probs = [_problem(n, n) for n in sizes]
    chis = [torch.from_numpy(p[2]).cuda() for p in probs]
    eps, inv = [torch.zeros_like(x) for x in chis], [torch.zeros_like(x) for x in chis]
    ctx.epsinv([p[0] for p in probs], [p[1] for p in probs], chis, eps, inv)
    ctx.sync()
    for e, x in zip(eps, inv):
        _check(e.cpu().numpy(), x.cpu().numpy())
        assert torch.equal(x, x.conj().T.resolve_conj())


@pytest.mark.parametrize("ng", [20, 33, 129, 300])
def test_real_and_general(ng):
    from paper_1111_4429_gb300 import bgw
    ctx = bgw.Context(0)
    cell, ge, chi = _problem(ng, 3 * ng, real=True)
    x, e, v = torch.from_numpy(chi.real.copy()).cuda(), torch.zeros((ng, ng), dtype=torch.float64, device="cuda"), None
    v = torch.zeros_like(e)
    ctx.epsinv_rflavor([cell], [ge], [x], [e], [v])
    ctx.sync()
    _check(e.cpu().numpy(), v.cpu().numpy())
    cell, ge, chi = _problem(ng, 5 * ng)
    g = torch.from_numpy(chi * (1 + 0.3j)).cuda()
    e, v = torch.zeros_like(g), torch.zeros_like(g)
    ctx.epsinv_general([cell], [ge], [g], [e], [v])
    ctx.sync()
    _check(e.cpu().numpy(), v.cpu().numpy())


def test_small_budget_and_values_that_are_not_finite():
    from paper_1111_4429_gb300 import bgw
    cell, ge, chi = _problem(300, 8)
    x = torch.from_numpy(chi).cuda()
    for budget in (0, 1 << 20):   # room for the panels only: the FMA sweep
        ctx = bgw.Context(0, budget)
        e, v = torch.zeros_like(x), torch.zeros_like(x)
        ctx.epsinv([cell], [ge], [x], [e], [v])
        ctx.sync()
        _check(e.cpu().numpy(), v.cpu().numpy())
    x[270, 40] = float("nan")     # an element of the lower triangle off the diagonal blocks
    ctx = bgw.Context(0)
    ctx.epsinv([cell], [ge], [x], None, [torch.zeros_like(x)])
    with pytest.raises(bgw.BgwError) as err:
        ctx.sync()
    assert err.value.code == bgw.BGW_ENUMERIC
    # a scale below FP64's range in the products (the pair exponents' sum) is zero, not garbage
    d = torch.zeros((70, 70), dtype=torch.complex128, device="cuda")
    d[40, 3] = d[3, 40] = -1e-250
    d[50, 60] = d[60, 50] = -1e-3
    out, e = torch.zeros_like(d), torch.zeros_like(d)
    ctx.epsinv([cell], [ge[:70]], [d], [e], [out])
    ctx.sync()
    _check(e.cpu().numpy(), out.cpu().numpy())
