"""The FP64 polarizability by digit products on the tensor cores: tile edges,
short and ragged pair counts, accumulation, chunked calls under a small HBM
budget, and operands that are not finite (the FP64 FMA kernel's)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELL = (np.eye(3) * 0.3, 8641.0, (0.1, 0.0, 0.0), 40)


def _case(ng, nv, nc, seed, real=False):
    r = np.random.default_rng(seed)
    m = r.standard_normal((nv * nc, ng)) + (0 if real else 1j * r.standard_normal((nv * nc, ng)))
    m = m * np.exp2(r.integers(-20, 20, ng))          # columns of very different sizes
    return m, np.sort(r.uniform(-0.5, 0.0, nv)), np.sort(r.uniform(0.04, 1.5, nc))


def _ref(m, ev, ec, omega):
    d = np.subtract.outer(ev, ec).ravel()
    w = 1.0 / d if omega is None else d / (d * d + omega * omega)
    return (m.conj().T * w) @ m * (4.0 / CELL[1])


def _err(x, ref):
    # per element, against the columns' norms: |chi_GG'| <= (chi_GG chi_G'G')^1/2, so a sum of K terms in FP64
    # is within K 2^-53 of it (NumPy's reference included), the digit products within 2^-58 (6 K)^1/2 2^2
    s = np.sqrt(np.abs(np.diagonal(ref)))
    return np.abs((x - ref) / np.outer(s, s)).max()


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("ng,nv,nc", [(1, 1, 8), (31, 2, 4), (32, 3, 5), (33, 1, 16), (127, 1, 17), (128, 4, 48),
                                      (129, 1, 193), (160, 5, 77), (257, 3, 9), (300, 2, 500)])
def test_edges_against_numpy(ng, nv, nc, real):
    from paper_1111_4429_gb300 import bgw
    ctx, cell = bgw.Context(0), bgw.make_cell(*CELL)
    m, ev, ec = _case(ng, nv, nc, 17 * ng + nc, real)
    M = torch.from_numpy(m).cuda()
    om = np.array([0.0, 0.7])
    chi = torch.zeros((2, ng, ng), dtype=M.dtype, device="cuda")
    prec = bgw.BGW_FLAVOR_REAL if real else 0
    for acc in (False, True):
        ctx.chi_sum(cell, nv, nc, ng, M, ev, ec, om, prec, acc, chi)
    ctx.sync()
    for f in range(2):
        ref = 2 * _ref(m, ev, ec, om[f])
        x = chi[f].cpu().numpy()
        assert _err(x, ref) <= 4 * nv * nc * 2.0 ** -53
        assert np.array_equal(x, x.conj().T)


def test_general_product_and_small_budget():
    from paper_1111_4429_gb300 import bgw
    ng, nv, nc = 140, 6, 400
    m, ev, ec = _case(ng, nv, nc, 5)
    M = torch.from_numpy(m).cuda()
    e = np.array([0.3])
    d = np.subtract.outer(ev, ec).ravel()
    w = 0.5 * (1 / (d - 0.3 - 0.05j) + 1 / (d + 0.3 + 0.05j))
    ref = (m.conj().T * w) @ m * (4.0 / CELL[1])
    s = np.sqrt((np.abs(m) ** 2).sum(0))
    # whole, in chunks of pairs, and with no room for the digits (FMA kernel)
    for budget in (0, 24 << 20, 1 << 20):
        ctx, cell = bgw.Context(0, budget), bgw.make_cell(*CELL)
        x = torch.zeros((1, ng, ng), dtype=torch.complex128, device="cuda")
        ctx.chi_sum_real(cell, nv, nc, ng, M, ev, ec, e, 0.05, False, 0, False, x)
        ctx.sync()
        got = (x[0].cpu().numpy() - ref) / np.outer(s, s)
        assert np.abs(got).max() <= nv * nc * 2.0 ** -53 * np.abs(w).max() * 4 / CELL[1]
        h = torch.zeros((1, ng, ng), dtype=torch.complex128, device="cuda")
        ctx.chi_sum(cell, nv, nc, ng, M, ev, ec, None, 0, False, h)
        ctx.sync()
        assert _err(h[0].cpu().numpy(), _ref(m, ev, ec, None)) <= 2 * nv * nc * 2.0 ** -53


def test_values_that_are_not_finite_take_the_fma_kernel():
    from paper_1111_4429_gb300 import bgw
    ctx, cell = bgw.Context(0), bgw.make_cell(*CELL)
    ng, nv, nc = 70, 2, 20
    m, ev, ec = _case(ng, nv, nc, 9)
    m[3, 17] = complex(np.inf, 0.0)
    m[9, 40] = complex(np.nan, 1.0)
    chi = torch.zeros((1, ng, ng), dtype=torch.complex128, device="cuda")
    ctx.chi_sum(cell, nv, nc, ng, torch.from_numpy(m).cuda(), ev, ec, None, 0, False, chi)
    ctx.sync()
    bad = ~np.isfinite(chi[0].cpu().numpy())
    rows = np.zeros(ng, bool)
    rows[[17, 40]] = True
    assert np.array_equal(bad, rows[:, None] | rows[None, :])


@pytest.mark.parametrize("no,ni,nocc", [(1, 1, 1), (1, 127, 9), (2, 64, 5), (3, 43, 4), (5, 77, 7)])
def test_sigma_forms_at_tile_edges(no, ni, nocc):
    """K = no ni pairs around the 128-row tile, whole and in blocks of pairs
    under a budget, against the oracle (the FP64 bar of the Sigma tests)."""
    import oracle
    from paper_1111_4429_gb300 import bgw, synth
    s = synth.make_system("sd", a=14.0, fft=24, ecut_wfn=6.0, ecut_eps=2.5, nv=3, nc=20, seed=61)
    r = oracle.solve(s)
    sb = synth.sigma_bands(s, no, ni, nocc, seed=ni)
    ref = oracle.sigma_cohsex(sb.gi, sb.ci, nocc, sb.go, sb.co, s.geps, r["epsinv"], r["v"], s.omega)
    for budget in (0, 48 << 20):
        ctx = bgw.Context(0, budget)
        got = ctx.sigma_cohsex(bgw.system_cell(s), sb.go, torch.from_numpy(sb.co).cuda(), sb.gi,
                               torch.from_numpy(sb.ci).cuda(), nocc, s.geps, torch.from_numpy(r["epsinv"]).cuda())
        for k, key in enumerate(("X", "SX", "CH")):
            want = np.real(ref[key])
            assert np.abs(got[k] - want).max() <= 1e-12 * np.abs(want).max()


@pytest.mark.parametrize("real", [False, True])
def test_columns_below_the_normal_range(real):
    """A column of subnormals against one near 1e290: their element of chi is an ordinary number.  Rounding an operand
    near 1e-309 to the subnormals' spacing of 5e-324 costs 5e-15 of it."""
    from paper_1111_4429_gb300 import bgw
    ctx, cell = bgw.Context(0), bgw.make_cell(*CELL)
    ng, nv, nc = 3, 2, 40
    r = np.random.default_rng(8)
    m = r.standard_normal((nv * nc, ng)) + (0 if real else 1j * r.standard_normal((nv * nc, ng)))
    m[:, 1] = m[:, 0] * np.exp(0.2j if not real else 0.0) + 0.1 * m[:, 1]
    big, small = m * 1.0, m[:, 0] * 1e-309
    m = np.stack([small, m[:, 1] * 1e290, m[:, 2]], 1)
    ev, ec = np.sort(r.uniform(-0.5, 0.0, nv)), np.sort(r.uniform(0.04, 1.5, nc))
    chi = torch.zeros((1, ng, ng), dtype=torch.float64 if real else torch.complex128, device="cuda")
    ctx.chi_sum(cell, nv, nc, ng, torch.from_numpy(m).cuda(), ev, ec, None, bgw.BGW_FLAVOR_REAL if real else 0, False,
                chi)
    ctx.sync()
    w = 1.0 / np.subtract.outer(ev, ec).ravel()
    want = np.sum(big[:, 0].conj() * w * (m[:, 1] * 1e-290)) * 1e-19 * (4.0 / CELL[1])
    assert abs(chi[0, 0, 1].item() - want) <= 1e-13 * abs(want)


def _exact_product(x, y):
    """sum_p conj(x_p) y_p of [K][a] and [K][b] in extended precision."""
    q = np.clongdouble
    return np.einsum("pa,pb->ab", x.conj().astype(q), y.astype(q))


# Pairs at most 2^9 apart (sizes up to 8 apart) keep operands to 2^(10 - 57) of their own largest entry, about 3
# standard deviations: 2^-45 of a block's norm.  Pairs further apart take running FP64 sums, K^1/2 2^-53.
@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("spread", [0, 6, 9, 13, 20, 27, 40])
def test_blocks_made_by_the_smaller_pairs(spread, real):
    """One pair 2^spread larger than the others in some columns and zero in the rest: the block between the two groups
    of columns is made by the smaller pairs alone."""
    from paper_1111_4429_gb300 import bgw
    ctx, cell = bgw.Context(0), bgw.make_cell(*CELL)
    ng, nv, nc = 40, 4, 60
    r = np.random.default_rng(spread)
    m = r.standard_normal((nv * nc, ng)) + (0 if real else 1j * r.standard_normal((nv * nc, ng)))
    m[7, :15] *= 2.0 ** spread
    m[7, 15:] = 0.0
    ev, ec = np.sort(r.uniform(-0.5, 0.0, nv)), np.sort(r.uniform(0.5, 1.5, nc))
    chi = torch.zeros((1, ng, ng), dtype=torch.float64 if real else torch.complex128, device="cuda")
    ctx.chi_sum(cell, nv, nc, ng, torch.from_numpy(m).cuda(), ev, ec, None, bgw.BGW_FLAVOR_REAL if real else 0, False,
                chi)
    ctx.sync()
    w = 1.0 / np.subtract.outer(ev, ec).ravel()
    want = (_exact_product(m[:, :15], m[:, 15:] * w[:, None]) * (4.0 / CELL[1])).astype(complex)
    got = chi[0].cpu().numpy()[:15, 15:]
    assert np.linalg.norm(got - want) <= 2.0 ** -45 * np.linalg.norm(want)


@pytest.mark.parametrize("delta", [0.05, 1e-4, 1e-8])
def test_resonance_on_the_real_axis(delta):
    """One pair in resonance, its elements zero in the second group of columns."""
    from paper_1111_4429_gb300 import bgw
    ctx, cell = bgw.Context(0), bgw.make_cell(*CELL)
    ng, nv, nc = 40, 4, 60
    r = np.random.default_rng(4)
    m = r.standard_normal((nv * nc, ng)) + 1j * r.standard_normal((nv * nc, ng))
    m[7, 15:] = 0.0
    ev, ec = np.sort(r.uniform(-0.5, 0.0, nv)), np.sort(r.uniform(0.5, 1.5, nc))
    d = np.subtract.outer(ev, ec).ravel()
    e = np.array([-d[7]])
    x = torch.zeros((1, ng, ng), dtype=torch.complex128, device="cuda")
    ctx.chi_sum_real(cell, nv, nc, ng, torch.from_numpy(m).cuda(), ev, ec, e, delta, False, 0, False, x)
    ctx.sync()
    w = 0.5 * (1 / (d - e[0] - 1j * delta) + 1 / (d + e[0] + 1j * delta))
    got = x[0].cpu().numpy()
    for rows, cols in ((slice(0, 15), slice(15, ng)), (slice(15, ng), slice(0, 15))):
        want = (_exact_product(m[:, rows], m[:, cols] * w[:, None]) * (4.0 / CELL[1])).astype(complex)
        assert np.linalg.norm(got[rows, cols] - want) <= 2.0 ** -45 * np.linalg.norm(want)
