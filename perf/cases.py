"""Timed cases of the RPA epsilon path, each through the calls a program makes (``paper_1111_4429_gb300.bgw``).

A case names one entry point (``kind``), a cubic cell of side ``a`` (bohr) with its wavefunction and epsilon cutoffs
(Ry) and FFT grid ``n``, band counts, a precision and, where the call has them, frequencies.  The three cells of the
configurations (sides 10.26, 20.52 and 30.78 bohr on 20^3, 40^3 and 60^3 grids) and sizes between them make up the
range: matrix elements on grids of 16 to 64 points, epsilon spheres of about 30 to 7200 G vectors, and one to a few
hundred thousand band pairs.

Bands are complex Gaussian vectors of norm one on their plane-wave spheres (real ones for the real flavor), energies
are uniform and sorted, as the configurations draw them.  A case that starts at the polarizability takes matrix
elements whose size falls off with |q + G| as computed ones do, and a case that starts at the inverse takes a
Hermitian negative polarizability built from such elements.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1111_4429_gb300 import bgw, synth

GRIDS = (16, 20, 24, 30, 32, 36, 40, 48, 50, 60, 64)   # grids of the drawn cells
Q = (0.1, 0.0, 0.0)


# ------------------------------------------------------------------ cases
def listed():
    c0 = dict(a=10.26, n=20, wfn=10.0, eps=3.0)     # the smallest cell: an oracle-sized solve
    c1 = dict(a=20.52, n=40, wfn=12.0, eps=6.0)     # the middle cell
    c2 = dict(a=30.78, n=60, wfn=12.0, eps=6.0)     # the large cell
    return [
        # one small q-point start to end in the default precision: latency and launches
        dict(name="epsilon_small_fp64", kind="epsilon", **c0, nv=4, nc=60, prec="fp64", nfreq=0, host=False),
        # a conduction chunk's matrix elements in the default precision, an odd number of bands
        dict(name="mtxel_mid_fp64", kind="mtxel", **c1, nv=16, nc=99, prec="fp64", real=False),
        # a conduction chunk of the large cell, mixed precision (a third of the chunk the large solve streams)
        dict(name="mtxel_large_mixed", kind="mtxel", **c2, nv=108, nc=160, prec="mix_fp16", real=False),
        # the polarizability of a chunk of pairs, default precision
        dict(name="chi_mid_fp64", kind="chi", **c1, nv=32, nc=75, prec="fp64", nfreq=0, accumulate=True),
        # the polarizability of the large sphere at an imaginary frequency, mixed precision
        dict(name="chi_large_mixed", kind="chi", **c2, nv=108, nc=125, prec="mix_fp16", nfreq=1, accumulate=False),
        # inverses of two q-points with epsilon spheres of different sizes, then W, default options
        dict(name="inverse_mid_pair", kind="inverse", a=20.52, n=40, wfn=12.0, eps=6.0, eps2=4.0, coulomb="bulk"),
        # a q-point of the middle cell from and to page-locked host memory, mixed precision, in chunks of bands
        dict(name="epsilon_mid_mixed_host", kind="epsilon", **c1, nv=32, nc=800, prec="mix_fp16", nfreq=0, host=True),
        # q-points x imaginary frequencies as one batch (full-frequency work on the imaginary axis)
        dict(name="batch_mid_mixed", kind="batch", **c1, nv=32, nc=400, prec="mix_fp16", nq=2, nfreq=6),
        # the real axis with broadening: complex weights and the pivoted inverse
        dict(name="real_axis_mixed", kind="real_axis", a=20.52, n=40, wfn=12.0, eps=5.0, nv=32, nc=200,
             prec="mix_fp16", nfreq=5, delta=0.05),
        # the real flavor (inversion symmetry), mixed precision, a grid between the configurations'
        dict(name="epsilon_real_flavor", kind="epsilon_real_flavor", a=25.65, n=50, wfn=10.0, eps=5.0, nv=48, nc=301,
             prec="mix_fp16"),
        # diagonal static COHSEX and bare exchange of a few bands, default precision
        dict(name="sigma_mid_fp64", kind="sigma", a=15.39, n=30, wfn=12.0, eps=6.0, no=4, ni=150, nocc=14,
             prec="fp64"),
        # the whole large solve, mixed precision: the headline workload
        dict(name="epsilon_large_mixed", kind="epsilon", **c2, nv=108, nc=3000, prec="mix_fp16", nfreq=0, host=False,
             chunk=500),
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _cell(rng, n_hi):
    n = rng.choice([g for g in GRIDS if g <= n_hi])
    return dict(a=round(n * rng.uniform(0.45, 0.513), 3), n=n, wfn=round(rng.uniform(8.0, 12.0), 2),
                eps=round(rng.uniform(2.5, 6.0), 2))


def draw(rng):
    kind = rng.choice(["mtxel", "mtxel", "chi", "chi", "inverse", "epsilon", "epsilon", "batch", "real_axis",
                       "epsilon_real_flavor", "sigma"])
    prec = rng.choice(["fp64", "mix_fp16", "mix_fp16", "mix_bf16"])
    wide = prec != "fp64"
    if kind == "mtxel":
        c = _cell(rng, 64 if wide else 48)
        nv = _logint(rng, 1, 108)
        top = (20000 if wide else 1600) * (60 if wide else 40) ** 3 // c["n"] ** 3
        return dict(kind=kind, **c, nv=nv, nc=_logint(rng, 1, max(2, min(3000, top // nv))), prec=prec,
                    real=rng.random() < 0.2)
    if kind == "chi":
        c = _cell(rng, 60 if wide else 40)
        nv = _logint(rng, 1, 108 if wide else 32)
        return dict(kind=kind, **c, nv=nv, nc=_logint(rng, 2, 125 if wide else 75), prec=prec,
                    nfreq=rng.choice([0, 0, 1, 3 if c["n"] <= 40 else 1]), accumulate=rng.random() < 0.5)
    if kind == "inverse":
        c = _cell(rng, 40)
        return dict(kind=kind, **c, eps2=round(rng.uniform(2.0, 5.0), 2),
                    coulomb=rng.choice(["bulk", "sphere", "slab"]))
    if kind == "epsilon":
        c = _cell(rng, 50 if wide else 32)
        return dict(kind=kind, **c, nv=_logint(rng, 2, 48), nc=_logint(rng, 8, 600 if wide else 60), prec=prec,
                    nfreq=rng.choice([0, 0, 2]), host=rng.random() < 0.5)
    if kind == "batch":
        c = _cell(rng, 40 if wide else 24)
        return dict(kind=kind, **c, nv=_logint(rng, 2, 32), nc=_logint(rng, 8, 300 if wide else 60), prec=prec,
                    nq=rng.choice([1, 2, 3]), nfreq=rng.choice([2, 5, 8]))
    if kind == "real_axis":
        c = _cell(rng, 40 if wide else 24)
        return dict(kind=kind, **c, nv=_logint(rng, 2, 32), nc=_logint(rng, 8, 200 if wide else 60), prec=prec,
                    nfreq=rng.choice([1, 3, 6]), delta=round(rng.uniform(0.02, 0.1), 3))
    if kind == "epsilon_real_flavor":
        c = _cell(rng, 50 if wide else 32)
        return dict(kind=kind, **c, nv=_logint(rng, 2, 48), nc=_logint(rng, 8, 400 if wide else 60), prec=prec)
    c = _cell(rng, 40 if wide else 30)
    no, ni = _logint(rng, 1, 8), _logint(rng, 8, 400 if wide else 150)
    return dict(kind="sigma", **c, no=no, ni=ni, nocc=max(1, ni // 10), prec=prec)


# ----------------------------------------------------------------- inputs
def _spheres(case, q=Q, eps=None):
    return _spheres_of(case["a"], case["wfn"], eps or case["eps"], q)


@functools.lru_cache(maxsize=64)
def _spheres_of(a, wfn, eps, q):
    b, omega = synth.cubic_cell(a)
    return (b, omega, synth.gsphere(b, q, wfn), synth.gsphere(b, (0.0, 0.0, 0.0), wfn), synth.gsphere(b, q, eps))


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _bands(g, nb, npw, real=False):
    c = torch.randn((nb, npw), generator=g, device="cuda", dtype=torch.float64 if real else torch.complex128)
    c /= torch.linalg.vector_norm(c, dim=1, keepdim=True)
    return c


def _energies(seed, nv, nc):
    r = np.random.default_rng(int(seed) + 77)
    return np.sort(r.uniform(-0.5, 0.0, nv)), np.sort(r.uniform(0.04, 1.5, nc))


def _elements(g, pairs, b, geps, npw, dtype, q=Q):
    """Matrix elements as the polarizability meets them: Gaussian, smaller at larger |q + G|."""
    k2 = torch.from_numpy((((geps + np.asarray(q)) @ b) ** 2).sum(1)).cuda()
    env = (1.0 / (1.0 + k2 / 2.0)) / math.sqrt(npw)
    m = torch.randn((pairs, len(geps)), generator=g, device="cuda", dtype=dtype)
    m *= env.to(m.real.dtype)
    return m


def _coulomb_cell(case, b, omega, q=Q):
    model = case.get("coulomb", "bulk")
    cut = {"bulk": 0.0, "sphere": case["a"] / 2, "slab": case["a"] / 2}[model]
    return bgw.make_cell(b, omega, q, case["n"], model, cut)


def _frequencies(case):
    return synth.gauss_legendre_frequencies(case["nfreq"]) if case.get("nfreq") else None


class _System:
    """The host arrays of one q-point (what ``Context.epsilon_batch`` reads)."""


def _inputs(case, seed):
    """Inputs of a case as tensors and arrays, without library objects (``exact`` takes the same)."""
    kind, g = case["kind"], _gen(seed)
    b, omega, gv, gc, geps = _spheres(case)
    s = dict(b=b, omega=omega, gv=gv, gc=gc, geps=geps)
    if kind in ("mtxel", "epsilon", "real_axis", "epsilon_real_flavor"):
        real = kind == "epsilon_real_flavor" or bool(case.get("real"))
        s.update(cv=_bands(g, case["nv"], len(gv), real), cc=_bands(g, case["nc"], len(gc), real))
    if kind == "chi":
        dt = torch.complex128 if case["prec"] == "fp64" else torch.complex64
        s["M"] = _elements(g, case["nv"] * case["nc"], b, geps, len(gc), dt)
        nf, ng = max(1, case["nfreq"]), len(geps)
        if case["accumulate"]:   # the sum of the chunks before this one
            x = _elements(g, min(ng, 256), b, geps, len(gc), torch.complex128)
            s["chi"] = (-(x.conj().T @ x) * (8.0 / omega)).expand(nf, ng, ng).contiguous()
    if kind in ("mtxel", "epsilon", "real_axis", "epsilon_real_flavor", "chi"):
        s["ev"], s["ec"] = _energies(seed, case["nv"], case["nc"])
    if kind == "inverse":
        s["mats"] = []
        for eps, q in ((case["eps"], Q), (case["eps2"], (0.25, 0.1, 0.0))):
            b, omega, _, gc, ge = _spheres(case, q, eps)
            x = _elements(g, 2 * len(ge), b, ge, len(gc), torch.complex128, q)
            # as strong as a sum over about sixty pairs for each plane wave, gaps around 1 Ha
            s["mats"].append((b, omega, q, ge, -(x.conj().T @ x) * (4.0 / omega * 30.0)))
    if kind == "batch":
        s["qs"] = []
        for j in range(case["nq"]):
            q = (0.05 * (j + 1), 0.0, 0.0)
            p = _System()
            p.bvec, p.omega, p.gv, p.gc, p.geps = _spheres(case, q)
            p.q_frac, p.fft = np.asarray(q), case["n"]
            p.ev, p.ec = _energies(seed + 1000 * j, case["nv"], case["nc"])
            s["qs"].append((p, _bands(g, case["nv"], len(p.gv)), _bands(g, case["nc"], len(p.gc))))
    if kind == "sigma":
        b, omega, gi, go, geps = _spheres(dict(case), tuple(-x for x in Q))
        s["geps"] = synth.gsphere(b, Q, case["eps"])
        s.update(go=go, gi=gi, co=_bands(g, case["no"], len(go)), ci=_bands(g, case["ni"], len(gi)))
        x = _elements(g, 64, b, s["geps"], len(go), torch.complex128)
        ng = len(s["geps"])
        # a Hermitian positive eps~^-1 <= I
        x = x / torch.linalg.vector_norm(x)
        s["epsinv"] = 0.7 * torch.eye(ng, device="cuda", dtype=torch.complex128) - 0.5 * (x.conj().T @ x)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    s["case"] = case
    s["prec"] = bgw.PREC[case.get("prec", "fp64")]
    s["ctx"] = bgw.Context(0)              # one handle per program
    s["stream"] = torch.cuda.Stream()      # a stream of its own, so that repeated calls may replay a graph
    s["omegas"] = _frequencies(case)
    s["cell"] = _coulomb_cell(case, s["b"], s["omega"])
    ng, dev = len(s["geps"]), "cuda"
    c16, c8 = torch.complex128, torch.complex64
    if kind == "mtxel":
        real = case["real"]
        dt = ({True: torch.float64, False: c16} if case["prec"] == "fp64" else {True: torch.float32, False: c8})[real]
        s["M"] = torch.empty((case["nv"] * case["nc"], ng), dtype=dt, device=dev)
        s["prec"] |= bgw.BGW_FLAVOR_REAL if real else 0
    elif kind == "chi":
        nf = max(1, case["nfreq"])
        s["start"] = s.get("chi")
        s["out"] = torch.empty((nf, ng, ng), dtype=c16, device=dev)
    elif kind == "inverse":
        s["cells"] = [_coulomb_cell(case, b, omega, q) for b, omega, q, _, _ in s["mats"]]
        s["lists"] = [m[3] for m in s["mats"]]
        s["chis"] = [m[4] for m in s["mats"]]
        s["invs"] = [torch.empty_like(x) for x in s["chis"]]
        s["ws"] = [torch.empty_like(x) for x in s["chis"]]
    elif kind in ("epsilon", "real_axis"):
        nf = max(1, case["nfreq"])
        if case.get("host"):
            s["cv"], s["cc"] = s["cv"].cpu().pin_memory(), s["cc"].cpu().pin_memory()
            s["inv"] = torch.empty((nf, ng, ng), dtype=c16).pin_memory()
        else:
            s["inv"] = torch.empty((nf, ng, ng), dtype=c16, device=dev)
        s["chunk"] = case.get("chunk") or (max(1, case["nc"] // 3) if case.get("host") else 0)
    elif kind == "epsilon_real_flavor":
        s["prec"] |= bgw.BGW_FLAVOR_REAL
        s["inv"] = torch.empty((1, ng, ng), dtype=torch.float64, device=dev)
    elif kind == "batch":
        s["invs"] = [torch.empty((case["nfreq"], len(p.geps), len(p.geps)), dtype=c16, device=dev)
                     for p, _, _ in s["qs"]]
    torch.cuda.synchronize()
    return s


# -------------------------------------------------------------------- run
def run(s):
    case, ctx, cell, prec = s["case"], s["ctx"], s["cell"], s["prec"]
    kind = case["kind"]
    with torch.cuda.stream(s["stream"]):
        if kind == "mtxel":
            ctx.mtxel(cell, s["gv"], s["cv"], s["gc"], s["cc"], s["geps"], prec, s["M"])
            return s["M"]
        if kind == "chi":
            if s["start"] is not None:
                s["out"].copy_(s["start"])
            ctx.chi_sum(cell, case["nv"], case["nc"], len(s["geps"]), s["M"], s["ev"], s["ec"], s["omegas"], prec,
                        case["accumulate"], s["out"])
            return s["out"]
        if kind == "inverse":
            ctx.epsinv(s["cells"], s["lists"], s["chis"], None, s["invs"])
            ctx.screened_w(s["cells"], s["lists"], s["invs"], s["ws"])
            return [s["invs"], s["ws"]]
        if kind == "epsilon":
            ctx.epsilon(cell, s["gv"], s["cv"], s["ev"], s["gc"], s["cc"], s["ec"], s["geps"], s["omegas"], prec,
                        s["chunk"], None, s["inv"])
            return s["inv"]
        if kind == "epsilon_real_flavor":
            ctx.epsilon(cell, s["gv"], s["cv"], s["ev"], s["gc"], s["cc"], s["ec"], s["geps"], None, prec, 0, None,
                        s["inv"])
            return s["inv"]
        if kind == "real_axis":
            ctx.epsilon_real(cell, s["gv"], s["cv"], s["ev"], s["gc"], s["cc"], s["ec"], s["geps"], s["omegas"],
                             case["delta"], False, prec, 0, None, s["inv"])
            return s["inv"]
        if kind == "batch":
            ctx.epsilon_batch([p for p, _, _ in s["qs"]], [v for _, v, _ in s["qs"]], [c for _, _, c in s["qs"]],
                              s["omegas"], prec, s["invs"])
            return s["invs"]
        return ctx.sigma_cohsex(cell, s["go"], s["co"], s["gi"], s["ci"], case["nocc"], s["geps"], s["epsinv"],
                                prec=prec)


# ------------------------------------------------------------------- work
def _mtxel_work(case, gv, gc, geps, pairs, nb):
    """Pruned transforms on the smallest grid that does not alias: 5 n log2 n flops per line over the lines that hold
    a kept value, 6 n^3 for each product, and three full passes for each band."""
    n = int((np.abs(gv).max(0) + np.abs(gc).max(0) + np.abs(geps).max(0)).max()) + 1
    gx, gy = int(np.abs(geps[:, 0]).max()), int(np.abs(geps[:, 1]).max())
    line = 5.0 * n * math.log2(n)
    return pairs * (line * (n * n + (2 * gx + 1) * n + (2 * gx + 1) * (2 * gy + 1)) + 6.0 * n ** 3) \
        + nb * 3.0 * n * n * line


def work(case):
    kind = case["kind"]
    b, omega, gv, gc, geps = _spheres(case)
    ng, nf = len(geps), max(1, case.get("nfreq") or 1)
    full = case.get("prec", "fp64") == "fp64"
    nv, nc = case.get("nv", 0), case.get("nc", 0)
    coef = 16.0 * (nv * len(gv) + nc * len(gc))
    if kind == "mtxel":
        r = 2 if case["real"] else 1
        return {"bytes": coef / r + nv * nc * ng * (16.0 if full else 8.0) / r,
                "flops": _mtxel_work(case, gv, gc, geps, nv * nc, nv + nc)}
    if kind == "chi":
        return {"bytes": nv * nc * ng * (16.0 if full else 8.0) + (32.0 if case["accumulate"] else 16.0) * nf * ng * ng,
                "flops": 4.0 * nf * ng * ng * nv * nc}
    if kind == "inverse":
        sizes = [ng, len(_spheres(case, (0.25, 0.1, 0.0), case["eps2"])[4])]
        return {"bytes": sum(48.0 * k * k for k in sizes), "flops": sum(4.0 * k ** 3 for k in sizes)}
    if kind in ("epsilon", "batch"):
        nq = case.get("nq", 1)
        return {"bytes": nq * (coef + 16.0 * nf * ng * ng),
                "flops": nq * (_mtxel_work(case, gv, gc, geps, nv * nc, nv + nc)
                               + nf * (4.0 * ng * ng * nv * nc + 4.0 * ng ** 3))}
    if kind == "real_axis":
        return {"bytes": coef + 16.0 * nf * ng * ng,
                "flops": _mtxel_work(case, gv, gc, geps, nv * nc, nv + nc)
                + nf * (8.0 * ng * ng * nv * nc + 8.0 * ng ** 3)}
    if kind == "epsilon_real_flavor":
        return {"bytes": coef / 2 + 8.0 * ng * ng,
                "flops": _mtxel_work(case, gv, gc, geps, nv * nc, nv + nc) + 2.0 * ng * ng * nv * nc + 1.0 * ng ** 3}
    no, ni = case["no"], case["ni"]
    return {"bytes": 16.0 * ng * ng + 16.0 * (no + ni) * len(gc),
            "flops": _mtxel_work(case, gv, gc, geps, no * ni, no + ni) + 8.0 * ng * ng * no * ni}


def tolerance(case):
    """About four times the largest error against exact() over the listed cases and thirty drawn ones: 1.3e-15 in FP64
    (an inverse), 2.4e-7 for FP32 matrix elements, 4.3e-6 for a mixed polarizability, 1.9e-7 for a mixed inverse
    (a scale the FP32 matrix elements and the tensor cores' FP32 sums set) and 2.9e-7 for a mixed Sigma with FP16
    splits (BF16 splits hold 16 bits of an operand, FP16 ones 22)."""
    if case.get("prec", "fp64") == "fp64":
        return {"rel": 5e-15}
    kind = case["kind"]
    if kind == "mtxel":
        return {"rel": 1e-6}
    if kind == "chi":
        return {"rel": 1.7e-5}
    if kind == "sigma":
        return {"rel": 3e-5 if case["prec"] == "mix_bf16" else 1.2e-6}
    return {"rel": 8e-7}


# ------------------------------------------------------------------ exact
def _grid(g, c, n):
    """u(r) = sum_G c(G) e^{+iG.r} on the n^3 grid."""
    idx = torch.from_numpy(((g % n).astype(np.int64) @ np.array([n * n, n, 1]))).cuda()
    u = torch.zeros((c.shape[0], n ** 3), dtype=torch.complex128, device="cuda")
    u[:, idx] = c.to("cuda", torch.complex128)
    return torch.fft.ifftn(u.view(-1, n, n, n), dim=(1, 2, 3), norm="forward")


def _mtxel(gv, cv, gc, cc, geps, n):
    """M[p][G] = (1/n^3) sum_r conj(u_v) u_c e^{+iG.r}, p = v nc + c."""
    idx = torch.from_numpy(((geps % n).astype(np.int64) @ np.array([n * n, n, 1]))).cuda()
    nv, nc = cv.shape[0], cc.shape[0]
    out = torch.empty((nv, nc, len(geps)), dtype=torch.complex128, device="cuda")
    uv = _grid(gv, cv, n)
    step = max(1, (1 << 26) // n ** 3)
    for c0 in range(0, nc, step):
        uc = _grid(gc, cc[c0:c0 + step], n)
        for v in range(nv):
            f = torch.fft.ifftn(uv[v].conj() * uc, dim=(1, 2, 3))
            out[v, c0:c0 + step] = f.reshape(uc.shape[0], -1)[:, idx]
    return out.view(nv * nc, len(geps))


def _weights(ev, ec, w=None, delta=None):
    d = torch.from_numpy(np.subtract.outer(ev, ec).ravel()).cuda()
    if w is None:
        return 1.0 / d
    if delta is None:
        return d / (d * d + w * w)
    return 0.5 * (1.0 / torch.complex(d - w, torch.full_like(d, -delta))
                  + 1.0 / torch.complex(d + w, torch.full_like(d, delta)))


def _chi(m, w, omega):
    m = m.to(torch.complex128)
    return (m.conj().T @ (m * w.to(torch.complex128)[:, None])) * (4.0 / omega)


def _v(cell_case, b, geps, q=Q):
    k = torch.from_numpy((geps + np.asarray(q)) @ b).cuda()
    k2 = (k * k).sum(1)
    model, cut = cell_case.get("coulomb", "bulk"), cell_case["a"] / 2
    if model == "sphere":
        x = torch.where(k2 == 0, 2 * math.pi * cut * cut * torch.ones_like(k2),
                        8 * math.pi / k2 * torch.sin(0.5 * cut * k2.sqrt()) ** 2)
        return x
    if model == "slab":
        kxy = (k[:, 0] ** 2 + k[:, 1] ** 2).sqrt()
        s = torch.sin(0.5 * k[:, 2] * cut)
        return 4 * math.pi / k2 * (-torch.expm1(-kxy * cut) + torch.exp(-kxy * cut) * 2 * s * s)
    return 4 * math.pi / k2


def _inverse(chi, v):
    sv = v.sqrt().to(torch.complex128)
    return torch.linalg.inv(torch.eye(len(v), device="cuda", dtype=torch.complex128) - sv[:, None] * chi * sv[None, :])


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    # matrix elements of the whole large cell alone take longer than is sensible
    if kind == "epsilon" and case["nv"] * case["nc"] * n ** 3 > 4e10:
        return None
    s = _inputs(case, seed)
    b, omega, geps = s["b"], s["omega"], s["geps"]
    freqs = _frequencies(case)
    if kind == "mtxel":
        m = _mtxel(s["gv"], s["cv"], s["gc"], s["cc"], geps, n)
        return m.real.contiguous() if case["real"] else m
    if kind == "chi":
        out = torch.stack([_chi(s["M"], _weights(s["ev"], s["ec"], w), omega)
                           for w in ([None] if freqs is None else freqs)])
        return out + s["chi"] if case["accumulate"] else out
    if kind == "inverse":
        invs, ws = [], []
        for b, omega, q, ge, x in s["mats"]:
            v = _v(case, b, ge, q)
            invs.append(_inverse(x, v))
            sv = v.sqrt().to(torch.complex128)
            ws.append(sv[:, None] * invs[-1] * sv[None, :])
        return [invs, ws]
    if kind in ("epsilon", "real_axis", "epsilon_real_flavor"):
        m = _mtxel(s["gv"], s["cv"], s["gc"], s["cc"], geps, n)
        v, outs = _v(case, b, geps), []
        for w in ([None] if freqs is None else freqs):
            wt = _weights(s["ev"], s["ec"], w, case["delta"] if kind == "real_axis" else None)
            outs.append(_inverse(_chi(m, wt, omega), v))
        out = torch.stack(outs)
        return out.real.contiguous() if kind == "epsilon_real_flavor" else out
    if kind == "batch":
        outs = []
        for p, cv, cc in s["qs"]:
            m = _mtxel(p.gv, cv, p.gc, cc, p.geps, n)
            v = _v(case, p.bvec, p.geps, tuple(p.q_frac))
            outs.append(torch.stack([_inverse(_chi(m, _weights(p.ev, p.ec, w), p.omega), v) for w in freqs]))
        return outs
    # Sigma: m_p(G) = sum_G2 conj(c_i(G2 - G)) c_o(G2), p = inner no + outer
    no, ni, nocc = case["no"], case["ni"], case["nocc"]
    m = _mtxel(s["gi"], s["ci"], s["go"], s["co"], -geps, n).view(ni, no, -1)
    v = _v(case, b, geps)
    sv = v.sqrt().to(torch.complex128)
    w = sv[:, None] * s["epsinv"] * sv[None, :]
    qw = (m.conj() * (m @ w.T)).sum(2).real
    qv = (m.abs() ** 2 * v).sum(2)
    d = (geps[:, None, :] - geps[None, :, :]).reshape(-1, 3)
    nr = 4 * int(np.abs(s["go"]).max()) + 2 * int(np.abs(d).max()) + 2
    idx = torch.from_numpy((d % nr).astype(np.int64) @ np.array([nr * nr, nr, 1])).cuda()
    wv = (w - torch.diag(v).to(torch.complex128)).reshape(-1)
    che = []
    for k in range(no):
        u = _grid(s["go"], s["co"][k:k + 1], nr)[0]
        rho = torch.fft.ifftn((u.conj() * u), dim=(0, 1, 2)).reshape(-1)
        che.append((rho[idx] * wv).sum().real / (2 * omega))
    return torch.stack([-qv[:nocc].sum(0) / omega, -qw[:nocc].sum(0) / omega,
                        0.5 * (qw - qv).sum(0) / omega, torch.stack(che)])
