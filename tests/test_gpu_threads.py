"""Contexts of several host threads at once, with problems of different sizes: a kernel's shared-memory limit belongs to
the process, so no thread may lower it under another's launch."""
import threading

import numpy as np
import pytest

import oracle
from paper_1111_4429_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
Q = (0.1, 0.0, 0.0)


def _run(jobs, loops):
    errors = []

    def work(job):
        st = torch.cuda.Stream()
        try:
            with torch.cuda.stream(st):
                for _ in range(loops):
                    job(st)
        except Exception as e:   # noqa: BLE001  (reported below)
            errors.append(repr(e))
    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]


def test_general_inverses_of_different_sizes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4429_gb300 import bgw
    bvec, _ = synth.cubic_cell(30.0)
    allg = synth.gsphere(bvec, Q, 12.0)
    jobs, checks = [], []
    for n in (20, 33, 70, 900):
        rng = np.random.default_rng(n)
        g = allg[:n]
        sv = np.sqrt(oracle.coulomb(bvec, Q, g))
        x = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))) / np.sqrt(n)
        e = 2 * np.eye(n) + 0.3 * x
        chi = torch.from_numpy((np.eye(n) - e) / np.outer(sv, sv)).cuda()
        inv = torch.zeros_like(chi)
        ctx, cell = bgw.Context(0), bgw.make_cell(bvec, 27000.0, Q, 64)
        torch.cuda.synchronize()

        def job(st, ctx=ctx, cell=cell, g=g, chi=chi, inv=inv):
            ctx.epsinv_general([cell], [g], [chi], None, [inv])
            ctx.sync(st)
        jobs.append(job)
        checks.append((e, inv))
    _run(jobs, 60)
    for e, inv in checks:
        ref = np.linalg.inv(e)
        assert np.linalg.norm(inv.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)


def test_pair_transforms_of_different_widths():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4429_gb300 import bgw
    jobs, checks = [], []
    for k, r in enumerate((11, 9, 11, 7)):   # kept rows on 48^3: 23, 19, 23, 15, so 48 to 60 KB of shared memory
        rng = np.random.default_rng(k)
        gv = np.unique(np.concatenate([rng.integers(-15, 16, (200, 3)), [[15, -15, 15], [-15, 15, 0]]]), axis=0)
        ge = np.unique(np.concatenate([rng.integers(-r, r + 1, (300, 3)), [[r, -r, r], [-r, r, 0]]]), axis=0)
        gv, ge = gv.astype(np.int32), ge.astype(np.int32)
        cv = rng.standard_normal((8, len(gv))) + 1j * rng.standard_normal((8, len(gv)))
        cc = rng.standard_normal((100, len(gv))) + 1j * rng.standard_normal((100, len(gv)))
        dv, dc = torch.from_numpy(cv).cuda(), torch.from_numpy(cc).cuda()
        M = torch.zeros((800, len(ge)), dtype=torch.complex64, device="cuda")
        ctx, cell = bgw.Context(0), bgw.make_cell(np.eye(3) * 0.3, 8641.0, Q, 48)
        ctx.set_option(bgw.BGW_OPT_PAIR_KERNEL, 1)
        torch.cuda.synchronize()

        def job(st, ctx=ctx, cell=cell, gv=gv, ge=ge, dv=dv, dc=dc, M=M):
            ctx.mtxel(cell, gv, dv, gv, dc, ge, bgw.BGW_PREC_MIX_FP16, M)
            ctx.sync(st)
        jobs.append(job)
        checks.append((oracle.mtxel_direct(gv, cv[:1], gv, cc[:2], ge), M))
    _run(jobs, 150)
    for ref, M in checks:
        got = M.cpu().numpy()[:2].reshape(ref.shape)
        assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
