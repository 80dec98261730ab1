"""The one-launch solver (csrc/team.cu) at the edges of its rules: one block per right-hand side, clusters of
2 to 16 blocks, cooperative teams, several pairs per block; extents and slice counts with one- and
two-factor FFT splits; right-hand sides that are zero, not finite, or out of iterations.

Solutions are checked by the FP64 true residual that the oracle's matrix-free operators give, 1.5 times the
solver's tolerance as in test_gpu_parity (the two evaluations of the residual differ by rounding, some 1e-14
of |b|)."""

import numpy as np
import pytest
import torch

from oracle import fermion
from oracle.model import Params
from paper_2204_14241_gb300 import inputs as I, presets

pytestmark = pytest.mark.gpu
KW = presets.baseline()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def context(L, Nt, **kw):
    from paper_2204_14241_gb300.hmc import Context
    return Context(L, Nt, **{**KW, **kw})


def residual(L, Nt, phi, x, b):
    P = Params(L=L, Nt=Nt, **KW)
    po, xo, bo = I.to_paper_boson(phi), I.to_paper_fermion(x), I.to_paper_fermion(b)
    return np.linalg.norm(bo - fermion.apply_A(P, po, xo)) / np.linalg.norm(bo)


# (L, Nt): 2 V items. 128, 448: one block; 1120, 5488, 12096: clusters of 2 or 4, 8, 16; 22680, 51200: cooperative
# teams; Nt = 7, 35, 49 and L = 14, 18: odd factors; L = 10, Nt = 2: single-step splits
@pytest.mark.parametrize("solver", ["mixed", "fp64"])
@pytest.mark.parametrize("precond", [False, True])
@pytest.mark.parametrize("L,Nt,nrhs", [(4, 4, 1), (4, 14, 3), (4, 35, 2), (14, 14, 1), (12, 42, 2), (18, 35, 3),
                                       (10, 2, 9), (2, 49, 1), (32, 25, 1)])
def test_solve(L, Nt, nrhs, solver, precond):
    tol = 1e-11
    ctx = context(L, Nt, solver=solver, nrhs_max=nrhs, cg_tol=tol)
    phi, b = I.gaussian_field(1, L, Nt), I.fermion_noise(2, nrhs, L, Nt)
    x, st = ctx.cg_solve(dev(phi), dev(b), precond=precond)
    x = x.cpu().numpy()
    assert st["converged"] and st["true_rel_resid"] <= tol and st["reliable_updates"] >= 1
    for k in range(nrhs):
        assert residual(L, Nt, phi, x[k], b[k]) <= 1.5 * tol
    again, st2 = ctx.cg_solve(dev(phi), dev(b), precond=precond)
    assert np.array_equal(again.cpu().numpy(), x) and st2 == st   # fixed order of all sums


@pytest.mark.parametrize("solver", ["mixed", "fp64"])
@pytest.mark.parametrize("precond", [False, True])
def test_zero_nonfinite_and_maxit(solver, precond):
    from paper_2204_14241_gb300.hmc import HMC_ERR_NOCONV, HMC_ERR_NONFINITE, HmcError
    L, Nt = 6, 10
    ctx = context(L, Nt, solver=solver, nrhs_max=2, cg_tol=1e-10)
    phi, b = I.gaussian_field(3, L, Nt), I.fermion_noise(4, 2, L, Nt)
    b[0] = 0
    x, st = ctx.cg_solve(dev(phi), dev(b), precond=precond)
    assert st["converged"] and not torch.any(x[0]).item()
    assert residual(L, Nt, phi, x[1].cpu().numpy(), b[1]) <= 1.5e-10
    x, st = ctx.cg_solve(dev(phi), dev(b), precond=precond, maxit=5, raise_on_noconv=False)
    assert st["status"] == HMC_ERR_NOCONV and st["iterations"] == 5 and not st["converged"]
    assert abs(residual(L, Nt, phi, x[1].cpu().numpy(), b[1]) - st["true_rel_resid"]) < 1e-12
    b[1].flat[7] = np.nan
    with pytest.raises(HmcError) as e:
        ctx.cg_solve(dev(phi), dev(b), precond=precond)
    assert e.value.code == HMC_ERR_NONFINITE


def test_tolerance_at_the_rounding_floor():
    # 1e-14 is a few times the floor of the FP64 true residual here: each mode still gets there
    L, Nt = 12, 20
    phi, b = I.gaussian_field(5, L, Nt), I.fermion_noise(6, 1, L, Nt)
    for solver in ("mixed", "fp64"):
        for precond in (False, True):
            _, st = context(L, Nt, solver=solver, cg_tol=1e-14).cg_solve(dev(phi), dev(b), precond=precond)
            assert st["converged"] and st["iterations"] < 2000


def test_batch_with_more_pairs_than_blocks():
    # 200 chains x 4 right-hand sides of 4 x 4 x 4: blocks solve several pairs in turn; each chain against the
    # serial path on the same noise (the bounds of the 64-chain test in test_gpu_parity)
    n, L, Nt = 200, 4, 4
    chains = [(L, Nt, 0.3 + 0.002 * i) for i in range(n)]
    kw = dict(solver="mixed", nrhs_max=4, cg_tol=1e-12, chains=chains)
    phis = [dev(I.gaussian_field(100 + i, L, Nt) * 0.5) for i in range(n)]
    phis_s = [p.clone() for p in phis]
    sigs = [torch.ones_like(p) for p in phis]
    a = context(L, Nt, batch_chains=1, **kw).trajectory(phis, sigs, 0.02, 1, nrhs=4, seed=5, counter=1)
    s = context(L, Nt, **kw).trajectory(phis_s, sigs, 0.02, 1, nrhs=4, precond=False, seed=5, counter=1)
    assert a["status"] == 0 and max(a["max_true_resid"]) <= 1e-12
    assert a["accepted"] == s["accepted"]
    assert np.max(np.abs(np.array(a["dH"]) - np.array(s["dH"]))) < 1e-8
    assert all(torch.linalg.norm(p - q) < 1e-9 * torch.linalg.norm(q) for p, q in zip(phis, phis_s))
