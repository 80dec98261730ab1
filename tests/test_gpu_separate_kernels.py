"""Solves with a launch per step (csrc/cg.cu), which take over where the one-launch solver does not go: plain
complex64 CG on strip lattices past 1.25 million sites in all (the fused update without a stored residual, x on every
other iteration), any solve past 2^23 sites (the update folded into the operator), and the preconditioner on slice
counts without a two-factor split. Each case checks by the launch count that it took that way.

The solver stops at a true relative residual that it computes in FP64; formed here with the FP64 normal operator it
differs by rounding, under 1e-12 of |b|."""

import pytest
import torch

from paper_2204_14241_gb300 import presets

pytestmark = pytest.mark.gpu


def context(L, Nt, K, solver="mixed", **kw):
    from paper_2204_14241_gb300.hmc import Context
    return Context(L, Nt, nrhs_max=K, solver=solver, **{**presets.baseline(), **kw})


def field(L, Nt, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    phi = 0.5 * torch.randn((3, Nt, L, L), generator=g, device="cuda", dtype=torch.float64)
    phi[2] += 1.2
    return phi


def noise(L, Nt, K, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.view_as_complex(torch.randn((K, Nt, L, L, 2, 2, 2), generator=g, device="cuda", dtype=torch.float64))


def residuals(ctx, phi, x, b):
    """||b - A x|| / ||b|| of each right-hand side, eight at a time."""
    out = []
    for k in range(0, b.shape[0], 8):
        r = b[k:k + 8] - ctx.apply_MdagM(phi, x[k:k + 8].contiguous())
        out.append(r.flatten(1).norm(dim=1) / b[k:k + 8].flatten(1).norm(dim=1))
    return torch.cat(out)


def solve(ctx, phi, b, **kw):
    before = ctx.launches()
    x, st = ctx.cg_solve(phi, b, **kw)
    assert ctx.launches() - before > 3 * st["iterations"]
    return x, st


@pytest.fixture(scope="module")
def strip():   # 1.31 million sites of a strip lattice
    L, Nt, K = 16, 160, 32
    ctx, phi, b = context(L, Nt, K), field(L, Nt, 1), noise(L, Nt, K, 2)
    for k in range(1, K, 3):   # weight on the upper modes: these stop earlier
        for _ in range(k % 4 + 1):
            b[k:k + 1] = ctx.apply_MdagM(phi, b[k:k + 1].contiguous())
    yield ctx, phi, b
    ctx.close()


def test_strip_cg(strip):
    ctx, phi, b = strip
    c = b.clone()
    c[5] = 0
    x, st = solve(ctx, phi, c, tol=1e-10, precond=False)
    assert st["converged"] and st["reliable_updates"] >= 2 and not torch.any(x[5]).item()
    live = [k for k in range(c.shape[0]) if k != 5]
    assert residuals(ctx, phi, x[live], c[live]).max().item() < 1.01e-10
    y, again = solve(ctx, phi, c, tol=1e-10, precond=False)
    assert torch.equal(x, y) and st == again


@pytest.mark.parametrize("maxit", [1, 2, 7, 8, 9, 30])   # around the deferred half of x and the host's checks
def test_strip_cg_out_of_iterations(strip, maxit):
    from paper_2204_14241_gb300.hmc import HMC_ERR_NOCONV
    ctx, phi, b = strip
    x, st = solve(ctx, phi, b, tol=1e-10, precond=False, maxit=maxit, raise_on_noconv=False)
    assert st["status"] == HMC_ERR_NOCONV and st["iterations"] == maxit and not st["converged"]
    assert abs(residuals(ctx, phi, x, b).max().item() - st["true_rel_resid"]) < 1e-12


def test_strip_force(strip):
    # S_PF is off by the square of the residual times the condition number, under 1e-12 of it; so the one-launch solver
    # gives the same sum in four parts, and the force, which is linear in the error, to 1e-6 at 1e-10
    ctx, phi, b = strip
    F, spf, _, _ = ctx.force(phi, b, include_boson=False, precond=False)
    parts = [ctx.force(phi, b[k:k + 8].contiguous(), include_boson=False, precond=False) for k in range(0, 32, 8)]
    assert abs(spf - sum(p[1] for p in parts)) < 1e-11 * spf
    G = sum(p[0] for p in parts)
    assert (F - G).norm().item() < 1e-6 * G.norm().item()


def test_strip_trajectory():
    # starts from extrapolated solutions, against FP64; bounds as in the other trajectory tests at 1e-12
    L, Nt, K = 16, 160, 32
    chi, z, phi0 = noise(L, Nt, K, 3) * 0.5 ** 0.5, field(L, Nt, 4), field(L, Nt, 5)
    out = {}
    for solver in ("mixed", "fp64"):
        ctx, phi = context(L, Nt, K, solver, cg_tol=1e-12, initial_guess=2), phi0.clone()
        out[solver] = ctx.trajectory([phi], [torch.ones_like(phi)], 0.01, 4, nrhs=K, precond=False, chi=[chi], z=[z],
                                     u=[0.5]), phi
        ctx.close()
    (m, pm), (f, pf) = out["mixed"], out["fp64"]
    assert m["status"] == 0 and m["max_true_resid"][0] <= 1e-12
    assert abs(m["dH"][0] - f["dH"][0]) < 1e-12 * 4 * L * L * Nt * K and m["accepted"] == f["accepted"]
    assert (pm - pf).norm() < 1e-9 * pf.norm()


@pytest.mark.parametrize("solver", ["mixed", "fp64"])
def test_past_2_23_sites(solver):
    L, Nt, K = 18, 448, 58
    ctx, phi, b = context(L, Nt, K, solver), field(L, Nt, 6), noise(L, Nt, K, 7)
    x, st = solve(ctx, phi, b, tol=1e-8, precond=False)
    assert st["converged"] and residuals(ctx, phi, x, b).max().item() < 1.01e-8
    ctx.close()


@pytest.mark.parametrize("solver", ["mixed", "fp64"])
@pytest.mark.parametrize("L,Nt,K", [(6, 125, 2), (16, 125, 3), (20, 147, 1)])
def test_preconditioner_without_a_split(L, Nt, K, solver):
    ctx, phi, b = context(L, Nt, K, solver), field(L, Nt, 8), noise(L, Nt, K, 9)
    x, st = solve(ctx, phi, b, tol=1e-10, precond=True)
    assert st["converged"] and residuals(ctx, phi, x, b).max().item() < 1.01e-10
    x, st = solve(ctx, phi, b, tol=1e-10, precond=True, maxit=5, raise_on_noconv=False)
    assert not st["converged"] and abs(residuals(ctx, phi, x, b).max().item() - st["true_rel_resid"]) < 1e-12
