"""One-launch solves with up to 64 items a block, where FP64 gives each spin component a lane, and past that; with
two-step transforms of 6 to 10 points in FP64; and with more blocks than (slice, band) planes: blocks without a plane,
planes that outnumber the blocks by a few, a plane per block. The solver stops at a true relative residual of 1e-10,
computed in complex128; the residual formed here with the FP64 normal operator differs from it by rounding, under
1e-12."""

import pytest
import torch

from paper_2204_14241_gb300 import presets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", [False, True])
@pytest.mark.parametrize("solver", ["mixed", "fp64"])
@pytest.mark.parametrize("L,Nt,k", [(2, 3, 2), (6, 9, 2), (8, 8, 1), (16, 16, 1), (10, 6, 3), (20, 5, 1), (20, 24, 1),
                                    (20, 40, 1), (20, 40, 4), (40, 80, 1), (24, 48, 2)])
def test_teams(L, Nt, k, solver, precond):
    from paper_2204_14241_gb300.hmc import Context
    ctx = Context(L, Nt, nrhs_max=k, solver=solver, **presets.baseline())
    g = torch.Generator(device="cuda")
    g.manual_seed(L + Nt + k)
    phi = torch.randn((3, Nt, L, L), generator=g, device="cuda", dtype=torch.float64) * 0.5
    phi[2] += 1.2
    b = torch.view_as_complex(torch.randn((k, Nt, L, L, 2, 2, 2), generator=g, device="cuda", dtype=torch.float64))
    x, st = ctx.cg_solve(phi, b, tol=1e-10, precond=precond)
    assert st["converged"]
    r = (b - ctx.apply_MdagM(phi, x)).flatten(1).norm(dim=1) / b.flatten(1).norm(dim=1)
    assert r.max().item() < 1.01e-10
