"""Mixed-precision solves of right-hand sides far from unit size: 2^-40 (1e-12) and 2^66 (7e19), whose squares
leave FP32's range on the way to the tolerance or at once. Multiplying b by a power of two changes no mantissa
anywhere in the solve, so x comes out multiplied by it bit for bit, in the same number of iterations. Every form of
the one-launch solver: one block, clusters, cooperative teams, with and without the preconditioner, batches."""

import numpy as np
import pytest
import torch

from paper_2204_14241_gb300 import inputs as I, presets

pytestmark = pytest.mark.gpu
KW = presets.baseline()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("power", [-40, 66])
@pytest.mark.parametrize("precond", [False, True])
@pytest.mark.parametrize("L,Nt,nrhs", [(4, 4, 1), (4, 35, 2), (12, 20, 1), (18, 35, 3)])
def test_solve(L, Nt, nrhs, precond, power):
    from paper_2204_14241_gb300.hmc import Context
    ctx = Context(L, Nt, solver="mixed", nrhs_max=nrhs, cg_tol=1e-11, **KW)
    phi, b = dev(I.gaussian_field(1, L, Nt)), dev(I.fermion_noise(2, nrhs, L, Nt))
    x, st = ctx.cg_solve(phi, b, precond=precond)
    y, sy = ctx.cg_solve(phi, b * 2.0 ** power, precond=precond)
    assert sy == st and st["converged"]
    assert torch.equal(y, x * 2.0 ** power)


@pytest.mark.parametrize("power", [-40, 66])
@pytest.mark.parametrize("n", [3, 200])   # teams of several blocks; pairs taken from the queue
def test_batch(n, power):
    from paper_2204_14241_gb300.hmc import Context
    chains = [(8, 10, 0.3) if i % 2 else (4, 6, 0.4) for i in range(n)]
    ctx = Context(8, 10, solver="mixed", nrhs_max=4, cg_tol=1e-11, chains=chains, batch_chains=1,
                  **{**KW, "r": 0.3})
    phis = [dev(0.5 * I.gaussian_field(10 + i, L, Nt)) for i, (L, Nt, _) in enumerate(chains)]
    sigs = [torch.ones_like(p) for p in phis]
    z = [dev(I.gaussian_field(300 + i, L, Nt)) for i, (L, Nt, _) in enumerate(chains)]
    chi = [dev(I.fermion_noise(600 + i, 4, L, Nt)) for i, (L, Nt, _) in enumerate(chains)]

    def run(f):   # no leapfrog step: one solve, whose action 2 Re<varphi, X> - |D^dagger X|^2 is the last energy
        return ctx.trajectory([p.clone() for p in phis], sigs, 0.1, 0, nrhs=4, chi=[c * f for c in chi], z=z,
                              u=[0.5] * n)

    one, far = run(1.0), run(2.0 ** power)
    assert far["cg_iterations"] == one["cg_iterations"] and far["max_true_resid"] == one["max_true_resid"]
    assert all(a[5] == b[5] * 4.0 ** power for a, b in zip(far["energies"], one["energies"]))
