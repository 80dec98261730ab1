"""A trajectory of step size zero proposes its own start: phi += 0 * velocity leaves every bit of the field, the
energies at both ends are those of one field and momentum, and the proposal is accepted. On each route of the
drift: planes, tiles of lines, complex transforms (L = 2), and all chains of a batch, with and without a graph.

Bounds: S_PF at the start is the noise's norm, at the end it comes from a solve to 1e-12, |dH| < 1e-8 as in
test_gpu_parity, for norms up to 1e5; 1e-12 of the norm past that."""

import pytest
import torch

from paper_2204_14241_gb300 import presets

pytestmark = pytest.mark.gpu


def field(L, Nt, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return 0.3 * torch.randn((3, Nt, L, L), generator=g, device="cuda", dtype=torch.float64)


@pytest.mark.parametrize("L,Nt,n_leap", [(18, 35, 2), (64, 128, 1), (2, 6, 1)])
def test_single_chain(L, Nt, n_leap):
    from paper_2204_14241_gb300.hmc import Context
    ctx = Context(L, Nt, solver="mixed", cg_tol=1e-12, **presets.baseline())
    phi = field(L, Nt, 1)
    start = phi.clone()
    out = ctx.trajectory([phi], [torch.full_like(phi, 0.7)], 0.0, n_leap, precond=False, seed=3, counter=0)
    assert torch.equal(phi, start)
    assert out["accepted"] == [True] and out["jump2"][0] == 0.0
    assert abs(out["dH"][0]) < max(1e-8, 1e-12 * 4 * L * L * Nt)


@pytest.mark.parametrize("graph", [False, True])
def test_batch(graph):
    from paper_2204_14241_gb300.hmc import Context
    chains = [(12, 24, 0.3), (18, 10, 0.4), (16, 32, 0.5)]
    L, Nt, r = chains[0]
    ctx = Context(L, Nt, solver="mixed", nrhs_max=2, cg_tol=1e-12, chains=chains, batch_chains=1, batch_graph=graph,
                  initial_guess=1, **{**presets.baseline(), "r": r})
    phis = [field(a, b, i) for i, (a, b, _) in enumerate(chains)]
    starts = [p.clone() for p in phis]
    for counter in range(2):
        out = ctx.trajectory(phis, [torch.full_like(p, 0.7) for p in phis], 0.0, 2, nrhs=2, seed=4, counter=counter)
        assert all(torch.equal(p, s) for p, s in zip(phis, starts))
        assert all(out["accepted"]) and max(abs(v) for v in out["dH"]) < 1e-8
