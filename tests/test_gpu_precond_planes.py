"""The preconditioner and the twisted Fourier transforms by planes (complex128; complex64 lattices without compiled passes) against the oracle: extents
of one and two transform factors, odd numbers of slices, tau tiles with a ragged end, blocks of several planes with
a short last one, and the fallbacks (x == y is the same route; 125 slices have no split and take the axis kernels).
Bounds: test_gpu_parity's operator bounds, 1e-12 (FP64) and 1e-5 (FP32)."""

import numpy as np
import pytest
import torch

from oracle import solver
from oracle.model import Params
from paper_2204_14241_gb300 import inputs as I, presets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("L,Nt,k", [(2, 2, 1), (2, 3, 3), (4, 6, 1), (6, 5, 2), (10, 9, 1), (14, 7, 3), (18, 15, 2),
                                    (20, 40, 1), (6, 125, 1), (30, 12, 1), (36, 21, 1)])
def test_planes(L, Nt, k, dtype):
    from paper_2204_14241_gb300.hmc import Context
    tol = 1e-5 if dtype == torch.complex64 else 1e-12
    ctx = Context(L, Nt, nrhs_max=k, **presets.baseline())
    P = Params(L=L, Nt=Nt, **presets.baseline())
    x = torch.from_numpy(I.fermion_noise(7, k, L, Nt)).cuda().to(dtype)
    y = torch.full_like(x, float("nan"))
    ctx.apply_precond(x, out=y)
    paper = lambda a: [I.to_paper_fermion(v) for v in a.cpu().numpy().astype(np.complex128)]
    for a, b in zip(paper(y), paper(x)):
        r = solver.apply_precond(P, b)
        assert np.linalg.norm(a - r) < tol * np.linalg.norm(r)
    ctx.apply_precond(x, out=x)
    assert torch.equal(x, y)


@pytest.mark.parametrize("L,Nt,k", [(2, 3, 1), (4, 6, 3), (6, 5, 2), (14, 15, 1), (10, 49, 1), (18, 8, 2)])
def test_twisted_transforms(L, Nt, k):
    """green_estimate at g = 0, r-independent: D is diagonal under F~, so the estimate with Rademacher probes is exactly
    1 / K-hat per Fourier mode up to the solver's tolerance (1e-12 here; the smallest |K-hat|^2 in play is above 1e-3)."""
    from paper_2204_14241_gb300.hmc import Context
    kw = dict(presets.baseline())
    kw["g"] = 0.0
    ctx = Context(L, Nt, nrhs_max=k, cg_tol=1e-12, **kw)
    g = torch.Generator().manual_seed(5)
    v = (torch.randint(0, 2, (k, Nt, L, L, 2, 2), generator=g) * 2 - 1).to(torch.complex128).cuda()
    phi = torch.zeros((3, Nt, L, L), dtype=torch.float64, device="cuda")
    out = ctx.green_estimate(phi, v, precond=True)[0].cpu().numpy().reshape(Nt, L, L, 2, 2)
    w = (2 * np.arange(Nt) + 1) * np.pi / Nt
    c = np.cos(2 * np.pi * np.arange(L) / L)
    dt, mu, th, tv = (kw[n] for n in ("dtau", "mu", "t_h", "t_v"))
    for a in range(2):
        eps = mu[a] + 2 * th[a] * c[None, None, :] + 2 * tv[a] * c[None, :, None]
        K = np.exp(1j * w)[:, None, None] - 1 - dt * eps
        assert np.abs(K).min() > 0.03
        for s in range(2):
            assert np.abs(out[..., a, s] - 1 / K).max() < 1e-8 * np.abs(1 / K).max()
