"""The operators' routes: complex64 with vectors 32- and 16-byte aligned (whole-site and half-site accesses, and
the strip kernel only in the first case), the two-pass normal operator with its norms. Against the oracle at
test_gpu_parity's operator bounds, 1e-12 (FP64) and 1e-5 (FP32)."""

import numpy as np
import pytest
import torch

from oracle import fermion
from oracle.model import Params
from paper_2204_14241_gb300 import inputs as I, presets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 2])   # complex64 entries: 16 bytes
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("L,Nt,k", [(2, 3, 1), (6, 5, 2), (16, 5, 2), (18, 15, 1), (36, 70, 3)])
def test_alignment_and_routes(L, Nt, k, dtype, shift):
    from paper_2204_14241_gb300.hmc import Context
    tol, rdt = (1e-5, torch.float32) if dtype == torch.complex64 else (1e-12, torch.float64)
    ctx = Context(L, Nt, nrhs_max=k, **presets.baseline())
    P = Params(L=L, Nt=Nt, **presets.baseline())
    phi, x = I.gaussian_field(1, L, Nt), I.fermion_noise(2, k, L, Nt)
    n = x.size

    def shifted(a):
        buf = torch.zeros(n + shift, dtype=dtype, device="cuda")
        v = buf[shift:].view(a.shape)
        v.copy_(torch.from_numpy(a))
        return v

    xd, pd = shifted(x), torch.from_numpy(phi).cuda().to(rdt)
    xo = [I.to_paper_fermion(v) for v in xd.cpu().numpy().astype(np.complex128)]
    po = I.to_paper_boson(pd.double().cpu().numpy())
    out = shifted(np.zeros_like(x))
    got = lambda: [I.to_paper_fermion(v) for v in out.cpu().numpy().astype(np.complex128)]
    err = lambda ref: max(np.linalg.norm(a - b) / np.linalg.norm(b) for a, b in zip(got(), ref))
    ctx.apply_M(pd, xd, out=out)
    assert err([fermion.apply_D(P, po, v) for v in xo]) < tol
    ctx.apply_M(pd, xd, dagger=True, out=out)
    t = [fermion.apply_Ddag(P, po, v) for v in xo]
    assert err(t) < tol
    _, norms = ctx.apply_MdagM(pd, xd, norms=True, out=out)
    assert err([fermion.apply_A(P, po, v) for v in xo]) < tol
    assert all(abs(a - np.vdot(b, b).real) < tol * a for a, b in zip(norms, t))
