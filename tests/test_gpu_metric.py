"""Metric operations on the real transforms (csrc/metric.cu) at the edges of their lattices: the smallest
extents, one- and two-factor splits, a column count that leaves a partial tau tile, a plane that takes one
block of an SM, and extents that keep the complex transforms. Against numpy's FFTs; bound 1e-12, as
test_gpu_parity has it for these operations, and sigma-hat both even and not even in the wave vector (the real
part of the complex transform is the result either way)."""

import numpy as np
import pytest
import torch

from paper_2204_14241_gb300 import inputs as I, presets

pytestmark = pytest.mark.gpu
AX = (1, 2, 3)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("even", [True, False])
@pytest.mark.parametrize("L,Nt", [(2, 6), (4, 2), (4, 160), (6, 35), (10, 9), (14, 49), (16, 16), (18, 27), (30, 4),
                                  (36, 20), (98, 4), (112, 2), (120, 3)])
def test_operations(L, Nt, even):
    from paper_2204_14241_gb300 import hmc
    ctx = hmc.Context(L, Nt, **presets.baseline())
    x, w = I.gaussian_field(1, L, Nt), I.gaussian_field(2, L, Nt)
    sig = np.abs(np.fft.fftn(w, axes=AX, norm="ortho")) ** 2 + 0.3 if even else np.abs(w) + 0.3
    f = np.fft.fftn(x, axes=AX, norm="ortho")
    back = lambda v: np.fft.ifftn(v, axes=AX, norm="ortho").real
    d, s = dev(x), dev(sig)
    assert rel(ctx.metric(hmc.METRIC_VELOCITY, s, d).cpu().numpy(), back(sig * f)) < 1e-12
    assert rel(ctx.metric(hmc.METRIC_MOMENTUM, s, d).cpu().numpy(), back(f / np.sqrt(sig))) < 1e-12
    a2 = np.abs(f) ** 2
    assert abs(ctx.metric(hmc.METRIC_KINETIC, s, d) - 0.5 * np.sum(sig * a2)) < 1e-12 * np.sum(sig * a2)
    assert abs(ctx.metric(hmc.METRIC_MNORM, s, d) - np.sum(a2 / sig)) < 1e-12 * np.sum(a2 / sig)
    acc = dev(w)
    ctx.metric(hmc.METRIC_ACCUM, s, d, out=acc)
    assert rel(acc.cpu().numpy(), w + a2) < 1e-12
    out = d.clone()
    ctx.metric(hmc.METRIC_VELOCITY, s, out, out=out)   # in place
    assert rel(out.cpu().numpy(), back(sig * f)) < 1e-12
