"""The -DHMC_BOUNDS build on the one-launch solver, the metric operations, the preconditioner and the twisted
transforms: solves as one block, a cluster and a cooperative team, with blocks that own nothing and tiles that are
partly empty, in both precisions; batches in flight and queued; planes and lines of the metric. Nothing may be
recorded, and every call returns its ordinary status (in a subprocess that loads the library through HMC_LIBRARY)."""

import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys, torch
sys.path.insert(0, sys.argv[1])
from paper_2204_14241_gb300 import hmc as H, presets
assert H.LIB_PATH.endswith("libhmc_bounds.so"), H.LIB_PATH
KW = presets.baseline()
words = {}
def note(name):
    torch.cuda.synchronize()
    w, enabled = H.bounds_status()
    assert enabled
    words[name] = w
g = torch.Generator(device="cuda")
g.manual_seed(1)
real = lambda *s: torch.randn(s, generator=g, device="cuda", dtype=torch.float64)
vec = lambda k, L, Nt: torch.view_as_complex(real(k, Nt, L, L, 2, 2, 2))
field = lambda L, Nt: 0.3 * real(3, Nt, L, L)
for L, Nt, K in ((4, 4, 1), (2, 35, 2), (6, 9, 2), (8, 8, 1), (12, 20, 1), (18, 35, 3), (20, 24, 2), (14, 42, 1)):
    for solver in ("mixed", "fp64"):
        ctx = H.Context(L, Nt, solver=solver, nrhs_max=K, cg_tol=1e-10, initial_guess=1, **KW)
        phi, b = field(L, Nt), vec(K, L, Nt)
        for precond in (False, True):
            _, st = ctx.cg_solve(phi, b, precond=precond)
            assert st["converged"]
            note(f"solve {L} {Nt} {K} {solver} {precond}")
        o = ctx.trajectory([phi], [torch.ones_like(phi)], 0.02, 2, nrhs=K, precond=True, seed=1, counter=0)
        assert o["status"] == 0
        note(f"trajectory {L} {Nt} {K} {solver}")
        if solver == "fp64":
            for t in (b, b.to(torch.complex64)):
                ctx.apply_precond(t)
                note(f"precond {L} {Nt} {t.dtype}")
            ctx.green_estimate(phi, torch.sign(b.real).to(torch.complex128))
            note(f"green {L} {Nt}")
        ctx.close()
for L, Nt in ((4, 7), (18, 35), (64, 128), (80, 160)):
    ctx = H.Context(L, Nt, **KW)
    phi, sig = field(L, Nt), 1.0 + real(3, Nt, L, L) ** 2
    for op in range(5):
        ctx.metric(op, sig, phi)
        note(f"metric {L} {Nt} {op}")
    ctx.close()
for n in (3, 260):
    chains = [(8, 10, 0.3) if i % 2 else (4, 6, 0.4) for i in range(n)]
    ctx = H.Context(8, 10, solver="mixed", nrhs_max=2, chains=chains, batch_chains=1, **{**KW, "r": 0.3})
    phis = [field(L, Nt) for L, Nt, _ in chains]
    o = ctx.trajectory(phis, [torch.ones_like(p) for p in phis], 0.02, 2, nrhs=2, seed=2, counter=0)
    assert o["status"] == 0
    note(f"batch {n}")
print(json.dumps(words))
"""


def test_nothing_recorded():
    from paper_2204_14241_gb300 import build
    lib = os.path.join(ROOT, "paper_2204_14241_gb300", "libhmc_bounds.so")
    if not os.path.exists(lib):
        build.build(variant="_bounds")
    env = dict(os.environ, HMC_LIBRARY=lib)
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    words = json.loads(r.stdout.strip().splitlines()[-1])
    assert len(words) > 80 and not any(words.values()), {k: w for k, w in words.items() if w}
