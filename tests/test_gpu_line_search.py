"""Badly conditioned closures in the 8-lane Newton step: the line search compares values of the dual
<exp(alpha.m)> - alpha.u whose second term is a sum of parts far larger than itself, and stalls where its
rounding noise exceeds the slack. alpha.u is summed in the order of the components, as elsewhere."""
import math

import numpy as np
import pytest

from paper_2205_08417_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_stalled_closures(N=4, order=24, rows=12000, seeds=(3, 4, 5, 6)):
    """von Mises-Fisher mixtures to kappa = 50 on a rule that barely resolves them, closed and closed again
    from 2^-6 of their density. With ordered sums 20 of 12,000 stall or break down (a thread per cell:
    121 of 72,000), with a sum over the lanes 33 to 37 (198 to 220 of 72,000): 110 of 48,000 lies three
    standard deviations from both."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_08417_gb300 import build, kitrt as K
    build.build()
    m = synth.jittered_mesh(90, 0.0, 1.0, seed=2)
    s = K.MNSolver(K.Mesh(m.xy, m.tri), N, order, tau=1e-10)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    status = torch.zeros(rows, dtype=torch.int32, device="cuda")
    failed = []
    for seed in seeds:
        c, kap, wt = synth.vmf_mixtures(rows, seed, kappa_hi=50.0)
        scale = np.exp(np.random.default_rng(seed + 1).uniform(-4.0, 3.0, size=rows))
        u = s.vmf_moments(dev(c), dev(kap), dev(wt * scale[:, None]))
        m0 = 1.0 / math.sqrt(4.0 * math.pi)
        a = torch.zeros_like(u)
        a[:, 0] = torch.log(u[:, 0] / (4 * math.pi * m0)) / m0
        s.closure_batch(u, a, status, check=False)
        a[:, 0] -= 6 * math.log(2.0) / m0
        s.closure_batch(u, a, status, check=False)
        failed.append(int((status != 0).sum()))
    print("failed", failed)
    assert sum(failed) <= 110, failed
