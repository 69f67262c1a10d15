"""Peaked closures of the mixed modes whose cells go over to the FP64 Hessian, at the degrees whose factor
takes two or three rows a lane, and with a regularized dual: the cells' moments come from the
handed-over sweep's parts, their factor from the FP64 path of the Newton step."""
import numpy as np
import pytest

import oracle as O
from paper_2205_08417_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_08417_gb300 import build, kitrt
    build.build()
    return kitrt


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("mode", ["mixed_tf32", "mixed_bf16"])
@pytest.mark.parametrize("N,order,gamma", [(2, 16, 0.0), (4, 24, 0.0), (5, 30, 0.0), (3, 20, 1e-9), (4, 24, 1e-9)])
def test_handed_over_cells_converge(K, mode, N, order, gamma):
    m = synth.jittered_mesh(30, 0.0, 1.0, seed=4)
    mesh, T, tau = K.Mesh(m.xy, m.tri), O.Tables(N, order), 1e-9
    C = mesh.ncells
    mu, phi, w, ox, oy = O.quadrature(order)
    c, kap, wt = synth.vmf_mixtures(C, 77, kappa_hi=400.0)
    psi = synth.vmf_density(np.stack([ox, oy, mu], axis=1), c, kap, wt)
    u = psi @ (T.w[:, None] * T.M)
    opts = dict(reg_gamma=gamma) if gamma else {}
    s = K.MNSolver(mesh, N, order, mode=mode, tau=tau, **opts)
    a, st = s.isotropic_alpha(dev(u)), torch.zeros(C, dtype=torch.int32, device="cuda")
    _, stats = s.closure(dev(u), a, st, stats=True, check=False)
    assert stats["handovers"] > C // 100, stats
    a, ok = a.cpu().numpy(), st.cpu().numpy() == 0
    assert ok.mean() > 0.95, ok.mean()
    g = (np.exp(a @ T.M.T) * T.w) @ T.M - u
    if gamma:
        g[:, 1:] += gamma * a[:, 1:]
    cond = (np.abs(a)[:, None, :] * np.abs(T.M)[None]).sum(axis=2).max(axis=1)
    # the closure's own test, and the moments of alpha rounded to 53 bits
    bound = 1.01 * tau * np.linalg.norm(u, axis=1) + (1e-14 + 16 * 2.0 ** -52 * cond) * np.abs(u).max(axis=1) * T.n
    assert (np.linalg.norm(g, axis=1)[ok] <= bound[ok]).all()
