"""A learned step whose network proposes points that overflow, on a solver that has stepped before: a
cell whose alpha the caller has replaced starts from that alpha, never from the stored moments and
factor of the point that the solver kept for it."""
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


@pytest.mark.parametrize("N,order", [(1, 6), (2, 8), (4, 12)])
def test_replaced_alpha_with_overflowing_network(K, N, order):
    m = synth.jittered_mesh(14, 0.0, 1.0, seed=2)
    mesh, G, T = K.Mesh(m.xy, m.tri), O.Geometry(m.xy, m.tri), O.Tables(N, order)
    C, rng = G.C, np.random.default_rng(5)
    al = 0.3 * rng.normal(size=(C, T.n))
    u0 = np.exp(al @ T.M.T) @ (T.w[:, None] * T.M)
    sa, ss, q = np.zeros(C), rng.uniform(0.0, 1.0, C), np.zeros(C)
    dt = 0.5 * G.cfl_dt(0.4)
    d = T.n - 1
    s = K.MNSolver(mesh, N, order, mode="learned", tau=1e-8)
    one, zero = torch.ones(d), torch.zeros(d)
    # outputs scaled by 1e6: exp overflows at half of the directions, so no proposal is finite
    g = torch.Generator().manual_seed(1)
    p = (0.2 * torch.randn(K.mlp_param_count(d, 64, d), generator=g)).cuda()
    s.set_mlp(p, torch.cat([zero, one, zero, 1e6 * one]).cuda())
    sad, ssd, qd = dev(sa), dev(ss), dev(q)
    u = dev(u0)
    a = s.isotropic_alpha(u)
    s.step(u, a, sad, ssd, qd, dt=dt)
    # the same moments again: the stored point is their closure; the caller's alpha is not
    u, want = dev(u0), u0.copy()
    start = O.isotropic_alpha(T, u0)
    start[:, 0] += 0.5
    a = dev(start)
    s.step(u, a, sad, ssd, qd, dt=dt)
    a_or = O.isotropic_alpha(T, want)
    assert O.mn_run(T, G, want, a_or, sa, ss, q, dt, 1)[0] == 0
    # FP32 ansatz and flux (6e-8 each) and a closure to 1e-8
    err = np.linalg.norm(u.cpu().numpy() - want) / np.linalg.norm(want)
    aerr = np.abs(a.cpu().numpy() - a_or).max()
    assert err <= 1e-6 and aerr <= 1e-5, (err, aerr)
