"""Cells whose exponent bound sum_c |alpha_c| max|m_c| exceeds the fixed-point range (245) with finite values:
very small moments (alpha_0 m_0 below -245) and very peaked densities. Their rows are scaled by a
power of two; moments, ansatz and the network's residual pass against FP64 on the oracle's rule.

Tolerance of moments: 1e-14 + 16 eps max_q sum_c |alpha_c m_c(q)| of the largest one (alpha is rounded to eps
of terms of that size, and the exponent's absolute error is the exponential's relative one)."""
import numpy as np
import pytest

import oracle as O
from paper_2205_08417_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def K():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_08417_gb300 import build, kitrt
    build.build()
    return kitrt


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def moments(T, a):
    return (np.exp(a @ T.M.T) * T.w) @ T.M, (np.abs(a)[:, None, :] * np.abs(T.M)[None]).sum(axis=2).max(axis=1)


def check(U, ref, cond):
    err = np.abs(U - ref).max(axis=1) / np.abs(ref).max(axis=1)
    assert (err <= 1e-14 + 16 * EPS * cond).all(), (err / (1e-14 + 16 * EPS * cond)).max()


@pytest.mark.parametrize("N,order", [(1, 7), (2, 8), (3, 20), (5, 12)])
def test_closure_of_tiny_moments(K, N, order):
    m = synth.jittered_mesh(13, 0.0, 1.0, seed=3)
    mesh, T = K.Mesh(m.xy, m.tri), O.Tables(N, order)
    s, rng = K.MNSolver(mesh, N, order, tau=1e-12), np.random.default_rng(1)
    a = 0.5 * rng.normal(size=(mesh.ncells, T.n))
    a[:, 0] -= np.resize([0.0, 900.0, 1000.0, 1100.0], mesh.ncells)  # exp(-310) and ordinary rows
    u, cond = moments(T, a)
    got = dev(O.isotropic_alpha(T, u))
    s.closure(dev(u), got)
    check(moments(T, got.cpu().numpy())[0], u, cond)


@pytest.mark.parametrize("order", [7, 10])
def test_step_of_tiny_moments(K, order):
    m = synth.jittered_mesh(13, 0.0, 1.0, seed=3)
    mesh, G, T = K.Mesh(m.xy, m.tri), O.Geometry(m.xy, m.tri), O.Tables(2, order)
    C, rng = G.C, np.random.default_rng(2)
    a = 0.4 * rng.normal(size=(C, T.n))
    a[:, 0] -= 900.0
    u0 = moments(T, a)[0]
    sa, ss, q = rng.uniform(0, 1, C), rng.uniform(0, 1, C), np.zeros(C)
    dt = 0.5 * G.cfl_dt(0.4)
    want, a_or = u0.copy(), O.isotropic_alpha(T, u0)
    assert O.mn_run(T, G, want, a_or, sa, ss, q, dt, 3)[0] == 0
    s = K.MNSolver(mesh, 2, order, tau=1e-12)
    u = dev(u0)
    al = s.isotropic_alpha(u)
    s.step(u, al, dev(sa), dev(ss), dev(q), dt=dt, nsteps=3)
    # the exponents are about 255: the ansatz is known to 16 eps 255, a step averages it
    assert np.abs(u.cpu().numpy() - want).max() <= 16 * EPS * 260 * np.abs(want).max()


@pytest.mark.parametrize("mode", ["mixed_tf32", "mixed_bf16"])
@pytest.mark.parametrize("N,order", [(2, 10), (3, 21), (5, 30)])
def test_peaked_rows(K, mode, N, order):
    """Bounds of 250 to 1e5 whose exponents stay below 700: column 0 of the Hessian."""
    m = synth.jittered_mesh(13, 0.0, 1.0, seed=3)
    mesh, T = K.Mesh(m.xy, m.tri), O.Tables(N, order)
    s, rng = K.MNSolver(mesh, N, order, mode=mode), np.random.default_rng(3)
    C = mesh.ncells
    a = rng.normal(size=(C, T.n))
    a[:, 0] = 0.0
    z = (a @ T.M.T).max(axis=1)
    a *= (np.resize([30.0, 150.0, 1e3, 1e4, 4e4], C) / z)[:, None]
    a[:, 0] = (rng.uniform(-60, 60, C) - (a @ T.M.T).max(axis=1)) / T.M[0, 0]
    H = s.hessian(dev(a)).cpu().numpy()
    ref, cond = moments(T, a)
    check(H[:, :, 0] / T.M[0, 0], ref, cond)


@pytest.mark.parametrize("N,order", [(2, 20), (3, 30), (4, 24)])
def test_learned_pass_of_peaked_proposals(K, N, order):
    """A network whose output is one peaked alpha (its parameters are zero, the output's mean is alpha):
    the residual pass must find it right in the cells whose moments are that alpha's."""
    m = synth.jittered_mesh(13, 0.0, 1.0, seed=3)
    mesh, T = K.Mesh(m.xy, m.tri), O.Tables(N, order)
    s, rng = K.MNSolver(mesh, N, order, mode="learned", tau=1e-8), np.random.default_rng(4)
    C, d = mesh.ncells, T.n - 1
    a = np.zeros(T.n)
    a[1:] = rng.normal(size=d)
    a *= 300.0 / (np.abs(a) * np.abs(T.M).max(axis=0)).sum()
    a = a.astype(np.float32).astype(np.float64)
    rows = np.repeat(a[None], C, axis=0)
    rows[:, 0] = (rng.uniform(-3, 3, C) - (rows @ T.M.T).max(axis=1)) / T.M[0, 0]
    u, cond = moments(T, rows)
    zero, one = torch.zeros(d), torch.ones(d)
    s.set_mlp(torch.zeros(K.mlp_param_count(d, 64, d)).cuda(),
              torch.cat([zero, one, torch.from_numpy(a[1:].astype(np.float32)), one]).cuda())
    got = s.isotropic_alpha(dev(u))
    _, st = s.closure(dev(u), got, stats=True)
    assert st["fallbacks"] == 0 and st["evaluations"] == C, st
    got = got.cpu().numpy()
    assert (got[:, 1:] == a[1:]).all()
    # exp(alpha_0 m_0) = u_0 / U'_0: alpha_0 to the error of the moments over m_0
    assert (np.abs(got[:, 0] - rows[:, 0]) * T.M[0, 0] <= 1e-14 + 16 * EPS * cond).all()
