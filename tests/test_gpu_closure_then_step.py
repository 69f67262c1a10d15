"""A step that continues from a closure: kitrt_closure leaves alpha and the solver's state, and a step on
the same moments with that alpha is the step that a fresh solver takes. In the mixed modes the step
transports the FP32 ansatz that the sweeps write, which a closure does not; cells that need no
Newton step must not transport the one of an earlier state."""
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


def solver(K, mesh, mode):
    s = K.MNSolver(mesh, 2, 8, mode=mode, tau=1e-8)
    if mode == "learned":
        g = torch.Generator().manual_seed(1)
        s.set_mlp((0.2 * torch.randn(K.mlp_param_count(5, 64, 5), generator=g)).cuda(),
                  torch.cat([torch.zeros(5), torch.ones(5), torch.zeros(5), torch.ones(5)]).cuda())
    return s


@pytest.mark.parametrize("mode", ["fp64", "mixed_tf32", "mixed_bf16", "learned"])
@pytest.mark.parametrize("stepped", [False, True])
def test_step_after_closure(K, mode, stepped):
    """stepped: the solver has stepped another state before, so that its ansatz is an old one."""
    m = synth.jittered_mesh(16, 0.0, 1.0, seed=2)
    mesh, G, T = K.Mesh(m.xy, m.tri), O.Geometry(m.xy, m.tri), O.Tables(2, 8)
    C, rng = G.C, np.random.default_rng(4)
    al = 0.4 * rng.normal(size=(C, T.n))
    u0 = np.exp(al @ T.M.T) @ (T.w[:, None] * T.M)
    sa, ss, q = rng.uniform(0.0, 1.0, C), rng.uniform(0.0, 1.0, C), np.zeros(C)
    dt = 0.5 * G.cfl_dt(0.4)
    s = solver(K, mesh, mode)
    if stepped:
        other = 3.0 * u0[::-1].copy()
        a = s.isotropic_alpha(dev(other))
        s.step(dev(other), a, dev(sa), dev(ss), dev(q), dt=dt)
    u, want = dev(u0), u0.copy()
    a = s.isotropic_alpha(u)
    s.closure(u, a)
    s.step(u, a, dev(sa), dev(ss), dev(q), dt=dt, nsteps=2)
    a_or = O.isotropic_alpha(T, want)
    assert O.mn_run(T, G, want, a_or, sa, ss, q, dt, 2)[0] == 0
    err = np.linalg.norm(u.cpu().numpy() - want) / np.linalg.norm(want)
    # FP64: round-off of two steps; mixed: the FP32 ansatz and flux (6e-8 each) and the closure's 1e-8;
    # learned: proposals are accepted at 1e-6. A stale ansatz gives 1e-2 or more.
    assert err <= {"fp64": 1e-12, "learned": 1e-5}.get(mode, 1e-6), err
