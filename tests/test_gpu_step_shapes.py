"""Steps and the adjoint against the oracle at the shapes where the quad layout of the FP64 flux, of
the ansatz and of the adjoint can go wrong: odd orders (no pi/2 pair), one to several cells per warp,
the smallest order of a degree, a ragged number of cells, both walls, a density.

Bars: 1e-11 relative L2 for FP64 steps (both sides solve the closure to round-off by the polish
step; the rest is rounding over a few steps), 1e-6 for the mixed modes' FP32 ansatz and flux,
1e-10 of the largest gradient for the adjoint (rounding through a few solves with H)."""
import numpy as np
import pytest

import oracle as O
from paper_2205_08417_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(1, 3), (1, 6), (2, 5), (3, 7), (3, 10), (3, 20), (4, 9), (5, 13), (3, 33), (2, 64)]


@pytest.fixture(scope="module")
def K():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_08417_gb300 import build, kitrt
    build.build()
    return kitrt


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def case(N, order, k=11, seed=4):
    """Anisotropic moments of exp(alpha . m) with smooth random alpha."""
    m = synth.jittered_mesh(k, 0.0, 7.0, seed=seed)
    G, T = O.Geometry(m.xy, m.tri), O.Tables(N, order)
    rng = np.random.default_rng(seed + order)
    x = m.centroids() / 7.0
    a = np.stack([np.cos(x @ rng.normal(size=2) * 4 + rng.uniform(0, 6)) for _ in range(T.n)], axis=1)
    a[:, 0] -= 3.0
    u = (np.exp(a @ T.M.T) * T.w) @ T.M
    blk, sa, ss = synth.block_coefficients(m.centroids(), 0.0, 7.0, 7, seed, sa_max=2.0)
    q = np.where(blk == 24, 1.0, 0.0)
    dt = min(G.cfl_dt(0.4), 0.3)
    return m, G, T, u, blk, sa, ss, q, dt


@pytest.mark.parametrize("mode,bar", [("fp64", 1e-11), ("mixed_tf32", 1e-6)])
def test_predictor_in_segments(K, mode, bar):
    """M_5 on more cells (a ragged last warp) than the predictor takes with whole factors in shared
    memory: its rows then come in segments."""
    m, G, T, u0, blk, sa, ss, q, dt = case(5, 12, k=90)
    assert len(u0) > 152 * 96 and len(u0) % 32
    u, a = u0.copy(), O.isotropic_alpha(T, u0)
    nf, _ = O.mn_run(T, G, u, a, sa[blk], ss[blk], q, dt, 3, bc=0)
    assert nf == 0
    s = K.MNSolver(K.Mesh(m.xy, m.tri), 5, 12, mode=mode, bc="neumann")
    ud = dev(u0)
    s.step(ud, s.isotropic_alpha(ud), dev(sa[blk]), dev(ss[blk]), dev(q), dt=dt, nsteps=3)
    assert rel_l2(ud.cpu().numpy(), u) <= bar


@pytest.mark.parametrize("bc", ["neumann", "vacuum"])
@pytest.mark.parametrize("mode,bar", [("fp64", 1e-11), ("mixed_tf32", 1e-6)])
@pytest.mark.parametrize("N,order", SHAPES)
def test_step(K, N, order, mode, bar, bc):
    m, G, T, u0, blk, sa, ss, q, dt = case(N, order)
    u, a = u0.copy(), O.isotropic_alpha(T, u0)
    nf, _ = O.mn_run(T, G, u, a, sa[blk], ss[blk], q, dt, 3, bc=int(bc == "vacuum"))
    assert nf == 0
    s = K.MNSolver(K.Mesh(m.xy, m.tri), N, order, mode=mode, bc=bc)
    ud = dev(u0)
    ad = s.isotropic_alpha(ud)
    s.step(ud, ad, dev(sa[blk]), dev(ss[blk]), dev(q), dt=dt, nsteps=3)
    err = rel_l2(ud.cpu().numpy(), u)
    print(mode, bc, N, order, err)
    assert err <= bar


@pytest.mark.parametrize("bc", ["neumann", "vacuum"])
@pytest.mark.parametrize("N,order", [(2, 5), (3, 10), (5, 13)])
def test_density_step(K, N, order, bc):
    m, G, T, u0, blk, sa, ss, q, dt = case(N, order)
    rho = 1.0 + 3.0 * np.random.default_rng(1).random(G.C)
    u, a = u0.copy(), O.isotropic_alpha(T, u0)
    nf, _ = O.mn_run_rho(T, G, rho, u, a, sa[blk], ss[blk], q, dt, 3, bc=int(bc == "vacuum"))
    assert nf == 0
    s = K.MNSolver(K.Mesh(m.xy, m.tri), N, order, bc=bc)
    s.set_density(dev(rho))
    ud = dev(u0)
    s.step(ud, s.isotropic_alpha(ud), dev(sa[blk]), dev(ss[blk]), dev(q), dt=dt, nsteps=3)
    assert rel_l2(ud.cpu().numpy(), u) <= 1e-11


@pytest.mark.parametrize("bc", ["neumann", "vacuum"])
@pytest.mark.parametrize("N,order", SHAPES[:8])
def test_adjoint(K, N, order, bc):
    m, G, T, u0, blk, sa, ss, q, dt = case(N, order)
    target = np.isin(blk, [16, 17, 18, 23, 24, 25, 30, 31, 32]).astype(np.uint8)
    a0 = O.isotropic_alpha(T, u0)
    J, ga, gs = O.mn_adjoint(T, G, blk, sa, ss, q, target, dt, 4, u0, a0, bc=int(bc == "vacuum"))
    s = K.MNSolver(K.Mesh(m.xy, m.tri), N, order, bc=bc)
    Jd, gad, gsd = s.adjoint(dev(u0), dev(a0), dev(sa[blk]), dev(ss[blk]), dev(q), dev(blk), 49, dev(target), dt, 4, 3)
    assert abs(Jd - J) <= 1e-12 * abs(J)
    for x, y in ((gad, ga), (gsd, gs)):
        err = np.abs(x - y).max() / np.abs(y).max()
        print(bc, N, order, err)
        assert err <= 1e-10
