"""The fixed-point quadrature sweeps against the oracle's full rule in FP64, at the shapes where their
bookkeeping can go wrong: odd and even orders (quads of azimuths with and without the pi/2 pair),
the smallest order of each degree, rings shorter than a work unit, the largest rule; exponents on
both sides of the fixed-point range; rows whose largest exponential comes late (the scale rises).

Tolerance: 1e-14 + 16 eps max_q sum_c |alpha_c m_c(q)| of the largest moment. The exponent is a sum
of terms of that size and alpha itself is rounded to eps of it, and its absolute error is the
exponential's relative one; 1e-14 covers the exponentials and the sums."""
import numpy as np
import pytest

import oracle as O
from paper_2205_08417_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(1, 2), (1, 7), (2, 3), (3, 4), (3, 9), (3, 20), (4, 15), (5, 6), (5, 30), (2, 64)]


@pytest.fixture(scope="module")
def K():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_08417_gb300 import build, kitrt
    build.build()
    return kitrt


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def solver(K, N, order, mode, k=13, **opts):
    m = synth.jittered_mesh(k, 0.0, 1.0, seed=3)
    mesh = K.Mesh(m.xy, m.tri)
    assert mesh.ncells % 128 != 0
    return K.MNSolver(mesh, N, order, mode=mode, **opts), O.Tables(N, order)


def alphas(T, count, size, seed):
    """Random alpha rows with sum_c |alpha_c| max|m_c| = size."""
    a = np.random.default_rng(seed).normal(size=(count, T.n))
    return a * (size / (np.abs(a) * np.abs(T.M).max(axis=0)).sum(axis=1))[:, None]


def moments(T, a):
    e = np.exp(a @ T.M.T) * T.w
    return e @ T.M, np.abs(a[:, None, :] * T.M[None]).sum(axis=2).max(axis=1)


def check(U, ref, cond):
    rel = np.abs(U - ref).max(axis=1) / np.abs(ref).max(axis=1)
    bound = 1e-14 + 16.0 * 2.0 ** -52 * cond
    print("max err", rel.max(), "max err/bound", (rel / bound).max())
    assert (rel <= bound).all(), (rel / bound).max()


@pytest.mark.parametrize("mode", ["mixed_tf32", "mixed_bf16"])
@pytest.mark.parametrize("N,order", SHAPES)
def test_mixed_sweep_moments(K, mode, N, order):
    """Column 0 of the Hessian is m_0 <m exp(alpha.m)>: small and large alpha, on both sides of the
    guard (245) beyond which a row's exponentials are formed in FP64."""
    s, T = solver(K, N, order, mode)
    C = s.mesh.ncells
    sizes = np.resize([0.0, 1e-9, 0.5, 20.0, 90.0, 244.9, 245.1, 600.0], C)
    a = np.concatenate([alphas(T, 1, z, i) for i, z in enumerate(sizes)])
    a[::5, 0] -= 30.0
    H = s.hessian(dev(a)).cpu().numpy()
    ref, cond = moments(T, a)
    check(H[:, :, 0] / T.M[0, 0], ref, cond)


@pytest.mark.parametrize("N,order", SHAPES)
@pytest.mark.parametrize("mode", ["fp64", "mixed_tf32"])
def test_closure_reproduces_moments(K, mode, N, order):
    """The closure's sweep (split over parts, scale from u_0): alpha closed from the isotropic start
    and from a start far off reproduces u."""
    s, T = solver(K, N, order, mode, tau=1e-13 if mode == "fp64" else 1e-12)
    C = s.mesh.ncells
    a = np.concatenate([alphas(T, 1, z, 100 + i) for i, z in enumerate(np.resize([0.1, 2.0, 6.0, 12.0], C))])
    a[:, 0] += np.random.default_rng(5).uniform(-40.0, 10.0, C)
    u, _ = moments(T, a)
    start = O.isotropic_alpha(T, u)
    start[::3, 0] -= 15.0  # e^-4 below the target: the scale comes from the row, not from u_0
    start[1::7, 1:] += 0.5
    got = dev(start)
    s.closure(dev(u), got)
    U, cond = moments(T, got.cpu().numpy())
    if mode == "fp64":
        check(U, u, cond)
    else:
        assert (np.linalg.norm(U - u, axis=1) <= 1e-11 * np.linalg.norm(u, axis=1)).all()


@pytest.mark.parametrize("mode", ["fp64", "mixed_tf32"])
def test_bad_rows_stay_alone(K, mode):
    """A NaN, an infinite and an overflowing start fail their own cells and no other."""
    s, T = solver(K, 3, 10, mode)
    C = s.mesh.ncells
    a = alphas(T, C, 3.0, 1)
    u, _ = moments(T, a)
    start = O.isotropic_alpha(T, u)
    start[5, 2], start[77, 0], start[130, 0] = np.nan, np.inf, 1e6
    st = torch.zeros(C, dtype=torch.int32, device="cuda")
    got = dev(start)
    s.closure(dev(u), got, st, check=False)
    bad = np.zeros(C, bool)
    bad[[5, 77, 130]] = True
    st = st.cpu().numpy()
    assert (st[bad] == 2).all() and (st[~bad] == 0).all(), st[bad]
