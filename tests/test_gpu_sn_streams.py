"""S_N calls of one solver on several streams, and in a captured graph: every call takes its own
coefficients (dt / A, cross sections, source), whatever runs beside it."""
import numpy as np
import pytest

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


def setup(K, dtype):
    m = synth.jittered_mesh(60, 0.0, 1.0, seed=3)
    s = K.MNSolver(K.Mesh(m.xy, m.tri), 3, 12)
    C, rng = s.mesh.ncells, np.random.default_rng(1)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    sets = [dict(sa=d(rng.uniform(0, 2, C)), ss=d(rng.uniform(0, 2, C)), q=d(rng.uniform(0, 1, C)),
                 psi=d(rng.uniform(0.5, 2.0, (C, s.Qf))).to(dtype)) for _ in range(4)]
    return s, sets


def call(s, c, psi, work, dt, n):
    s.sn_step(psi, work, c["sa"], c["ss"], c["q"], dt=dt, nsteps=n)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_calls_on_two_streams(K, dtype):
    s, sets = setup(K, dtype)
    dt = s.mesh.geometry()["min_inradius"] * 0.3
    want = []
    for i, c in enumerate(sets):
        p, w = c["psi"].clone(), torch.empty_like(c["psi"])
        call(s, c, p, w, dt * (1 + i) / 4, 7 + i)
        torch.cuda.synchronize()
        want.append(p)
    streams = [torch.cuda.Stream() for _ in range(2)]
    bufs = [(c["psi"].clone(), torch.empty_like(c["psi"])) for c in sets]
    torch.cuda.synchronize()
    for i, (c, (p, w)) in enumerate(zip(sets, bufs)):
        with torch.cuda.stream(streams[i % 2]):
            call(s, c, p, w, dt * (1 + i) / 4, 7 + i)
    torch.cuda.synchronize()
    for (p, _), ref in zip(bufs, want):
        assert torch.equal(p, ref)


def test_captured_call(K):
    """A graph's replay beside an eager call on another stream."""
    s, sets = setup(K, torch.float32)
    dt = s.mesh.geometry()["min_inradius"] * 0.3
    want = []
    for c, n in zip(sets[:2], (6, 20)):
        p, w = c["psi"].clone(), torch.empty_like(c["psi"])
        call(s, c, p, w, dt, n)
        want.append(p)
    (a, b), (p, q) = sets[:2], [c["psi"].clone() for c in sets[:2]]
    wp, wq = torch.empty_like(p), torch.empty_like(q)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call(s, a, p, wp, dt, 6)
    assert torch.equal(p, a["psi"])  # captured, not run
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        call(s, b, q, wq, dt, 20)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(p, want[0]) and torch.equal(q, want[1])
    p.copy_(a["psi"])
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(p, want[0])
