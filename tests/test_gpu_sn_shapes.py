"""The S_N step by quads of azimuths at the shapes where its layout can go wrong, against the oracle's step:
every degree, the smallest orders, odd orders (no pi/2 pair), rings of more than 16 quads (one cell
per warp), lanes without a quad, cell counts that leave a warp partly empty."""
import numpy as np
import pytest

from test_gpu_sn import K, _run_pair  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("aniso", [False, True])
@pytest.mark.parametrize("N,order", [(1, 2), (1, 3), (4, 5), (5, 6), (4, 9), (5, 15), (3, 21), (2, 33), (3, 34), (5, 40)])
def test_sn_shapes(K, N, order, aniso, fp32):  # noqa: F811
    g = [0.7 ** l for l in range(N + 1)] if aniso else None
    bc = "vacuum" if order % 2 else "neumann"
    got, ref, _ = _run_pair(K, 7, N, order, bc, g, 3, fp32=fp32, seed=order)
    # FP64 as the other S_N tests; FP32: the start, three steps of about twenty operations, and a sum
    # over Q' ordinates per step, each at 6e-8
    assert np.abs(got - ref).max() <= (5e-6 if fp32 else 1e-12) * np.abs(ref).max()


@pytest.mark.parametrize("aniso", [False, True])
@pytest.mark.parametrize("N,order,k", [(1, 2, 7), (1, 3, 75), (4, 5, 75), (3, 9, 75), (5, 15, 40), (2, 22, 30), (1, 34, 24)])
def test_sn_layouts(K, N, order, k, aniso):  # noqa: F811
    """FP64 on meshes of both sides of the rule between a warp and a block per group of cells, and of one to
    eight parts of the rings."""
    g = [0.7 ** l for l in range(N + 1)] if aniso else None
    got, ref, _ = _run_pair(K, k, N, order, "vacuum", g, 2, fp32=False, seed=order)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
