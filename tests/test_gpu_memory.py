"""Device memory of a solver: what it keeps per cell is its state, one column of moments, the ansatz
and the coefficients of the S_N step, in every mode."""
import gc

import numpy as np
import pytest

from paper_2205_08417_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["fp64", "mixed_tf32", "mixed_bf16", "learned"])
def test_bytes_per_cell(mode):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_08417_gb300 import build, kitrt as K
    build.build()
    N, order = 5, 6
    n, n2, npairs, qp = 21, 66, 231, 64  # Q' = 36 padded to a multiple of 32
    doubles = 3 * n + 4 + npairs + n2 + qp + 12
    ints = 7
    if mode != "fp64":
        doubles += 1 + qp / 2  # residual, FP32 ansatz
        ints += 3
    if mode == "learned":
        doubles += n
        ints += 1
    gc.collect()  # no solver of another test is freed between the readings
    used, cells, keep = [], [], []
    for k in (60, 480):  # the first one also loads the kernels
        m = synth.jittered_mesh(k, 0.0, 1.0, seed=1)
        mesh = K.Mesh(m.xy, m.tri)
        if not keep:
            keep.append(K.MNSolver(mesh, N, order, mode=mode))
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        keep.append(K.MNSolver(mesh, N, order, mode=mode))
        used.append(free - torch.cuda.mem_get_info()[0])
        cells.append(mesh.ncells)
    per_cell = (used[1] - used[0]) / (cells[1] - cells[0])
    # each of about 25 allocations is rounded up to 2 MiB at most
    slack = 25 * 2 ** 21 / (cells[1] - cells[0])
    print(mode, "bytes per cell", per_cell, "state", 8 * doubles + 4 * ints)
    assert np.isfinite(per_cell) and per_cell <= 8 * doubles + 4 * ints + slack
