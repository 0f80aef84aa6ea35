"""The coarse grid's sine transforms at the edges of their tiling."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,c", [(12, 2), (62, 2), (64, 2), (66, 3), (330, 2), (654, 2)])
def test_sine_transform_solve_matches_dense_transform(N, c):
    """The coarse solve's four transform passes (rows paired about the middle of the range) against
    the same products with a dense sine matrix, for even and odd Nc, one and several tiles, and more
    pairs than are staged at a time.  FP64: orthogonal transforms, 1e-13 of the largest |D⁻¹| ‖y‖;
    FP32 accordingly 2e-6 (each pass rounds within √m·u, m <= 326)."""
    from paper_2103_17081_gb300 import Solver
    torch = pytest.importorskip("torch")
    k = 0.55 * N
    s = Solver(0).assemble(k, N).setup_dd(1 if N < 250 else 3, 1 if N < 250 else 3, 1).setup_coarse_grid(c)
    Nc = N // c
    m = Nc - 1
    i = np.arange(1, Nc)
    S = np.sqrt(2.0 / Nc) * np.sin(np.pi * np.outer(i, i) / Nc)
    lam = 4 * np.sin(np.pi * i / (2 * Nc)) ** 2
    D = lam[:, None] + lam[None, :] - (k / Nc) ** 2
    y = W.random_complex_fast(m * m, 3).reshape(m, m)
    ref = S @ ((S @ y @ S) / D) @ S
    scale = np.linalg.norm(y) / np.min(np.abs(D))
    for prec, bar in ((128, 1e-13), (64, 2e-6)):
        x = s.coarse_grid_op("S", torch.from_numpy(y.reshape(-1)).cuda(), prec).cpu().numpy().reshape(m, m)
        assert np.linalg.norm(x - ref) <= bar * scale, (N, c, prec, np.linalg.norm(x - ref) / scale)
