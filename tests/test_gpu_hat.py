"""Restriction and interpolation of the coarse grid against the hat functions themselves, with the
weights from the table and beyond it, and grids of one and several blocks."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,c", [(12, 2), (264, 2), (60, 3), (96, 16), (516, 258)])
def test_restrict_and_prolong_are_the_hat_sums(N, c):
    """φ(dx, dy) = max(0, 1 - max(|dx|, |dy|, |dx ∓ dy|)/c) with the mesh's diagonal: FP64 sums of at
    most (2c-1)² products, 1e-14·√terms; FP32 coarse vectors 2e-7."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    s = Solver(0).assemble(0.2 * N / max(1, c // 8), N).setup_dd(4 if N > 250 else 1, 4 if N > 250 else 1, 1)
    s.setup_coarse_grid(c)
    m, w = N // c - 1, N - 1
    d = np.arange(1 - c, c)
    diff = np.maximum(np.maximum(np.abs(d)[:, None], np.abs(d)[None, :]), np.abs(d[None, :] - d[:, None]))
    hats = [np.maximum(0.0, 1.0 - diff / c), np.maximum(0.0, 1.0 - diff / c)[:, ::-1]]     # [dy, dx], either diagonal
    v = W.random_complex_fast(w * w, 5).reshape(w, w)
    y = W.random_complex_fast(m * m, 6).reshape(m, m)
    want = []
    for hat in hats:
        r, p = np.zeros((m, m), complex), np.zeros((w, w), complex)
        for J in range(m):
            for I in range(m):
                sl = (slice(c * J, c * J + 2 * c - 1), slice(c * I, c * I + 2 * c - 1))
                r[J, I] = (hat * v[sl]).sum()
                p[sl] += hat * y[J, I]
        want.append((r, p))
    for prec, bar in ((128, 1e-14 * (2 * c - 1)), (64, 2e-7)):
        r = s.coarse_grid_op("R", torch.from_numpy(v.reshape(-1)).cuda(), prec).cpu().numpy().reshape(m, m)
        p = s.coarse_grid_op("P", torch.from_numpy(y.reshape(-1)).cuda(), prec).cpu().numpy().reshape(w, w)
        err = [max(np.linalg.norm(r - a) / np.linalg.norm(a), np.linalg.norm(p - b) / np.linalg.norm(b)) for a, b in want]
        assert min(err) <= bar, (prec, err)
