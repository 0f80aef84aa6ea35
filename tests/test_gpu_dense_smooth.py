"""Coarse products of large order on smooth data, where the digits' products add up instead of
cancelling: against the banded kernels."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# one box, so that right-hand sides can be shaped like its modes: orders 64², 81² and 90², 64² next to
# the first resonance, complex 64²
CASES = {
    "m4096": W.custom(4.0, 130, 1, 2),
    "m6561": W.custom(4.0, 164, 1, 2),
    "m8100": W.custom(4.0, 182, 1, 2),
    "m4096_resonant": W.custom(4.4, 130, 1, 2),
    "m4096_complex": W.custom(0.5, 127, 1, 2, bc=1),
}
NRHS = 100      # several column tiles: more than a tile's operator columns per SM


@pytest.mark.parametrize("name", CASES)
def test_smooth_right_hand_sides_match_banded(name):
    """Half-sines (the dominant mode of E⁻¹ for k below the first resonance), constants, a mode of
    higher order and a field of one sign, of all significands.  complex128: either form carries
    κ(E)·2^-53, κ(E) < 4e5 here; bar 1e-10.  complex64: the fine arithmetic sets the distance from the
    complex128 result, so the form with products may be at most twice as far from it as the banded one."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    w = CASES[name]
    s = Solver(0).assemble(w.k, w.N, bc=w.bc).setup_dd(1, 1, w.overlap).setup_batch(NRHS).setup_deflation()
    side = int(round(s.n ** 0.5))
    x = (np.arange(side) + (0 if w.bc else 1)) / w.N
    sx, s3 = np.sin(np.pi * x), np.sin(3 * np.pi * x)
    g = np.random.default_rng(3)
    shapes = [sx[:, None] * sx, np.ones((side, side)), s3[:, None] * s3, sx[:, None] * sx * g.uniform(0.9, 1.0, (side, side))]
    v = np.stack([shapes[r % 4] * (1.0 + r / NRHS) * (1.0 - 0.7j if r % 3 else 1.0) for r in range(NRHS)])
    v = torch.from_numpy(np.ascontiguousarray(v.astype(np.complex128).reshape(-1))).cuda()
    z = {}
    for prec in (128, 64):
        for dense in (0, 1):
            s.set_option("coarse_dense", dense).profile(True)
            z[prec, dense] = s.ras_apply(v, inner_tol=1e-2, inner_prec=prec)[0].reshape(NRHS, -1)
            used = {d["name"] for d in s.profile_stats() if d["launches"]}
            s.profile(False)
            assert ("coarse_solve_dense" in used) == bool(dense), used
    ref = z[128, 0]
    far = {q: torch.linalg.vector_norm(z[q] - ref, dim=1) / torch.linalg.vector_norm(ref, dim=1) for q in z}
    assert float(far[128, 1].max()) <= 1e-10, far[128, 1].topk(4)
    assert float(far[64, 1].max()) <= 2.0 * float(far[64, 0].max()), (far[64, 1].topk(4), far[64, 0].topk(4))
