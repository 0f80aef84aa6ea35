"""The clustered banded LU (and the one-CTA kernel that serves wider windows) through the solves
made from its factors."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# (workload, both matrices): bandwidths of one and several columns per CTA of a cluster, windows
# wider than the matrix, uneven shapes
CASES = {
    "tiny_boxes": W.custom(3.0, 8, 2, 1, Sy=2, ifx=[0, 3, 8]),
    "one_row_of_boxes": W.custom(20.0, 40, 1, 1, Sy=13),
    "uneven": W.custom(50.0, 90, 3, 3, Sy=2, ifx=[0, 17, 61, 90]),
    "widest_box": W.custom(30.0, 257, 1, 1, Sy=36),
    "impedance": W.custom(40.0, 60, 2, 2, bc=1),
    "impedance_wide": W.custom(20.0, 200, 1, 1, Sy=50, bc=1),      # window too wide for the cluster kernel
}


@pytest.mark.parametrize("name", CASES)
def test_factors_solve_like_the_oracle(name):
    """E⁻¹ and A_j⁻¹ in FP64 by the banded kernels: the parity bars of the local operators, scaled
    by the condition where the box is closer to a resonance: backward error of the solution on the
    oracle's own matrices below 1e-13·order."""
    torch = pytest.importorskip("torch")
    import oracle
    from paper_2103_17081_gb300 import Solver
    w = CASES[name]
    s = Solver.from_workload(w, exact=True)
    p = oracle.from_workload(w, exact=False)
    fo, co = s.offsets()
    for op, off, seed in (("Ainv", fo, 3), ("Einv", co, 4)):
        x = W.random_complex_fast(off[-1], seed)
        y = s.local_op(op, torch.from_numpy(x).cuda(), 128).cpu().numpy()
        for q in range(0, p.nsub, max(1, p.nsub // 8)):
            b, u = x[off[q]:off[q + 1]], y[off[q]:off[q + 1]]
            A = p.sub_A(q)
            if op == "Einv":
                Z = p.sub_Z(q)
                A = Z.T @ A @ Z
            r = b - A @ u
            scale = float(abs(A).sum(axis=1).max()) * np.linalg.norm(u) + np.linalg.norm(b)
            assert np.linalg.norm(r) <= 1e-13 * len(b) * scale, (op, q)


def test_far_interchanges_stay_refused():
    """Four points per wavelength: pivoting carries multipliers beyond the window of the blocked
    solve, which set-up reports instead of solving wrongly."""
    from paper_2103_17081_gb300 import HDDError, Solver
    with pytest.raises(HDDError) as e:
        Solver.from_workload(W.custom(60.0, 40, 2, 2))
    assert e.value.code == 1
