"""The one-launch Arnoldi step where its work splits change: clusters with CTAs that hold no rows,
boxes narrower than a warp, bases past four and eight vectors, a Krylov space that is exhausted
(the directly summed norm), the impedance rows."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "boxes_of_3_rows": (W.custom(3.0, 8, 2, 1, Sy=4), 1e-10, 30),
    "exhausted": (W.custom(2.0, 6, 2, 1), 1e-14, 40),
    "long_bases": (W.custom(45.0, 72, 3, 2, Sy=2, ifx=[0, 19, 47, 72]), 1e-10, 40),
    "restarted": (W.custom(45.0, 72, 3, 2), 1e-8, 5),
    "one_wide_row": (W.custom(12.0, 90, 1, 2, Sy=9), 1e-10, 30),
    "impedance": (W.custom(30.0, 64, 2, 2, Sy=3, bc=1), 1e-10, 40),
}


@pytest.mark.parametrize("name", CASES)
def test_step_matches_separate_kernels(name):
    """complex128: the solution bar of 1e-9, counts within one per task (a residual on the tolerance
    may fall on either side); complex64 at 1e-3: 1e-4."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    w, tol, restart = CASES[name]
    s = Solver.from_workload(w)
    v = torch.from_numpy(W.random_complex_fast(s.n, 3)).cuda()
    for prec, t, bar in ((128, tol, 1e-9), (64, 1e-3, 1e-4)):
        z, its = {}, {}
        for fused in (0, 1):
            s.set_option("fused_inner", fused)
            z[fused], its[fused] = s.ras_apply(v, inner_tol=t, inner_prec=prec, inner_restart=restart,
                                               inner_maxit=60)
        assert float(torch.linalg.vector_norm(z[1] - z[0])) <= bar * float(torch.linalg.vector_norm(z[0])), prec
        if prec == 128:
            assert np.abs(np.array(its[1]) - np.array(its[0])).max() <= 1
