"""Coarse solves of small order as FP64 products with explicit inverses, against the banded kernels."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# orders 1, next to multiples of 8 rows, below and above the 128 columns loaded ahead, several shapes
# and right-hand sides, complex E
CASES = {
    "m1": (W.custom(1.0, 6, 2, 1), 1),
    "m64": (W.custom(20.0, 32, 2, 1), 1),
    "m_ragged": (W.custom(17.0, 45, 3, 2, Sy=4, ifx=[0, 11, 29, 45]), 2),
    "m144": (W.custom(15.0, 48, 2, 1), 1),
    "m529": (W.custom(25.0, 90, 2, 1), 1),
    "impedance": (W.custom(20.0, 40, 2, 1, bc=1), 3),
    "impedance_ragged": (W.custom(12.0, 36, 3, 2, Sy=2, ifx=[0, 10, 23, 36], bc=1), 1),
}


@pytest.mark.parametrize("name", CASES)
def test_small_products_match_banded(name):
    """RAS applications with both forms: complex128 to 1e-11 with equal counts (either inverse
    carries κ(E)·2^-53), complex64 to 1e-4, the bars of the product by digits."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    w, nrhs = CASES[name]
    s = Solver(0).assemble(w.k, w.N, bc=w.bc).setup_dd(w.Sx, w.Sy, w.overlap, w.ifx, w.ify)
    if nrhs > 1:
        s.setup_batch(nrhs)
    s.setup_deflation()
    v = torch.from_numpy(W.random_complex_fast(nrhs * s.n, 7)).cuda()
    for prec, bar in ((128, 1e-11), (64, 1e-4)):
        z, its, used = {}, {}, {}
        for form in (0, 1):
            s.set_option("coarse_dense", form)
            s.profile(True)
            z[form], its[form] = s.ras_apply(v, inner_tol=1e-2, inner_prec=prec)
            used[form] = {d["name"]: d["launches"] for d in s.profile_stats() if d["launches"]}
            s.profile(False)
        assert used[1].get("coarse_solve_dense", 0) > 0 and "coarse_solve_dense" not in used[0]
        assert float(torch.linalg.vector_norm(z[1] - z[0])) <= bar * float(torch.linalg.vector_norm(z[0])), prec
        if prec == 128:
            assert np.array_equal(its[0], its[1])
