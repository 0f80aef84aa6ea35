"""The two forms of the coarse operators' digits: bytes up to 32 columns a shape, BF16 beyond, and the
change between them when the batch changes."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,bar", [(128, 1e-11), (64, 1e-4)])
def test_digit_forms_match_banded_across_batches(prec, bar):
    """RAS applications with 1, 16, 17 and again 2 right-hand sides (2, 32, 34 and 4 columns a shape)
    against the banded kernels, at the bars of the product by digits."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    w = W.custom(40.0, 129, 2, 1, ifx=[0, 61, 129])           # boxes of different sizes: four shapes
    s = Solver(0).assemble(w.k, w.N).setup_dd(w.Sx, w.Sy, w.overlap, w.ifx, w.ify).setup_deflation()
    for nrhs in (1, 16, 17, 2):
        s.setup_batch(nrhs)
        v = torch.from_numpy(W.random_complex_fast(nrhs * s.n, 11)).cuda()
        z, its = {}, {}
        for form in (0, 1):
            s.set_option("coarse_dense", form)
            z[form], its[form] = s.ras_apply(v, inner_tol=1e-2, inner_prec=prec)
        assert float(torch.linalg.vector_norm(z[1] - z[0])) <= bar * float(torch.linalg.vector_norm(z[0])), nrhs
        if prec == 128:
            assert np.array_equal(its[0], its[1])
