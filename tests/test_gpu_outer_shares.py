"""The outer iteration's dots and update where their plans change: few and many chunks of the
vectors, shares of the basis, one, two and four thread groups per element pair."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


# (k, N, S, iterations, right-hand sides): vectors shorter than the chunks, odd lengths, lengths on
# either side of 32 k and 64 k pairs, bases past the 64 and 128 vectors from which groups share them
@pytest.mark.parametrize("k,N,S,its,nrhs", [(4.0, 8, 2, 12, 1), (30.0, 64, 4, 70, 3), (60.0, 150, 8, 140, 1),
                                            (60.0, 256, 8, 140, 2), (60.0, 258, 8, 80, 1), (40.0, 364, 4, 40, 1)])
def test_shared_dots_and_updates_give_the_fp64_iteration(k, N, S, its, nrhs):
    """Against FP64 dots and updates with complex128 inner solves: residual histories to 1e-6 while
    above 1e-4 and solutions to 1e-5 (the bars of the double-FP32 form), also of the first
    right-hand side of a batch."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    w = W.custom(k, N, S)
    s = Solver.from_workload(w)
    f = torch.from_numpy(W.random_complex_fast(s.n, 5)).cuda()
    opt = dict(inner_prec=128, outer_maxit=its, outer_restart=its, raise_on_error=False, outer_tol=1e-6)
    xl, stl = s.solve(f, **opt)
    if nrhs > 1:
        b = Solver.from_workload(w, deflation=False)
        b.setup_batch(nrhs)
        b.setup_deflation()
        fb = torch.from_numpy(np.concatenate([W.random_complex_fast(s.n, 5 + r) for r in range(nrhs)])).cuda()
        xb, _ = b.solve(fb, **opt)
    s.set_option("outer_dots_df", 0)
    x64, st64 = s.solve(f, **opt)
    h, h64 = np.array(stl["res_history"]), np.array(st64["res_history"])
    m = min(len(h), len(h64))
    early = h64[:m] >= 1e-4
    np.testing.assert_allclose(h[:m][early], h64[:m][early], rtol=1e-6)
    assert float(torch.linalg.vector_norm(xl - x64)) <= 1e-5 * float(torch.linalg.vector_norm(x64))
    if nrhs > 1:
        assert float(torch.linalg.vector_norm(xb[:s.n] - x64)) <= 1e-5 * float(torch.linalg.vector_norm(x64))
