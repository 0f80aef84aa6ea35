"""FP64 outer dots on short vectors: chunks of up to two rounds of a warp, groups of four vectors with
a remainder, few chunks."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,N,S,its", [(6.0, 12, 2, 30), (20.0, 33, 3, 45), (40.0, 100, 5, 60), (50.0, 140, 4, 40)])
def test_short_fp64_dots_give_the_double_fp32_iteration(k, N, S, its):
    """Residual histories to 1e-6 while above 1e-4, solutions to 1e-5: the bars between the two
    forms of the outer dots."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    s = Solver.from_workload(W.custom(k, N, S))
    f = torch.from_numpy(W.random_complex_fast(s.n, 15)).cuda()
    opt = dict(inner_prec=128, outer_maxit=its, outer_restart=its, raise_on_error=False, outer_tol=1e-8)
    h, x = {}, {}
    for df in (0, 1):
        s.set_option("outer_dots_df", df)
        x[df], st = s.solve(f, outer_reorth32=df, **opt)
        h[df] = np.array(st["res_history"])
    m = min(len(h[0]), len(h[1]))
    early = h[0][:m] >= 1e-4
    np.testing.assert_allclose(h[1][:m][early], h[0][:m][early], rtol=1e-6)
    assert float(torch.linalg.vector_norm(x[1] - x[0])) <= 1e-5 * float(torch.linalg.vector_norm(x[0]))
