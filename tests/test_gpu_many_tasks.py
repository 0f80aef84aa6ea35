"""More (box, right-hand side) tasks than a grid's second dimension holds."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [4095, 4096])          # 65520 and 65536 tasks
def test_small_products_of_many_tasks_match_banded(nrhs):
    """The FP64 product of small orders (2 x 2 to 3 x 3 here) against the banded kernels, at its bar."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    s = Solver(0).assemble(5.0, 16).setup_dd(4, 4, 2).setup_batch(nrhs).setup_deflation()
    assert s.nsub * s.nrhs == 16 * nrhs
    v = torch.from_numpy(W.random_complex_fast(nrhs * s.n, 2)).cuda()
    z = {}
    for form in (0, 1):
        s.set_option("coarse_dense", form)
        s.profile(True)
        z[form], its = s.ras_apply(v, inner_tol=1e-2, inner_prec=128)
        used = {d["name"] for d in s.profile_stats() if d["launches"]}
        s.profile(False)
        assert ("coarse_solve_dense" in used) == bool(form), used
    assert float(torch.linalg.vector_norm(z[1] - z[0])) <= 1e-11 * float(torch.linalg.vector_norm(z[0]))
