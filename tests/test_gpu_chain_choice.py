"""FP64 outer passes on either side of the line between chained and plain launches."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [138, 142])       # 137² <= 64·304 < 141²
def test_chained_and_plain_fp64_passes_repeat(N):
    """The same bits with and without a synchronisation between the calls that surround a solve."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    s = Solver.from_workload(W.custom(40.0, N, 3))
    s.set_option("outer_dots_df", 0)
    f = torch.from_numpy(W.random_complex_fast(s.n, 4)).cuda()
    opt = dict(inner_prec=128, outer_maxit=25, outer_restart=25, raise_on_error=False, outer_tol=1e-10, outer_reorth32=0)
    torch.cuda.synchronize()
    x, st = s.solve(f, **opt)
    torch.cuda.synchronize()
    for _ in range(3):
        g = f.clone()
        y, st2 = s.solve(g, **opt)
        g.zero_()
        assert torch.equal(x, y) and st2["outer_its"] == st["outer_its"]
