"""The SPIKE option counts at hdd_setup_deflation, not at a change of the batch."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("at_setup", [1, 0])
def test_batch_change_leaves_the_spike_form_as_the_set_up_chose_it(at_setup):
    """The option switched over while the batch changes and back after it: split solves run if, and
    only if, the set-up was asked for them (their matrices are formed when first used)."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    w = W.custom(100.0, 320, 4)
    s = Solver(0).assemble(w.k, w.N).setup_dd(4, 4, w.overlap)
    s.set_option("coarse_spike", at_setup).setup_deflation()
    s.set_option("coarse_spike", 1 - at_setup).setup_batch(1)
    s.set_option("coarse_spike", 1).set_option("coarse_dense", 0)
    v = torch.from_numpy(W.random_complex_fast(s.n, 6)).cuda()
    s.profile(True)
    s.ras_apply(v, inner_tol=1e-2, inner_prec=64)
    used = {d["name"] for d in s.profile_stats() if d["launches"]}
    s.profile(False)
    assert ("coarse_solve_df32_spike" in used) == bool(at_setup), used
