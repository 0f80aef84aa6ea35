"""First calls of a context on a stream that does not wait for the default one: what a solve prepares on
first use is uploaded on the caller's stream."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dense", [1, 0])
@pytest.mark.parametrize("prec", [64, 128])
def test_first_application_on_a_side_stream(prec, dense):
    """Plans of the coarse products (dense) and the SPIKE matrices of the banded solves (not dense, formed
    late as the set-up took the products): the bits of a context that has run on the default stream."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    w = W.custom(60.0, 190, 3)
    ref = None
    for stream in (torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.Stream()):
        s = Solver(0).assemble(w.k, w.N).setup_dd(3, 3, w.overlap).setup_batch(2)
        v = torch.from_numpy(W.random_complex_fast(2 * s.n, 3)).cuda()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            s.setup_deflation()
            s.set_option("coarse_dense", dense)
            z, its = s.ras_apply(v, inner_tol=1e-3, inner_prec=prec)
            y, _ = s.ras_apply(v, inner_tol=1e-3, inner_prec=prec)
            stream.synchronize()
        assert torch.equal(y, z)
        if ref is None:
            ref = z, its
        assert torch.equal(z, ref[0]) and its == ref[1]
