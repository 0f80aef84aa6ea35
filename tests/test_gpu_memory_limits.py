"""Calls next to the end of the device's memory: the coarse inverses and their plans are an option that
costs no call its memory."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _fill(torch, leave):
    """A tensor over all of the device's free memory but `leave` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


def test_no_room_for_the_products_plan_takes_the_banded_kernels():
    """64 right-hand sides on 16 boxes: a plan of more than 60 MB (right-hand sides' digits and sums) where
    20 MB are left; the banded kernels' result, bit for bit, and the products again when there is room."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    s = Solver(0).assemble(100.0, 320).setup_dd(4, 4, 2).setup_batch(64).setup_deflation()
    v = torch.from_numpy(W.random_complex_fast(64 * s.n, 5)).cuda()
    z = s.empty(64 * s.n)
    opt = dict(out=z, inner_tol=1e-2, inner_prec=64)

    def families():
        return {d["name"] for d in s.profile_stats() if d["launches"]}

    s.set_option("coarse_dense", 0)
    s.ras_apply(v, **opt)
    ref = z.clone()
    s.set_option("coarse_dense", 1)
    s.profile(True)
    rest = _fill(torch, 20 << 20)
    try:
        s.ras_apply(v, **opt)
    finally:
        del rest
        torch.cuda.empty_cache()
    assert "coarse_solve_dense" not in families()
    assert torch.equal(z, ref)
    s.profile(True)
    s.ras_apply(v, **opt)
    assert "coarse_solve_dense" in families()
    s.profile(False)
    assert float(torch.linalg.vector_norm(z - ref)) <= 1e-4 * float(torch.linalg.vector_norm(ref))
