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


def test_a_solve_that_needs_the_inverses_memory_runs_without_them():
    """A solve whose Krylov basis fits the free memory only together with half of what the inverses
    hold: it runs with the banded kernels, to the result it has with them from the start."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver

    def solver():
        return Solver(0).assemble(100.0, 320).setup_dd(4, 4, 2)

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    twin = solver()
    before = free()
    twin.set_option("coarse_dense", 0).setup_deflation()
    banded = before - free()
    f = torch.from_numpy(W.random_complex_fast(twin.n, 8)).cuda()
    x, opt = twin.empty(), dict(outer_maxit=60, outer_restart=60, outer_tol=1e-10, raise_on_error=False)
    before = free()
    _, st = twin.solve(f, out=x, **opt)
    need = before - free()
    twin.close()
    s = solver()
    before = free()
    s.setup_deflation()
    held = before - free() - banded
    assert held > 40 << 20 and need > 200 << 20
    y = s.empty()
    s.profile(True)
    rest = _fill(torch, need - held // 2)
    try:
        _, st2 = s.solve(f, out=y, **opt)
    finally:
        del rest
        torch.cuda.empty_cache()
    assert "coarse_solve_dense" not in {d["name"] for d in s.profile_stats() if d["launches"]}
    assert st2["status_code"] == st["status_code"] and st2["outer_its"] == st["outer_its"]
    assert torch.equal(x, y)
