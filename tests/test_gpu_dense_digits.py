"""The product by digits where it is sure to have run (the FP64 product of small orders reports under the
same name): remainders of its tiles, and batches that split its work differently."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _apply(s, v, **kw):
    """(z, steps, kernels per coarse product): three by digits, one in FP64, none banded."""
    s.profile(True)                    # (clears the counts)
    before = s.launch_count()
    z, its = s.ras_apply(v, **kw)
    stats = s.profile_stats()
    extra = s.launch_count() - before - sum(d["launches"] for d in stats)
    s.profile(False)
    products = sum(d["launches"] for d in stats if d["name"] == "coarse_solve_dense")
    return z, its, 1 + extra // products if products else 0


def _solver(w, nrhs):
    from paper_2103_17081_gb300 import Solver
    return Solver(0).assemble(w.k, w.N, bc=w.bc).setup_dd(w.Sx, w.Sy, w.overlap, w.ifx, w.ify).setup_batch(nrhs).setup_deflation()


# orders 4·128 + 113 = 39·16 + 1; 256, whole tiles; 289 complex = 2·128 + 33; 32, 96 and 20 columns a shape
CASES = {"m625": (W.custom(40.0, 100, 2, 2), 4), "m256": (W.custom(30.0, 64, 2, 2), 12), "m289_complex": (W.custom(30.0, 66, 2, 2, bc=1), 10)}


@pytest.mark.parametrize("name", CASES)
def test_digits_match_banded(name):
    """complex128, κ(E)·2^-53 in either form: 1e-11, the bar of test_gpu_dense.py."""
    torch = pytest.importorskip("torch")
    w, nrhs = CASES[name]
    s = _solver(w, nrhs)
    v = torch.from_numpy(W.random_complex_fast(nrhs * s.n, 7)).cuda()
    opt = dict(inner_tol=1e-4, inner_prec=128)
    z, its, form = _apply(s, v, **opt)
    assert form == 3
    s.set_option("coarse_dense", 0)
    zb, itb, form = _apply(s, v, **opt)
    assert form == 0 and its == itb
    assert float(torch.linalg.vector_norm(z - zb)) <= 1e-11 * float(torch.linalg.vector_norm(zb))


def test_digits_of_a_batch_and_of_its_halves():
    """The same right-hand sides as one batch and as two, by digits both times: the integer sums agree up
    to the rounding of the two last ones in every part of a tile (2^-60 of a full product), so 1e-14."""
    torch = pytest.importorskip("torch")
    w = W.custom(40.0, 129, 2, 1)
    whole, half = _solver(w, 12), _solver(w, 6)
    v = torch.from_numpy(W.random_complex_fast(12 * whole.n, 11)).cuda()
    opt = dict(inner_tol=1e-3, inner_prec=128)
    z, its, form = _apply(whole, v, **opt)
    assert form == 3
    again, _, _ = _apply(whole, v, **opt)
    assert torch.equal(z, again)
    for q in (0, 1):
        part = v[q * 6 * half.n:(q + 1) * 6 * half.n].clone()
        zh, ith, form = _apply(half, part, **opt)
        assert form == 3
        assert ith == its[q * 6 * half.nsub:(q + 1) * 6 * half.nsub]
        ref = z[q * 6 * half.n:(q + 1) * 6 * half.n]
        assert float(torch.linalg.vector_norm(zh - ref)) <= 1e-14 * float(torch.linalg.vector_norm(ref))
