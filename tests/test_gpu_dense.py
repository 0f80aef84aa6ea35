"""The inner iteration's coarse solves as products with explicit inverses (kernels_dense.cu) against
the banded kernels they replace and the oracle."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


# (workload, right-hand sides): order of E next to a multiple of 128 rows and 16 columns on both
# sides, one and two column tiles per shape, several shapes, complex E
CASES = {
    "m625": (W.custom(40.0, 100, 2, 2), 1),                                  # 25 x 25: 4·128 + 113, 39·16 + 1
    "m1024_two_column_tiles": (W.custom(40.0, 129, 2, 1), 12),                # 32 x 32, 24 or 48 columns
    "m_ragged": (W.custom(50.0, 150, 3, 2, Sy=2, ifx=[0, 48, 99, 150]), 3),   # six shapes
    "many_columns": (W.custom(45.0, 108, 2, 2), 41),                          # 82 columns per shape
    "wide_box": (W.custom(60.0, 190, 1, 2, Sy=2), 2),                         # 189 nodes wide, m = 94 x 48
    "impedance": (W.custom(30.0, 96, 2, 2, bc=1), 2),                         # 24 x 24 complex
    "impedance_ragged": (W.custom(35.0, 110, 3, 2, Sy=2, ifx=[0, 34, 74, 110], bc=1), 5),
}


def _solver(w, nrhs):
    from paper_2103_17081_gb300 import Solver
    s = Solver(0).assemble(w.k, w.N, bc=w.bc).setup_dd(w.Sx, w.Sy, w.overlap, w.ifx, w.ify)
    if nrhs > 1:
        s.setup_batch(nrhs)
    return s.setup_deflation()


def _launched(s):
    return {d["name"]: d["launches"] for d in s.profile_stats() if d["launches"]}


def _vectors(s, seed, holes=False):
    """Random vectors; with holes, zero over the lower left quarter and the last vector zero
    everywhere (tasks that are done at the start)."""
    import torch
    v = W.random_complex_fast(s.nrhs * s.n, seed).reshape(s.nrhs, -1)
    if holes:
        side = int(round(s.n ** 0.5))
        v = v.reshape(s.nrhs, side, side)
        v[:, : 2 * side // 3, : 2 * side // 3] = 0.0
        if s.nrhs > 1:
            v[-1] = 0.0
    v = v.reshape(-1) / np.linalg.norm(v)
    return torch.from_numpy(np.ascontiguousarray(v)).to("cuda")


@pytest.mark.parametrize("prec", [128, 64])
@pytest.mark.parametrize("name", CASES)
def test_dense_coarse_solves_match_banded(name, prec):
    """RAS applications with both forms.  complex128: E⁻¹ of both carries κ(E)·2^-53 (bar 1e-11 as for
    the operator itself) and the same stopping decisions.  complex64: the fine arithmetic's 2^-24
    amplified by the deflated operator (1e-4 bar of that precision's RAS applications)."""
    w, nrhs = CASES[name]
    s = _solver(w, nrhs)
    for holes in (False, True):
        v = _vectors(s, 7, holes)
        out = {}
        for dense in (0, 1):
            s.set_option("coarse_dense", dense).profile(True)
            z, its = s.ras_apply(v, inner_tol=1e-4 if prec == 128 else 1e-2, inner_prec=prec)
            fam = _launched(s)
            s.profile(False)
            assert ("coarse_solve_dense" in fam) == bool(dense), fam
            assert sum(f.startswith("coarse_solve") for f in fam) >= 1
            out[dense] = (z.cpu().numpy(), its)
        assert np.isfinite(out[1][0]).all()
        if prec == 128:
            assert out[0][1] == out[1][1]
            assert _rel(out[1][0], out[0][0]) <= 1e-11
        else:
            assert _rel(out[1][0], out[0][0]) <= 1e-4


def test_dense_form_repeats_bitwise_and_per_right_hand_side():
    """Integer sums: the same bits whatever the split of the work, so a batch gives each right-hand
    side the result it has alone, and repeated calls agree."""
    w, _ = CASES["m1024_two_column_tiles"]
    s1, sb = _solver(w, 1), _solver(w, 12)
    v = _vectors(sb, 11)
    zb, itb = sb.ras_apply(v, inner_tol=1e-3, inner_prec=128)
    z2, it2 = sb.ras_apply(v, inner_tol=1e-3, inner_prec=128)
    assert bool((zb == z2).all()) and itb == it2
    for r in (0, 5, 11):
        s1.profile(True)
        z1, it1 = s1.ras_apply(v[r * s1.n:(r + 1) * s1.n].clone(), inner_tol=1e-3, inner_prec=128)
        assert "coarse_solve_dense" in _launched(s1)
        s1.profile(False)
        assert it1 == itb[r * s1.nsub:(r + 1) * s1.nsub]
        assert _rel(z1.cpu().numpy(), zb[r * s1.n:(r + 1) * s1.n].cpu().numpy()) <= 1e-14


def test_dense_warm_start_and_batch_change():
    """The doubled task table of the warm start (two coarse solves per task in one product), and a
    batch set up after the factors."""
    from paper_2103_17081_gb300 import warmstart
    w = W.custom(40.0, 128, 2, 2)
    s = _solver(w, 1).setup_batch(3)
    s.cnn_set_params(warmstart.init_params(s.cnn_num_params(), 3))
    v = _vectors(s, 5)
    out = {}
    for dense in (0, 1):
        s.set_option("coarse_dense", dense).profile(True)
        out[dense] = s.ras_apply(v, inner_tol=1e-6, inner_prec=128, warm_start=1)[0].cpu().numpy()
        assert ("coarse_solve_dense" in _launched(s)) == bool(dense)
        s.profile(False)
    # both reach 1e-6 of the deflated residual from the same guess: equal steps, κ(E)·2^-53 apart
    assert _rel(out[1], out[0]) <= 1e-11
