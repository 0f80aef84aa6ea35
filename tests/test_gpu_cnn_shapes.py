"""The training kernels' forward and backward passes on boxes at the edges of their tilings."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    # 249 nodes wide: strips of fewer rows than a tile has, several chunks of 128 pixels per row
    "wide": W.custom(40.0, 250, 1, 2, Sy=14),
    # 7 and 9 nodes: fewer pixels than a chunk, empty stretches of a row
    "narrow": W.custom(6.0, 16, 2, 1, Sy=3, ifx=[0, 7, 16]),
    # tiles whose last one is short, widths next to a multiple of 32
    "ragged": W.custom(20.0, 66, 2, 2, Sy=3, ifx=[0, 30, 66]),
}


@pytest.mark.parametrize("name", CASES)
def test_loss_and_gradient_match_oracle(name):
    """Loss and every layer's gradient against the FP64 oracle: bars of the training path's parity
    test (FP32 sums of at most 288 terms per activation, FP32 projections around FP64 coarse solves)."""
    torch = pytest.importorskip("torch")
    import oracle
    from oracle import cnn
    from paper_2103_17081_gb300 import Solver
    from paper_2103_17081_gb300.warmstart import init_params
    from test_oracle_cnn import projections
    w = CASES[name]
    s = Solver.from_workload(w)
    p = oracle.from_workload(w)
    params = init_params(s.cnn_num_params(), seed=5)
    params[cnn.offsets()[3]:] *= 10.0
    s.cnn_set_params(params)
    fo, _ = s.offsets()
    f = W.random_complex_fast(fo[-1], 13)
    batch = [(f[fo[t]:fo[t + 1]], (p.box(t)["ny"], p.box(t)["nx"]), p.sub_A(t)) + projections(p, t) for t in range(p.nsub)]
    kh = w.k / w.N
    L, g = s.cnn_loss_grad(torch.from_numpy(f).cuda())
    Lr, gr = cnn.loss_and_grad(cnn.bf16_round(params), batch, kh)
    assert L == pytest.approx(Lr, rel=1e-4)
    off = cnn.offsets()
    for l in range(4):
        a, b = g[off[l]:off[l + 1]], gr[off[l]:off[l + 1]]
        assert np.linalg.norm(a - b) <= 2e-3 * np.linalg.norm(b), l
