"""Kernels that start before the one in front has ended wait for what they read: results on a side
stream, behind and in front of other work and with tasks that stop at different steps, are bitwise
those of a run with a synchronisation after every call."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,k,N,S,nrhs,two", [(64, 40.0, 96, 3, 1, 0), (128, 17.0, 45, 3, 3, 0), (64, 60.0, 120, 4, 2, 1)])
def test_chained_launches_give_the_synchronised_results(prec, k, N, S, nrhs, two):
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    w = W.custom(k, N, S)
    s = Solver.from_workload(w, deflation=False)
    if nrhs > 1:
        s.setup_batch(nrhs)
    s.setup_deflation()
    if two:
        s.setup_coarse_grid(2)
    base = torch.from_numpy(W.random_complex_fast(s.n * nrhs, 9)).cuda()
    opt = dict(inner_prec=prec, inner_tol=1e-3, inner_restart=4)
    ref = []
    for q in range(6):
        v = base * (1.0 + q)
        torch.cuda.synchronize()
        z, _ = s.ras_apply(v, **opt)
        torch.cuda.synchronize()
        ref.append(s.apply_A(z).clone())
        torch.cuda.synchronize()
    solve = dict(inner_prec=prec, outer_tol=1e-3, outer_maxit=12, outer_restart=12, raise_on_error=False, two_level=two,
                 outer_reorth32=int(prec == 64))
    xr, st = s.solve(base, **solve)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for rep in range(3):
            for q in range(6):
                v = base * (1.0 + q)                      # on the same stream just before
                z, _ = s.ras_apply(v, **opt)
                v.zero_()                                 # and just behind
                y = s.apply_A(z)
                z.zero_()
                assert torch.equal(y, ref[q]), (rep, q)
            x, st2 = s.solve(base, **solve)
            assert st2["outer_its"] == st["outer_its"] and torch.equal(x, xr)
