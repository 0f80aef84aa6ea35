"""Contexts of different sizes in several host threads at once (one context per thread)."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_contexts_of_different_sizes_in_two_threads():
    """Set-up, a solve and a training gradient of a wide and of a narrow problem, repeated in two threads
    on streams of their own: the results each has alone, bit for bit."""
    torch = pytest.importorskip("torch")
    from paper_2103_17081_gb300 import Solver
    from paper_2103_17081_gb300.warmstart import init_params
    problems = [W.custom(40.0, 250, 1, 2, Sy=6), W.custom(30.0, 96, 2)]

    def job(w, stream):
        with torch.cuda.stream(stream):
            s = Solver(0).assemble(w.k, w.N).setup_dd(w.Sx, w.Sy, w.overlap).setup_deflation()
            f = torch.from_numpy(W.random_complex_fast(s.n, 3)).to("cuda")
            x, _ = s.solve(f, outer_tol=1e-12, outer_maxit=40, outer_restart=40, raise_on_error=False)
            s.cnn_set_params(init_params(s.cnn_num_params(), 2))
            loss, grad = s.cnn_loss_grad(s.local_op("R", f))
            stream.synchronize()
            s.close()
        return x.cpu().numpy(), loss, grad

    streams = [torch.cuda.Stream() for _ in problems]
    ref = [job(w, st) for w, st in zip(problems, streams)]
    out, err = [[] for _ in problems], []

    def run(q):
        try:
            for _ in range(5):
                out[q].append(job(problems[q], streams[q]))
        except Exception as e:                      # to the test's thread
            err.append(e)

    ts = [threading.Thread(target=run, args=(q,)) for q in range(len(problems))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not err, err
    for q, r in enumerate(ref):
        for x, loss, grad in out[q]:
            assert np.array_equal(x, r[0]) and loss == r[1] and np.array_equal(grad, r[2])
