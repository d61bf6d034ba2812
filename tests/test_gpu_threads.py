"""A host thread per handle, sizes that differ: the limit of dynamic shared
memory belongs to the kernel, so no thread's launch may take it below what
another's needs."""
import threading

import pytest

from paper_1606_06107_gb300 import workloads

pytestmark = pytest.mark.gpu


def run_together(rounds, *work):
    start, errors = threading.Barrier(len(work)), []

    def body(f):
        try:
            start.wait()
            for _ in range(rounds):
                f()
        except Exception as e:  # noqa: BLE001 (any failure of a call)
            errors.append(e)

    threads = [threading.Thread(target=body, args=(f,)) for f in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    import torch
    torch.cuda.synchronize()
    assert not errors, errors


def test_tubes_of_several_lengths():
    import torch
    from paper_1606_06107_gb300 import Lbm
    rounds, sims = 20000, []
    for X in (8192, 4000, 7000, 3500):
        wl = workloads.smooth_random((X,), seed=X, kind="D1Q7", n=4)
        sims.append(Lbm("D1Q7", 4, 0.8, (X,), ("copy",), mode="fd", stream=torch.cuda.Stream()))
        sims[-1].set_macro(wl.rho, wl.u, wl.T)
    torch.cuda.synchronize()
    run_together(rounds, *[lambda s=s: s.step(4) for s in sims])
    assert all(s.steps == 4 * rounds and s.status() == 0 for s in sims)


def test_lift_backward_of_two_widths(lbmlib):
    import torch
    P, F, rounds = 64, 16, 3000

    def call(C):
        g, feat = torch.ones(P, C, device="cuda"), torch.ones(P, F, device="cuda")
        gW, gb, stream = torch.zeros(C, F, device="cuda"), torch.zeros(C, device="cuda"), torch.cuda.Stream()

        def f():
            rc = lbmlib.lbm_nn_lift_backward(g.data_ptr(), feat.data_ptr(), gW.data_ptr(), gb.data_ptr(), P, F, C,
                                             stream.cuda_stream)
            assert rc == 0, rc
        f.sums = (gW, gb)
        return f

    calls = [call(1024), call(768)]
    torch.cuda.synchronize()
    run_together(rounds, *calls)
    for f in calls:
        assert all(bool((t == P * rounds).all()) for t in f.sums)
