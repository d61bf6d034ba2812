"""Many steps of one tube in one launch: the same bits as one launch per step,
at the sizes where the pieces, halos and block sizes change; and steps
captured in a CUDA graph."""
import numpy as np
import pytest

from paper_1606_06107_gb300 import workloads

pytestmark = pytest.mark.gpu


def tube(X, bc, mode, n):
    from paper_1606_06107_gb300 import Lbm
    wl = workloads.smooth_random((X,), seed=X, kind="D1Q7", n=n, u_mean=[0.1])
    sim = Lbm("D1Q7", n, 0.8, (X,), (bc,), mode=mode)
    sim.set_macro(wl.rho, wl.u, wl.T)
    return sim


@pytest.mark.parametrize("X", [5, 31, 32, 33, 64, 95, 257, 1000, 2048, 2049, 8192, 8193])
@pytest.mark.parametrize("bc", ["periodic", "copy"])
@pytest.mark.parametrize("mode,n", [("stream", 0), ("stream", 4), ("fd", 0), ("fd", 4)])
def test_one_launch_equals_single_steps(X, bc, mode, n):
    import torch
    a, b = tube(X, bc, mode, n), tube(X, bc, mode, n)
    for steps in (4, 7):
        a.step(steps)
        for _ in range(steps):
            b.step(1)
        for x, y in zip((*a.state(), *a.moments()), (*b.state(), *b.moments())):
            assert torch.equal(x, y)
    assert a.steps == b.steps == 11 and a.status() == b.status() == 0
    if 32 <= X <= 8192:
        assert a.launches < b.launches


@pytest.mark.parametrize("at", [0, 499, 999])
def test_status_of_a_failing_node(at):
    sim = tube(1000, "copy", "fd", 4)
    ft, fr = sim.state()
    ft[:, at] = float("nan")
    sim.set_state(ft, fr)
    sim.step(8)
    assert sim.status() == -4


@pytest.mark.parametrize("kind,shape,storage", [("D1Q7", (300,), "f32"), ("D2Q49", (70, 9), "f32"),
                                                ("D2Q37", (70, 9), "f16"), ("D2Q49", (64, 5), "bf16_node"),
                                                ("D3Q343", (20, 5, 4), "f16")])
def test_captured_steps(kind, shape, storage):
    """Six steps replayed from a graph equal six steps launched directly."""
    import torch
    from paper_1606_06107_gb300 import Lbm
    wl = workloads.smooth_random(shape, seed=3, kind=kind, n=3)
    stream = torch.cuda.Stream()
    sims = [Lbm(kind, 3, wl.tau, shape, wl.bc, storage=storage, stream=stream) for _ in range(2)]
    with torch.cuda.stream(stream):
        for s in sims:
            s.set_macro(wl.rho, wl.u, wl.T)
            s.step(4)  # kernel attributes are set before the capture
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            sims[0].step(6)
        g.replay()
        sims[1].step(6)
        torch.cuda.synchronize()
        for x, y in zip(sims[0].moments(), sims[1].moments()):
            assert bool(torch.isfinite(x).all()) and torch.equal(x, y)


@pytest.mark.parametrize("mode", ["fd", "stream"])
@pytest.mark.parametrize("block", [32, 96, 512, 1024])
def test_windowed_ensemble_equals_single_runs(mode, block):
    """Tubes around the window's size and several windows long, for step
    counts around a pass and of both parities, with a block of one warp and
    of more threads than a short tube has nodes."""
    from paper_1606_06107_gb300 import Lbm, LbmBatch
    lengths = [1, 2, 3, 63, 895, 896, 897, 1337, 1745, 5000]
    ns = [0, 2, 4, 6, 7, 2, 4, 6, 7, 4]
    wl = [workloads.smooth_random((L,), seed=L, kind="D1Q7", n=4, u_mean=[0.1]) for L in lengths]
    cat = [np.concatenate([np.asarray(getattr(w, f)).reshape(-1) for w in wl]) for f in ("rho", "u", "T")]
    ens = LbmBatch(lengths, ns, [0.8] * len(lengths), mode=mode)
    ens.set_block(block)
    sims = [Lbm("D1Q7", n, 0.8, (L,), ("copy",), mode=mode) for L, n in zip(lengths, ns)]
    for steps in ([1, 2, 7, 8], [9, 16], [33]):
        ens.set_macro(*cat)
        for s, w in zip(sims, wl):
            s.set_macro(w.rho, w.u, w.T)
        for k in steps:
            ens.run(k)
            for s in sims:
                s.step(k)
        got = [x.cpu().numpy() for x in ens.moments()]
        for k, s in enumerate(sims):
            sl = slice(ens.offsets[k], ens.offsets[k] + lengths[k])
            for a, b in zip(got, s.moments()):
                assert np.array_equal(a[sl], b.cpu().numpy().reshape(-1)), (k, steps)
    assert ens.status()[1] == 0
