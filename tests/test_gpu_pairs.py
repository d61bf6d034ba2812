"""Kernels that take two x-adjacent nodes a thread (16-bit storage), at the rows
where their blocks, last pairs and boundaries differ."""
import numpy as np
import pytest

import test_gpu_d3q343 as d3q343
from paper_1606_06107_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("X", [63, 64, 65, 128, 129, 193])
@pytest.mark.parametrize("bc", [("periodic",) * 3, ("copy", "periodic", "copy")])
def test_d3q343_step_by_row_length(orc, storage, X, bc):
    """Rows of one, two, three and four warps of pairs (blocks of one warp or
    of two), whole and ragged, against the oracle as in the test it calls."""
    d3q343.test_one_step_per_population_16bit(orc, storage, (X, 3, 2), bc, 4)


@pytest.mark.parametrize("kind", ["D2Q37", "D2Q49"])
@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("shape", [(131, 5), (130, 6), (1, 2), (2, 3), (3, 4), (257, 3)])
@pytest.mark.parametrize("bc", [("periodic", "copy"), ("copy", "periodic"), ("copy", "copy")])
@pytest.mark.parametrize("n", [0, 3])
def test_moments_2d_are_those_of_the_state(kind, storage, shape, bc, n):
    """rho, u, T against FP64 sums over the decoded populations of the same
    state, gathered as the pull does.  A float32 sum of 49 terms t is off by at
    most 49 2^-24 sum |t| = 3e-6 sum |t|: sum f = rho, r sum |e_a| f <= 1.2 rho,
    and T's energy sums are at most three times T's share of them."""
    from paper_1606_06107_gb300 import Lbm, lbm
    wl = workloads.smooth_random(shape, seed=21, kind=kind, n=n, u_mean=[0.1, -0.05])
    sim = Lbm(kind, n, wl.tau, shape, bc, storage=storage)
    sim.set_macro(wl.rho, wl.u, wl.T)
    sim.step(1)
    f, h = (x.cpu().numpy().astype(np.float64) for x in sim.state())
    r, e, _ = lbm.lattice_info(kind)
    g = f.reshape((len(e),) + shape[::-1]).copy()
    for i in range(len(e)):
        for a in range(2):
            at = np.arange(shape[a]) - e[i][a]
            at = at % shape[a] if bc[a] == "periodic" else np.clip(at, 0, shape[a] - 1)
            g[i] = np.take(g[i], at, axis=1 - a)
    g = g.reshape(len(e), -1)
    rho = g.sum(0)
    u = np.stack([r * (e[:, a, None] * g).sum(0) / rho for a in range(2)])
    energy = 0.5 * (r * r * ((e ** 2).sum(1)[:, None] * g).sum(0) / rho - (u ** 2).sum(0))
    if n:
        energy = energy + 0.5 * n * sum((r * (j - 3)) ** 2 * h[j].reshape(-1) for j in range(7))
    T = energy / (0.5 * (2 + n))
    got = [x.cpu().numpy().astype(np.float64).reshape(w.shape) for x, w in zip(sim.moments(), (rho, u, T))]
    for a, b, tol in zip(got, (rho, u, T), (3e-6, 4e-6, 1e-5)):
        assert np.abs(a - b).max() <= tol * rho.max(), np.abs(a - b).max()


@pytest.mark.parametrize("n", [0, 4])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_d3q343_moments_at_rest(n, storage):
    """Opposite velocities are combined before anything else: a uniform state at
    rest has exactly no momentum."""
    from paper_1606_06107_gb300 import Lbm
    shape = (70, 4, 3)
    N = int(np.prod(shape))
    for rho, T in ((1.1, 0.9), (0.7, 1.3), (1.0, 1.01)):
        sim = Lbm("D3Q343", n, 0.8, shape, ("periodic",) * 3, storage=storage)
        sim.set_macro(np.full(N, rho), np.zeros((3, N)), np.full(N, T))
        assert not sim.moments()[1].cpu().numpy().any()
