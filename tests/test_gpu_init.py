"""The initial state, population by population, against the FP64 oracle on
grids where the pull pre-image can go wrong: extents below the stencil's
width, edges of copy axes (one node owns several destinations, or none),
ragged rows; and D3Q343's moments.

Tolerances: float storage 1e-5 of each population array's magnitude (float32
unit roundoff times a few tens of operations); 16-bit storage one unit in the
last place of the stored deviation on top of that (half an ulp of rounding,
plus float arithmetic that may cross a rounding boundary)."""
import numpy as np
import pytest

from paper_1606_06107_gb300 import workloads

pytestmark = pytest.mark.gpu

KIND = {"D1Q7": 1, "D2Q37": 2, "D2Q49": 3, "D3Q343": 4}
BC = {"periodic": 0, "copy": 1}
ULP = {"f32": 0.0, "f16": 2.0 ** -10, "bf16": 2.0 ** -7, "f16_node": 2.0 ** -10, "bf16_node": 2.0 ** -7}


def pair(orc, kind, shape, bc, n, storage="f32", mode="stream"):
    from paper_1606_06107_gb300 import Lbm
    wl = workloads.smooth_random(shape, seed=11, kind=kind, n=n, u_mean=[0.1] * len(shape))
    gpu = Lbm(kind, n, wl.tau, shape, bc, storage=storage, mode=mode)
    for b in (gpu.buf_a, gpu.buf_b):
        b.fill_(0xff)  # NaN bit patterns: a destination that nothing writes shows
    ref = orc.Sim(KIND[kind], n, wl.tau, shape, tuple(BC[b] for b in bc), mode=0 if mode == "stream" else 1)
    f32 = [np.asarray(v, np.float32).astype(np.float64) for v in (wl.rho, wl.u, wl.T)]
    gpu.set_macro(*f32)
    ref.set_macro(*f32)
    return gpu, ref


CASES = [("D1Q7", (s,), (b,), 4) for s in (1, 2, 5, 130) for b in BC]
CASES += [(k, s, b, n) for k in ("D2Q37", "D2Q49") for s in ((1, 2), (4, 7), (133, 5))
          for b in (("periodic", "copy"), ("copy", "periodic"), ("copy", "copy")) for n in (0, 3)]
CASES += [("D3Q343", s, b, n) for s in ((1, 2, 3), (9, 4, 7), (131, 3, 2))
          for b in (("periodic",) * 3, ("copy",) * 3, ("copy", "periodic", "copy")) for n in (0, 4)]


@pytest.mark.parametrize("kind,shape,bc,n", CASES)
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16_node"])
def test_initial_state(orc, kind, shape, bc, n, storage):
    if storage == "bf16_node" and kind == "D3Q343":
        pytest.skip("no per-node reference on D3Q343")
    gpu, ref = pair(orc, kind, shape, bc, n, storage)
    got = [x.cpu().numpy().astype(np.float64) for x in gpu.state()]
    want = ref.state()
    from paper_1606_06107_gb300 import lbm
    w = [lbm.lattice_info(kind)[2], lbm.lattice_info("D1Q7")[2]]
    for k in range(2 if n else 1):
        for i in range(got[k].shape[0]):
            scale = np.abs(want[k][i]).max()
            # |d| + |R - 1| of the stored deviation, both at most the departure
            # from rest of this node's value and of its reference
            dev = 2.0 * np.abs(want[k][i] / w[k][i] - 1.0).max() + 1.0 * (storage == "bf16_node")
            tol = 1e-5 * scale + ULP[storage] * w[k][i] * dev
            assert np.abs(got[k][i] - want[k][i]).max() <= tol, (k, i)


@pytest.mark.parametrize("shape,bc,n,storage", [((5, 4, 9), ("copy", "periodic", "copy"), 4, "f32"),
                                                ((131, 3, 2), ("periodic",) * 3, 0, "f16"),
                                                ((130, 4, 5), ("copy",) * 3, 4, "bf16")])
def test_d3q343_moments_are_those_of_its_state(shape, bc, n, storage, orc):
    """rho, u, T against FP64 sums over the decoded populations of the same
    state, gathered as the pull does; float32 sums of 343 values: 2e-6."""
    from paper_1606_06107_gb300 import lbm
    gpu, _ = pair(orc, "D3Q343", shape, bc, n, storage)
    gpu.step(1)
    f, h = (x.cpu().numpy().astype(np.float64) for x in gpu.state())
    r, e, _ = lbm.lattice_info("D3Q343")
    f = f.reshape((343,) + shape[::-1])
    g = np.empty_like(f)
    for i in range(343):
        v = f[i]
        for a in range(3):
            at = np.arange(shape[a]) - e[i][a]
            at = at % shape[a] if bc[a] == "periodic" else np.clip(at, 0, shape[a] - 1)
            v = np.take(v, at, axis=2 - a)
        g[i] = v
    g = g.reshape(343, -1)
    rho = g.sum(0)
    u = np.stack([r * (e[:, a, None] * g).sum(0) / rho for a in range(3)])
    energy = 0.5 * (r * r * ((e ** 2).sum(1)[:, None] * g).sum(0) / rho - (u ** 2).sum(0))
    if n:
        energy = energy + 0.5 * n * sum((r * (j - 3)) ** 2 * h[j] for j in range(7))
    T = energy / (0.5 * (3 + n))
    for got, want in zip(gpu.moments(), (rho, u, T)):
        got = got.cpu().numpy().astype(np.float64)
        assert np.abs(got - want).max() <= 2e-6 * np.abs(want).max()
