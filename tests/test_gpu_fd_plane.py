"""Finite-difference transport on planes around one wave of blocks, where the
step changes from the four-blocks-per-SM kernel to the three-block one: one
step from the same float32 state, population by population, within 1e-5 of
each population array's magnitude of the FP64 oracle (float32 unit roundoff
times a few tens of operations)."""
import numpy as np
import pytest

from paper_1606_06107_gb300 import workloads

pytestmark = pytest.mark.gpu

KIND = {"D2Q37": 2, "D2Q49": 3}


@pytest.mark.parametrize("kind", ["D2Q37", "D2Q49"])
@pytest.mark.parametrize("shape", [(129, 304), (129, 305), (1, 700), (300, 230)])
@pytest.mark.parametrize("bc,n", [(("copy", "copy"), 3), (("periodic", "copy"), 0)])
def test_one_step(orc, kind, shape, bc, n):
    from paper_1606_06107_gb300 import Lbm
    wl = workloads.smooth_random(shape, seed=5, kind=kind, n=n, u_mean=[0.1, -0.1])
    gpu = Lbm(kind, n, wl.tau, shape, bc, mode="fd")
    ref = orc.Sim(KIND[kind], n, wl.tau, shape, tuple({"periodic": 0, "copy": 1}[b] for b in bc), mode=1)
    ref.set_macro(wl.rho, wl.u, wl.T)
    ft, fr = (x.astype(np.float32) for x in ref.state())
    ref.set_state(ft.astype(np.float64), fr.astype(np.float64) if n else None)
    gpu.set_state(ft, fr if n else None)
    gpu.step(1)
    ref.step(1)
    for got, want in zip(gpu.state(), ref.state()):
        got = got.cpu().numpy().astype(np.float64)
        for i in range(got.shape[0]):
            assert np.abs(got[i] - want[i]).max() <= 1e-5 * np.abs(want[i]).max(), i
