"""Ensembles around the sizes where the launch's shape changes (threads by the
longest problem and by the number of problems, a block per problem at most):
the same bits as single runs, and a status word for the failing problem only."""
import numpy as np
import pytest

from paper_1606_06107_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,longest", [(1, 1), (3, 33), (460, 40), (460, 256), (460, 257), (460, 512), (460, 513),
                                           (2000, 65)])
@pytest.mark.parametrize("block", [None, 1024])
def test_equals_single_runs(count, longest, block):
    from paper_1606_06107_gb300 import Lbm, LbmBatch
    rng = np.random.default_rng(longest)
    lengths = rng.integers(max(1, longest // 2), longest + 1, count)
    lengths[0] = longest
    n, tau = rng.choice([2, 4, 6, 7], count), rng.uniform(0.7, 1.0, count)
    wl = [workloads.smooth_random((int(L),), seed=int(L), kind="D1Q7", n=4, u_mean=[0.1]) for L in lengths]
    fields = [np.concatenate([np.asarray(getattr(w, f)).reshape(-1) for w in wl]) for f in ("rho", "u", "T")]
    bad = count // 2
    ens = LbmBatch(lengths, n, tau, mode="fd")
    if block:
        ens.set_block(block)
    fields[2][ens.offsets[bad]] = np.nan
    ens.set_macro(*fields)
    ens.run(5)
    got = [m.cpu().numpy() for m in ens.moments()]
    for k in sorted({0, 1 % count, count // 3, count - 1} - {bad}):
        sim = Lbm("D1Q7", int(n[k]), float(tau[k]), (int(lengths[k]),), ("copy",), mode="fd")
        sim.set_macro(wl[k].rho, wl[k].u, wl[k].T)
        sim.step(5)
        at = slice(ens.offsets[k], ens.offsets[k] + lengths[k])
        for a, b in zip(got, sim.moments()):
            assert np.array_equal(a[at], b.cpu().numpy().reshape(-1)), k
    words, failed = ens.status()
    assert failed == 1 and np.flatnonzero(np.asarray(words)).tolist() == [bad]
