"""Kernels launched while their predecessor on the stream is still running
(programmatic dependent launch): they are resident while that one writes what
they will read, so none of their loads may take the read-only path, which is
defined for data that nobody writes during the kernel's lifetime.  The sources
are checked for that, and queued steps against steps that are waited for one by
one."""
import glob
import os
import re

import pytest

from paper_1606_06107_gb300 import _build, workloads

# a function's name and the text from there to the closing brace in column 0
FUNCTION = re.compile(r"^(?:template[^\n]*\n)?(?:[^\n#/]*\n)?[^\n#/;]*?\b(\w+)\([^;{]*\)\n\{\n(.*?)^\}", re.S | re.M)
ONE_LINE = re.compile(r"^(?:template[^\n{]*> )?__device__[^\n{;]*?\b(\w+)\([^\n{;]*\)\s*\{([^\n]*)\}$", re.M)
READ_ONLY = re.compile(r"\b(__ldg|ld_ro)\(|\bld\(p\b|__restrict__|ld\.global\.nc")


def functions():
    found = {}
    for path in sorted(glob.glob(os.path.join(_build.CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*|__launch_bounds__\([^)]*\)", "", f.read())
        for pattern in (FUNCTION, ONE_LINE):
            for name, body in pattern.findall(text):
                found.setdefault((os.path.basename(path), name), []).append(body)
    return found


def test_no_read_only_loads():
    found = functions()
    waiting = {k for k, bodies in found.items()
               if any(re.search(r"\bpdl_(wait|chain)\(\)", b) for b in bodies)}
    assert {n for _, n in waiting} >= {"k_step", "k_step_node", "k_tube_step", "k_conv_tcn", "k_conv_tcp", "k_wgrad_tc",
                                       "k_lift", "k_head", "k_head_bwd", "k_lift_bwd", "k_colsum8", "k_mse",
                                       "k_features", "k_targets", "k_apply"}
    # what these call, function by function; `ld` itself has both paths, and
    # which one a call takes is its first template argument
    seen, todo = set(), set(waiting)
    while todo:
        file, name = todo.pop()
        seen.add((file, name))
        for body in found[(file, name)]:
            m = READ_ONLY.search(body)
            assert not m, f"{file}: {name}: {m.group(0)}"
            for call, args in re.findall(r"\b(load_node|rot_advect)<([^>]*)>", body):
                assert args.split(",")[-1].strip() in ("true", "LATE"), f"{file}: {name}: {call}<{args}>"
            for other in found:
                same = other[0] == file or not file.startswith("nn_")
                if same and other[1] not in ("ld", "ld_ro") and other not in seen \
                        and re.search(r"\b%s\b" % other[1], body):
                    todo.add(other)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,shape,storage,mode", [
    ("D1Q7", (9001,), "f32", "fd"), ("D1Q7", (700,), "f16", "stream"), ("D2Q37", (1000, 16), "f32", "stream"),
    ("D2Q49", (257, 130), "bf16", "stream"), ("D2Q49", (257, 130), "f16_node", "stream"),
    ("D2Q37", (129, 40), "f32", "fd"), ("D2Q37", (513, 200), "f32", "fd"), ("D3Q343", (20, 9, 8), "f16", "stream")])
def test_queued_steps_equal_single_ones(kind, shape, storage, mode):
    import torch
    from paper_1606_06107_gb300 import Lbm
    wl = workloads.smooth_random(shape, seed=9, kind=kind, n=3)
    sims = [Lbm(kind, 3, wl.tau, shape, wl.bc, storage=storage, mode=mode) for _ in range(2)]
    for s in sims:
        s.set_macro(wl.rho, wl.u, wl.T)
    sims[0].step(24)
    for _ in range(24):
        sims[1].step(1)
        torch.cuda.synchronize()
    for x, y in zip(sims[0].state(), sims[1].state()):
        assert torch.equal(x, y)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,shape,bc,init", [("D2Q37", (20, 10), ("copy", "copy"), 1), ("D3Q343", (9, 8, 7), ("periodic",) * 3, 1),
                                                ("D3Q343", (9, 8, 7), ("periodic", "periodic", "copy"), 2)])
def test_launch_count(kind, shape, bc, init):
    from paper_1606_06107_gb300 import Lbm
    wl = workloads.smooth_random(shape, seed=2, kind=kind, n=3)
    sim = Lbm(kind, 3, wl.tau, shape, bc)
    at = sim.launches
    sim.set_macro(wl.rho, wl.u, wl.T)
    assert sim.launches - at == init
    sim.step(3)
    assert sim.launches - at == init + 3
