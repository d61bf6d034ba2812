"""The work that a user of this framework has it do, as cases that can be timed and compared.

Every case goes through the package's public entry points (``Lbm``,
``LbmBatch``, ``ConvOperator``) as a user's program calls them:

- a flow case starts a solver from macroscopic fields, advances it and reads
  the fields back (``set_macro``, ``step``, ``moments``) -- the restarted
  cycle that the surrogate's training data, its fallback and the end-to-end
  benchmark run;
- an ensemble case does the same for many 1-D tubes at once (``set_macro``,
  ``run``, ``moments``);
- a surrogate case is one network call: a prediction, or the loss and the
  gradients of one training minibatch.

The solvers, their buffers and the network's weights are made once
(``prepare``), as such a program does; the fields are the inputs.
"""
import math

import numpy as np
import torch

from paper_1606_06107_gb300 import Lbm, LbmBatch
from paper_1606_06107_gb300.surrogate import ConvOperator

DIM = {"D1Q7": 1, "D2Q37": 2, "D2Q49": 2, "D3Q343": 3}
Q = {"D1Q7": 7, "D2Q37": 37, "D2Q49": 49, "D3Q343": 343}
TAU = 2.0 / 3.0   # relaxation time of the paper's run and of the benchmark
M_FD = 10         # sub-steps of the finite-difference transport (the default)
L2_BYTES = 129e6  # states larger than this have to pass through HBM every step


def listed():
    flow = dict(kind="flow", z=1, n=3, mode="stream", storage="f32", bcx="periodic", bcy="periodic", bcz="periodic")
    return [
        # Sod's shock tube, the README's first example: 1000 nodes, so a step
        # is a launch and little else.
        dict(flow, name="tube_1d_fd", lattice="D1Q7", x=1000, y=1, n=4, mode="fd", bcx="copy", steps=200),
        # The paper's own validation run: 1000 x 16 on D2Q37, open ends.
        dict(flow, name="paper_tube_2d", lattice="D2Q37", x=1000, y=16, bcx="copy", steps=30),
        # The benchmark's main workload: 2048^2 on D2Q49, float storage.
        dict(flow, name="plane_f32_2048", lattice="D2Q49", x=2048, y=2048, steps=20),
        # The same plane in half-precision deviations from rest (half the bytes).
        dict(flow, name="plane_f16_2048", lattice="D2Q49", x=2048, y=2048, storage="f16", steps=10),
        # Per-node reference storage on a ragged grid with open ends in x.
        dict(flow, name="plane_bf16_node_ragged", lattice="D2Q49", x=1021, y=771, storage="bf16_node", bcx="copy", steps=10),
        # The paper-literal finite-difference transport in two dimensions.
        dict(flow, name="plane_fd_d2q37", lattice="D2Q37", x=600, y=420, mode="fd", bcx="copy", bcy="copy", steps=20),
        # The 3-D blast, half-precision deviations, translational only.
        dict(flow, name="blast_f16_256", lattice="D3Q343", x=256, y=256, z=256, n=0, storage="f16", steps=4),
        # The same lattice with rotation, float storage, odd extents, open in z.
        dict(flow, name="blast_f32_ragged", lattice="D3Q343", x=101, y=96, z=90, n=4, bcz="copy", steps=4),
        # An ensemble of uneven tubes, 256 to 8192 nodes, advanced by one launch.
        dict(kind="ensemble", name="ensemble_mixed", count=1024, lmin=256, lmax=8192, mode="fd", steps=50),
        # The surrogate's spot check: one short window per tube, restarted every 32 steps.
        dict(kind="ensemble", name="ensemble_windows", count=1024, lmin=384, lmax=384, mode="fd", steps=32),
        # The surrogate's inference call at the benchmark's size.
        dict(kind="predict", name="surrogate_predict", tubes=1024, length=4096, patch=4),
        # One training minibatch of the surrogate: loss and every gradient.
        dict(kind="train", name="surrogate_train", tubes=32, length=4096, patch=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "plane", "plane", "plane", "fd", "blast", "blast", "ensemble", "ensemble", "predict", "train"])
    bc = lambda: rng.choice(["periodic", "copy"])  # noqa: E731
    flow = dict(kind="flow", y=1, z=1, n=3, mode="stream", storage="f32", bcx="periodic", bcy="periodic", bcz="periodic")
    if kind == "tube":
        return dict(flow, lattice="D1Q7", x=_log(rng, 50, 8000), n=rng.choice([2, 4, 6]), mode="fd", bcx="copy",
                    steps=_log(rng, 20, 400))
    if kind == "plane":
        return dict(flow, lattice=rng.choice(["D2Q37", "D2Q49"]), x=_log(rng, 40, 2048), y=_log(rng, 16, 2048),
                    n=rng.choice([0, 3, 3]), storage=rng.choice(["f32", "f32", "f16", "bf16", "f16_node", "bf16_node"]),
                    bcx=bc(), bcy=bc(), steps=rng.randint(4, 10))
    if kind == "fd":
        return dict(flow, lattice=rng.choice(["D2Q37", "D2Q49"]), x=_log(rng, 40, 1000), y=_log(rng, 16, 1000), mode="fd",
                    bcx=bc(), bcy=bc(), steps=rng.randint(5, 20))
    if kind == "blast":
        side = _log(rng, 24, 128)
        return dict(flow, lattice="D3Q343", x=side + rng.randint(0, 7), y=side + rng.randint(0, 7), z=side - rng.randint(0, 7),
                    n=rng.choice([0, 4]), storage=rng.choice(["f32", "f16", "f16", "bf16"]), bcx=bc(), bcy=bc(), bcz=bc(),
                    steps=rng.randint(2, 4))
    if kind == "ensemble":
        lmin = _log(rng, 100, 2000)
        return dict(kind="ensemble", count=_log(rng, 16, 1024), lmin=lmin, lmax=lmin + _log(rng, 1, 4000),
                    mode=rng.choice(["fd", "fd", "stream"]), steps=rng.randint(8, 50))
    patch = rng.choice([1, 4, 4, 8])
    length = patch * _log(rng, 128, 1024)
    if kind == "predict":
        return dict(kind="predict", tubes=_log(rng, 1, 512), length=length, patch=patch)
    return dict(kind="train", tubes=_log(rng, 2, 32), length=length, patch=patch)


# --------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(g, *shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda", dtype=torch.float32)


def _shape(case):
    return (case["x"], case["y"], case["z"])[:DIM[case["lattice"]]]


def _bc(case):
    return (case["bcx"], case["bcy"], case["bcz"])[:DIM[case["lattice"]]]


def _tubes(g, lengths, mode):
    """Concatenated shock tubes, diaphragm at mid-tube: left rho = 1, p = 1,
    right lower by the ratios the transport mode keeps finite."""
    count = len(lengths)
    pr = _rand(g, count, lo=2.0, hi=8.0) if mode == "fd" else _rand(g, count, lo=1.5, hi=2.8)
    dr = _rand(g, count, lo=1.5, hi=6.0) if mode == "fd" else _rand(g, count, lo=1.5, hi=2.4)
    ll = torch.as_tensor(lengths, device="cuda")
    tube = torch.repeat_interleave(torch.arange(count, device="cuda"), ll)
    first = torch.cumsum(ll, 0) - ll
    left = (torch.arange(tube.numel(), device="cuda") - first[tube]) < (ll // 2)[tube]
    one = torch.ones((), device="cuda")
    rho = torch.where(left, one, (1.0 / dr)[tube])
    T = torch.where(left, one, (dr / pr)[tube])
    return rho, torch.zeros_like(rho), T


def _flow_fields(case, seed):
    """Discontinuous states within the lattices' envelope, carried by a mean
    flow: a shock tube in 1-D and for open-ended planes, four quadrants for
    periodic ones, a hot sphere in 3-D."""
    g = _gen(seed)
    X, Y, Z = case["x"], case["y"], case["z"]
    D = DIM[case["lattice"]]
    if D == 1:
        rho, u, T = _tubes(g, [X], case["mode"])
        return rho, u[None], T
    wind = _rand(g, D, lo=0.1, hi=0.2)
    if D == 2:
        x = torch.arange(X, device="cuda")[None, :].expand(Y, X)
        y = torch.arange(Y, device="cuda")[:, None].expand(Y, X)
        if case["bcx"] == "copy":
            part = (x >= X // 2).long()
            r4 = torch.cat([_rand(g, 1, lo=1.6, hi=2.2), _rand(g, 1, lo=0.9, hi=1.1)])
            t4, w4 = _rand(g, 2, lo=0.95, hi=1.05), _rand(g, 2, 2, lo=-0.02, hi=0.02)
        else:
            part = 2 * (y >= Y // 2).long() + (x >= X // 2).long()
            r4, t4, w4 = _rand(g, 4, lo=0.8, hi=1.2), _rand(g, 4, lo=0.6, hi=1.4), _rand(g, 2, 4, lo=-0.07, hi=0.07)
        rho, T = r4[part], t4[part]
        u = torch.stack([wind[a] + w4[a][part] for a in range(2)])
    else:
        c = [(torch.arange(s, device="cuda") + 0.5 - s * float(v)) for s, v in zip((X, Y, Z), _rand(g, 3, lo=0.4, hi=0.6))]
        r2 = c[0][None, None, :] ** 2 + c[1][None, :, None] ** 2 + c[2][:, None, None] ** 2
        hot, cold = _rand(g, 1, lo=1.2, hi=1.4), _rand(g, 1, lo=0.6, hi=0.8)
        T = torch.where(r2 <= (min(X, Y, Z) / 6.0) ** 2, hot, cold)
        rho = torch.ones_like(T)
        u = wind[:, None, None, None].expand(3, Z, Y, X)
    return rho.reshape(-1).contiguous(), u.reshape(D, -1).contiguous(), T.reshape(-1).contiguous()


def _ensemble(case, seed):
    """Lengths, rotational degrees of freedom and relaxation times of the
    tubes (the same for every seed: a user's plan), and this seed's fields."""
    rng = np.random.default_rng(case["count"] + 7 * case["lmax"])
    lengths = rng.integers(case["lmin"], case["lmax"] + 1, case["count"])
    n = rng.choice(np.array([2, 4, 6, 7]), case["count"])
    tau = rng.uniform(0.7, 1.0, case["count"])
    return lengths, n, tau, _tubes(_gen(seed), lengths, case["mode"])


def _surrogate_states(case, seed):
    """Tube states with smoothed shocks, and the same a moment later."""
    g = _gen(seed)
    B, L = case["tubes"], case["length"]
    x = torch.arange(L, device="cuda", dtype=torch.float32)[None, :]
    at, dr, pr = _rand(g, B, 1, lo=0.3, hi=0.7) * L, _rand(g, B, 1, lo=1.0, hi=10.0), torch.exp(_rand(g, B, 1, lo=0.7, hi=3.0))
    speed, v = _rand(g, B, 1, lo=3.0, hi=12.0), _rand(g, B, 1, lo=0.1, hi=0.6)
    gamma = torch.tensor([5 / 3, 1.4, 9 / 7, 1.25], device="cuda")[torch.randint(4, (B,), generator=g, device="cuda")]

    def state(shift):
        s = torch.sigmoid((at + shift - x) / 4.0)
        rho = 1.0 / dr + (1.0 - 1.0 / dr) * s
        p = 1.0 / pr + (1.0 - 1.0 / pr) * s
        return [f.reshape(-1).contiguous() for f in (rho, v * s * (1.0 - s) * 4.0, p / rho)]

    return state(0.0), state(speed), gamma.contiguous()


def _network(case, seed):
    net = ConvOperator(C=128, k=5, patch=case["patch"], seed=int(seed) % 65536, out_scale=(0.05, 0.04, 0.06))
    return net


def prepare(case, seed):
    if case["kind"] == "flow":
        sim = Lbm(case["lattice"], case["n"], TAU, _shape(case), _bc(case), mode=case["mode"], m_fd=M_FD,
                  storage=case["storage"])
        return dict(kind="flow", sim=sim, fields=_flow_fields(case, seed), steps=case["steps"])
    if case["kind"] == "ensemble":
        lengths, n, tau, fields = _ensemble(case, seed)
        ens = LbmBatch(lengths, n, tau, mode=case["mode"], m_fd=M_FD)
        if case["lmin"] == case["lmax"]:  # windows: one node per thread, as the surrogate sets it
            ens.set_block(min(1024, -(-case["lmax"] // 32) * 32))
        return dict(kind="ensemble", ens=ens, fields=fields, steps=case["steps"])
    s0, s1, gamma = _surrogate_states(case, seed)
    return dict(kind=case["kind"], net=_network(case, seed), s0=s0, s1=s1, gamma=gamma, B=case["tubes"], L=case["length"])


def run(state):
    if state["kind"] == "flow":
        sim = state["sim"]
        sim.set_macro(*state["fields"])
        sim.step(state["steps"])
        return sim.moments()
    if state["kind"] == "ensemble":
        ens = state["ens"]
        ens.set_macro(*state["fields"])
        ens.run(state["steps"])
        return ens.moments()
    net, B, L = state["net"], state["B"], state["L"]
    if state["kind"] == "predict":
        return net.predict(*state["s0"], state["gamma"], B, L)
    feat = net.features(*state["s0"], state["gamma"], B, L)
    target = net.targets(*state["s0"], *state["s1"])
    loss = net.loss_and_grad(feat, target, B, L)
    grads = {name: net.grads[off:off + math.prod(shape)].view(shape) for name, (off, shape) in net.offsets.items()}
    return {"loss": loss, **grads}


# ----------------------------------------------------------------------- work
def work(case):
    """Bytes and operations of one pass.  Flows: the fields in and out, and
    every population read and written once a step where the state does not
    stay on the chip; per node and step about 14 operations a translational
    population (pull sums, equilibrium, relaxation), 9 a rotational one and
    axis, and 9 a population and axis for finite-difference transport."""
    if case["kind"] == "flow":
        D, q, nodes = DIM[case["lattice"]], Q[case["lattice"]], case["x"] * case["y"] * case["z"]
        qr = 7 if case["n"] else 0
        size = 4 if case["storage"] == "f32" else 2
        per_node = (q + qr) * size + (16 if case["storage"].endswith("_node") else 0)
        io = 2 * 4 * (D + 2) * nodes
        steps = case["steps"]
        state = per_node * nodes
        flops = nodes * steps * (14.0 * q + qr * (14.0 + 9.0 * D) + (9.0 * D * q if case["mode"] == "fd" else 0.0))
        return {"bytes": float(io + (2 * state * steps if 2 * state > L2_BYTES else 0)), "flops": flops}
    if case["kind"] == "ensemble":
        nodes = int(_ensemble_nodes(case))
        flops = nodes * case["steps"] * (14.0 * 7 + 7 * 23.0 + (9.0 * 7 if case["mode"] == "fd" else 0.0))
        return {"bytes": 24.0 * nodes, "flops": flops}
    nodes, C, k, layers = case["tubes"] * case["length"], 128, 5, 12
    P = nodes // case["patch"]
    body = 2.0 * P * C * (k * C * layers + 7.0 * case["patch"])
    act = 2.0 * P * C  # one activation tensor
    if case["kind"] == "predict":
        return {"bytes": 24.0 * nodes + 2.0 * act * layers, "flops": body}
    # forward: each layer's input, pre-activation and output; backward: the
    # gradient, the pre-activation and the input of each layer once more
    weights = 4.0 * (k * C * C * layers)
    return {"bytes": 40.0 * nodes + act * layers * 6 + 2 * weights, "flops": 3.0 * body}


def _ensemble_nodes(case):
    rng = np.random.default_rng(case["count"] + 7 * case["lmax"])
    return rng.integers(case["lmin"], case["lmax"] + 1, case["count"]).sum()


# ---------------------------------------------------------- 64-bit references
def _d1q7():
    """Spacing r and weights of the 7 velocities r (-3..3): moments 0, 2, 4,
    6 and 8 of the unit Gaussian."""
    e2 = np.array([0.0, 1.0, 4.0, 9.0])
    mult = np.array([1.0, 2.0, 2.0, 2.0])

    def weights(r):
        a = np.stack([mult * (e2 * r * r) ** k for k in range(4)])
        return np.linalg.solve(a, np.array([1.0, 1.0, 3.0, 15.0]))

    def miss(r):
        return float(np.sum(mult * weights(r) * (e2 * r * r) ** 4) - 105.0)

    lo, hi = 1.1, 1.3
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        if (miss(lo) < 0) != (miss(mid) < 0):
            hi = mid
        else:
            lo = mid
    w = weights(lo)
    return lo, [float(w[abs(j - 3)]) for j in range(7)]


def _lattice(name):
    r, w1 = _d1q7()
    D = DIM[name]
    e = [(i % 7 - 3, i // 7 % 7 - 3, i // 49 - 3)[:D] for i in range(7 ** D)]
    if name != "D2Q37":
        return r, e, [math.prod(w1[v + 3] for v in ei) for ei in e], w1
    e = [v for v in e if sorted(map(abs, v)) not in ([2, 2], [2, 3])]
    groups = sorted({tuple(sorted(map(abs, v))) for v in e})
    moment = {0: 1.0, 2: 1.0, 4: 3.0, 6: 15.0, 8: 105.0}
    rows, want = [], []
    for a in range(0, 9, 2):
        for b in range(0, min(a, 8 - a) + 1, 2):
            rows.append([sum((r * v[0]) ** a * (r * v[1]) ** b for v in e if tuple(sorted(map(abs, v))) == k) for k in groups])
            want.append(moment[a] * moment[b])
    scale = 1.0 / np.array(want)
    sol = np.linalg.lstsq(np.array(rows) * scale[:, None], np.array(want) * scale, rcond=None)[0]
    return r, e, [float(sol[groups.index(tuple(sorted(map(abs, v))))]) for v in e], w1


def _geq(D, r, e, w, rho, u, u2, T):
    """Fourth-order Hermite projection of the Maxwellian, one velocity."""
    c = r * sum(e[a] * u[a] for a in range(D)) if any(e) else torch.zeros_like(rho)
    s, t = r * r * sum(v * v for v in e), T - 1.0
    p = 1.0 + c + 0.5 * (c * c - u2 + t * (s - D)) + c * (c * c - 3.0 * u2 + 3.0 * t * (s - D - 2.0)) / 6.0
    p = p + (c ** 4 - 6.0 * c * c * u2 + 3.0 * u2 * u2 + 6.0 * t * (c * c * (s - D - 4.0) + (D + 2.0 - s) * u2)
             + 3.0 * t * t * (s * s - 2.0 * (D + 2.0) * s + D * (D + 2.0))) / 24.0
    return w * rho * p


def _upwind(f, nu, axis, shift):
    """nu df/dx, third-order upwind; nu a number or a field."""
    if isinstance(nu, float):
        s = -1 if nu >= 0 else 1
        return abs(nu) / 6.0 * (shift(f, axis, 2 * s) - 6.0 * shift(f, axis, s) + 3.0 * f + 2.0 * shift(f, axis, -s))
    lo = shift(f, axis, -2) - 6.0 * shift(f, axis, -1) + 3.0 * f + 2.0 * shift(f, axis, 1)
    hi = shift(f, axis, 2) - 6.0 * shift(f, axis, 1) + 3.0 * f + 2.0 * shift(f, axis, -1)
    return nu.abs() / 6.0 * torch.where(nu >= 0, lo, hi)


def _evolve(name, n, tau, mode, rho, u, T, steps, shift):
    """The method in 64 bits; n and tau numbers or fields; shift(f, axis, k)
    is f at x + k along the axis, wrapped or clamped."""
    r, e, w, wr = _lattice(name)
    D, m = DIM[name], float(M_FD) if mode == "fd" else 1.0
    omega, rot = 1.0 / (m * tau), not isinstance(n, int) or n > 0

    def at(f, ei, sign):
        for a in range(D):
            if ei[a]:
                f = shift(f, a, sign * ei[a])
        return f

    def heq(T):
        t, out = T - 1.0, []
        for j in range(7):
            s = (r * (j - 3)) ** 2
            out.append(wr[j] * (1.0 + 0.5 * t * (s - 1.0) + 0.125 * t * t * (s * s - 6.0 * s + 3.0)))
        return out

    def moments(f, h):
        rho, e2 = torch.zeros_like(f[0]), torch.zeros_like(f[0])
        j = [torch.zeros_like(f[0]) for _ in range(D)]
        for i, ei in enumerate(e):
            g = at(f[i], ei, -1) if mode == "stream" else f[i]
            rho += g
            e2 += g * float(sum(v * v for v in ei))
            for a in range(D):
                if ei[a]:
                    j[a] += g * float(ei[a])
        u = [r * v / rho for v in j]
        u2 = sum(v * v for v in u)
        energy = 0.5 * (r * r * e2 / rho - u2)
        if rot:
            energy = energy + 0.5 * n * sum((r * (k - 3)) ** 2 * h[k] for k in range(7))
        return rho, u, u2, energy / (0.5 * (D + n))

    u2 = sum(v * v for v in u)
    f = [at(_geq(D, r, ei, w[i], rho, u, u2, T), ei, 1) if mode == "stream" else _geq(D, r, ei, w[i], rho, u, u2, T)
         for i, ei in enumerate(e)]
    h = heq(T) if rot else []
    for _ in range(steps):
        rho, u, u2, T = moments(f, h)
        new = []
        for i, ei in enumerate(e):
            if mode == "stream":
                new.append((1.0 - omega) * at(f[i], ei, -1) + omega * _geq(D, r, ei, w[i], rho, u, u2, T))
            else:
                adv = sum(_upwind(f[i], ei[a] / m, a, shift) for a in range(D) if ei[a])
                new.append((1.0 - omega) * f[i] + omega * _geq(D, r, ei, w[i], rho, u, u2, T) - adv)
        if rot:
            eq = heq(T)
            h = [(1.0 - omega) * h[k] + omega * eq[k] - sum(_upwind(h[k], u[a] / (m * r), a, shift) for a in range(D))
                 for k in range(7)]
        f = new
    rho, u, _, T = moments(f, h)
    return rho, u, T


def _exact_flow(case, seed):
    D, X, Y, Z = DIM[case["lattice"]], case["x"], case["y"], case["z"]
    if X * Y * Z * (Q[case["lattice"]] + 7) * 16 > 120e9:
        return None
    rho, u, T = _flow_fields(case, seed)
    shape = (Z, Y, X)[3 - D:]
    size, bc = _shape(case), _bc(case)

    def shift(f, axis, k):
        i = torch.arange(size[axis], device="cuda") + k
        i = i % size[axis] if bc[axis] == "periodic" else i.clamp(0, size[axis] - 1)
        return f.index_select(D - 1 - axis, i)

    out = _evolve(case["lattice"], case["n"], TAU, case["mode"], rho.double().view(shape),
                  [v.double().view(shape) for v in u], T.double().view(shape), case["steps"], shift)
    return out[0].reshape(-1), torch.stack([v.reshape(-1) for v in out[1]]), out[2].reshape(-1)


def _exact_ensemble(case, seed):
    lengths, n, tau, fields = _ensemble(case, seed)
    ll = torch.as_tensor(lengths, device="cuda")[:, None]
    x = torch.arange(int(lengths.max()), device="cuda")[None, :]
    inside = x < ll

    def grid(f, fill):
        g = torch.full(inside.shape, fill, device="cuda", dtype=torch.float64)
        g[inside] = f.double()
        return g

    def shift(f, axis, k):
        return f.gather(1, torch.minimum((x + k).clamp(min=0), ll - 1))

    col = lambda v: torch.as_tensor(v, device="cuda", dtype=torch.float64)[:, None]  # noqa: E731
    rho, u, T = _evolve("D1Q7", col(n), col(tau), case["mode"], grid(fields[0], 1.0), [grid(fields[1], 0.0)],
                        grid(fields[2], 1.0), case["steps"], shift)
    return rho[inside], u[0][inside], T[inside]


def _network64(params, feat, B, patch, dilations, k):
    """The network in 64 bits on [B, positions, 4 patch] features."""
    x = torch.nn.functional.linear(feat, params["Wl"], params["bl"])
    for i, d in enumerate(dilations):
        pad = torch.nn.functional.pad(x, (0, 0, k // 2 * d, k // 2 * d))
        z = params["b"][i].expand_as(x)
        for t in range(k):
            z = z + pad[:, t * d:t * d + x.shape[1]] @ params["W"][i, t].T
        x = x + torch.nn.functional.gelu(z, approximate="tanh")
    return torch.nn.functional.linear(x, params["Wp"], params["bp"])


def _exact_network(case, seed):
    s0, s1, gamma = _surrogate_states(case, seed)
    net = _network(case, seed)
    B, L, patch = case["tubes"], case["length"], case["patch"]
    params = {name: net.params[off:off + math.prod(shape)].view(shape).double() for name, (off, shape) in net.offsets.items()}
    sc, so = net.in_scale, torch.tensor(net.out_scale, device="cuda", dtype=torch.float64)
    d0, d1 = [f.double() for f in s0], [f.double() for f in s1]
    gam = torch.repeat_interleave(gamma.double(), L)
    feat = torch.stack([(d0[0] - 1) / sc[0], d0[1] / sc[1], (d0[2] - 1) / sc[2], (gam - 1.4) / sc[3]], 1)
    feat = feat.reshape(B, L // patch, 4 * patch)
    if case["kind"] == "predict":
        out = []
        with torch.no_grad():
            for b in range(0, B, 64):
                out.append(_network64(params, feat[b:b + 64], B, patch, net.dil, net.k).reshape(-1, 3))
        out = torch.cat(out) * so
        return tuple(d0[i] + out[:, i] for i in range(3))
    for p in params.values():
        p.requires_grad_(True)
    target = torch.stack([(b - a) for a, b in zip(d0, d1)], 1) / so
    out = _network64(params, feat, B, patch, net.dil, net.k).reshape(-1, 3)
    loss = ((out - target) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach().reshape(1), **{name: p.grad for name, p in params.items()}}


def exact(case, seed):
    if case["kind"] == "flow":
        return _exact_flow(case, seed)
    return _exact_ensemble(case, seed) if case["kind"] == "ensemble" else _exact_network(case, seed)
