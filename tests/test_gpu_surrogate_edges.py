"""The surrogate's lift, head and reduction kernels where their dispatch and
their blocks end: positions short of a block, one past one, and past the
size at which a thread takes two; every output and feature count; channel
counts off the vector path; tensors off the vectors' alignment.

Tolerances: float32 products and sums, 1e-5 of the sum of the terms'
magnitudes (a few thousand terms at unit roundoff 6e-8, summed in blocks);
bfloat16 results 2^-9 of a scale about twice the value's or more (half an ulp
is at most 2^-8 of the value), and 2^-10 of it for the hardware tanh."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1606_06107_gb300 import load_library
    return load_library()


def make(seed, *shape, dtype="float32", skip=0):
    """Seeded normal values; `skip` elements off the allocation's alignment."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = int(np.prod(shape))
    buf = torch.zeros(n + skip, device="cuda", dtype=getattr(torch, dtype))
    buf[skip:] = torch.randn(n, generator=g, device="cuda").to(buf.dtype)
    return buf[skip:].view(*shape)


def close(got, want, scale, rel=1e-5):
    assert bool(((got.double() - want).abs() <= rel * scale + 1e-30).all()), float(
        ((got.double() - want).abs() / scale.clamp_min(1e-30)).max())


@pytest.mark.parametrize("P", [1, 127, 129, 77823, 77824, 77825])
@pytest.mark.parametrize("C,Fo", [(128, 3), (128, 12), (256, 6), (256, 24), (40, 12)])
def test_head(lib, P, C, Fo):
    import torch
    x, W, b = make(1, P, C, dtype="bfloat16"), make(2, Fo, C), make(3, Fo)
    out = torch.full((P + 1, Fo), float("nan"), device="cuda")
    assert lib.lbm_nn_head(x.data_ptr(), W.data_ptr(), b.data_ptr(), out.data_ptr(), P, C, Fo, None) == 0
    xd, Wd = x.double(), W.double()
    close(out[:P], xd @ Wd.T + b.double(), xd.abs() @ Wd.abs().T + b.double().abs())
    assert bool(out[P].isnan().all())


@pytest.mark.parametrize("P", [1, 9, 4865])
@pytest.mark.parametrize("C,Fo,skip", [(128, 3, 0), (128, 12, 0), (128, 12, 1), (128, 24, 0), (256, 6, 1), (256, 12, 0),
                                       (256, 24, 0)])
def test_head_backward(lib, P, C, Fo, skip):
    import torch
    go, W = make(1, P, Fo), make(2, Fo, C)
    x, z = make(3, P, C, dtype="bfloat16", skip=skip), make(4, P, C, dtype="bfloat16", skip=skip)
    gx, gz = make(5, P, C, skip=skip), make(6, P, C, dtype="bfloat16", skip=skip)
    gW, gb = torch.zeros(Fo, C, device="cuda"), torch.zeros(Fo, device="cuda")
    assert lib.lbm_nn_head_backward(*[v.data_ptr() for v in (go, x, W, z, gx, gz, gW, gb)], P, C, Fo, None) == 0
    god, Wd, xd = go.double(), W.double(), x.double()
    want = god @ Wd
    close(gx, want, god.abs() @ Wd.abs())
    zd = z.double().requires_grad_(True)
    torch.nn.functional.gelu(zd, approximate="tanh").sum().backward()
    # gelu' is at most 1.13 and its tanh enters with at most |z| + 1
    scale = god.abs() @ Wd.abs() * 1.13
    close(gz, want * zd.grad, scale * (1 + z.double().abs()), rel=2.0 ** -9 + 2.0 ** -10)
    close(gW, god.T @ xd, god.abs().T @ xd.abs())
    close(gb, god.sum(0), god.abs().sum(0))


@pytest.mark.parametrize("P", [1, 127, 129, 4999])
@pytest.mark.parametrize("C,F", [(32, 4), (96, 8), (128, 16), (512, 16), (1024, 32)])
def test_lift_backward(lib, P, C, F):
    import torch
    gx, feat = make(1, P, C), make(2, P, F, skip=1)
    gW, gb = torch.zeros(C, F, device="cuda"), torch.zeros(C, device="cuda")
    assert lib.lbm_nn_lift_backward(gx.data_ptr(), feat.data_ptr(), gW.data_ptr(), gb.data_ptr(), P, F, C, None) == 0
    close(gW, gx.double().T @ feat.double(), gx.double().abs().T @ feat.double().abs())
    close(gb, gx.double().sum(0), gx.double().abs().sum(0))


@pytest.mark.parametrize("P", [1, 15, 65, 40001])
@pytest.mark.parametrize("C,skip", [(128, 0), (256, 0), (384, 0), (128, 1), (100, 0), (3, 0)])
def test_bias_gradient(lib, P, C, skip):
    import torch
    gz, gb = make(1, P, C, dtype="bfloat16", skip=skip), make(2, C)
    before = gb.double()
    assert lib.lbm_nn_bias_grad(gz.data_ptr(), gb.data_ptr(), P, C, None) == 0
    close(gb, before + gz.double().sum(0), before.abs() + gz.double().abs().sum(0))


@pytest.mark.parametrize("impl", [0, 3])
@pytest.mark.parametrize("B,L,C,k,d", [(1, 1, 128, 5, 4), (3, 300, 128, 5, 3), (2, 77, 256, 3, 2), (2, 257, 128, 5, 1),
                                       (1200, 300, 128, 3, 1)])
def test_forward_without_the_pre_activation(lib, impl, B, L, C, k, d):
    """The inference product takes other accesses and packed arithmetic: the
    same bits as the product that also stores the pre-activation."""
    import torch
    x, W, b = make(1, B * L, C, dtype="bfloat16"), make(2, k, C, C, dtype="bfloat16"), make(3, C)
    y = [torch.full((B * L + 1, C), 7.0, device="cuda", dtype=torch.bfloat16) for _ in range(2)]
    z = torch.empty(B * L, C, device="cuda", dtype=torch.bfloat16)
    st = torch.zeros(1, device="cuda", dtype=torch.int32)
    for out, pre in ((y[0], z.data_ptr()), (y[1], None)):
        assert lib.lbm_nn_conv_forward(x.data_ptr(), W.data_ptr(), b.data_ptr(), out.data_ptr(), pre, B, L, C, k, d, impl,
                                       st.data_ptr(), None) == 0
    assert int(st) == 0 and torch.equal(y[0], y[1])
    assert bool((y[0][B * L] == 7.0).all())


@pytest.mark.parametrize("impl", [0, 1, 2, 3])
@pytest.mark.parametrize("B,L,C,k,d", [(3, 300, 128, 5, 3), (1, 64, 128, 3, 1), (2, 77, 256, 3, 2), (40, 130, 128, 5, 1)])
def test_bias_gradient_with_the_weight_gradient(lib, impl, B, L, C, k, d):
    """Both gradients of the joint entry; the bias sums over a few thousand
    terms in blocks of 64, the weight gradient as its own entry gives it."""
    import torch
    gz, x = make(1, B * L, C, dtype="bfloat16"), make(2, B * L, C, dtype="bfloat16")
    gw, gw2, gb = torch.zeros(k, C, C, device="cuda"), torch.zeros(k, C, C, device="cuda"), make(3, C)
    before = gb.double()
    st = torch.zeros(1, device="cuda", dtype=torch.int32)
    assert lib.lbm_nn_conv_backward_weight_bias(gz.data_ptr(), x.data_ptr(), gw.data_ptr(), gb.data_ptr(), B, L, C, k, d,
                                                impl, st.data_ptr(), None) == 0
    assert lib.lbm_nn_conv_backward_weight(gz.data_ptr(), x.data_ptr(), gw2.data_ptr(), B, L, C, k, d, impl, st.data_ptr(),
                                           None) == 0
    assert int(st) == 0
    close(gb, before + gz.double().sum(0), before.abs() + gz.double().abs().sum(0))
    close(gw, gw2.double(), (gz.double().abs().T @ x.double().abs())[None].expand(k, -1, -1))


@pytest.mark.parametrize("B,L,skip", [(1, 1, 0), (3, 7, 0), (5, 12, 0), (255, 4112, 0), (256, 4096, 0),
                                      (256, 4096, 1), (1051, 1001, 0), (1051, 1004, 0)])
def test_features_targets_and_update(lib, B, L, skip):
    import ctypes
    import torch
    n = B * L
    a, b = [make(k, n, skip=skip) for k in (1, 2, 3)], [make(k, n, skip=skip) for k in (4, 5, 6)]
    gamma, out = make(7, B), make(8, 3 * n, skip=skip)
    feat, tgt = torch.empty(n, 4, device="cuda"), make(9, 3 * n, skip=skip)
    new = [make(9 + k, n, skip=skip) for k in (1, 2, 3)]
    s4, s3 = (ctypes.c_float * 4)(1.0, 0.5, 2.0, 0.25), (ctypes.c_float * 3)(0.05, 0.04, 0.06)
    ptr = lambda v: [x.data_ptr() for x in v]  # noqa: E731
    assert lib.lbm_nn_features(*ptr(a), gamma.data_ptr(), feat.data_ptr(), B, L, s4, None) == 0
    assert lib.lbm_nn_targets(*ptr(a), *ptr(b), tgt.data_ptr(), n, s3, None) == 0
    assert lib.lbm_nn_apply(*ptr(a), out.data_ptr(), *ptr(new), n, s3, None) == 0
    da, db = [v.double() for v in a], [v.double() for v in b]
    g = torch.repeat_interleave(gamma.double(), L)
    want = torch.stack([(da[0] - 1), da[1] / 0.5, (da[2] - 1) / 2, (g - 1.4) / 0.25], 1)
    close(feat, want, 10 * (1 + want.abs()), rel=1e-6)
    scale = torch.tensor([np.float32(v) for v in (0.05, 0.04, 0.06)], device="cuda", dtype=torch.float64)
    want = torch.stack([y - x for x, y in zip(da, db)], 1) / scale
    close(tgt.view(n, 3), want, want.abs() + 100, rel=1e-6)
    for k in range(3):
        want = da[k] + out.double().view(n, 3)[:, k] * scale[k]
        close(new[k], want, da[k].abs() + 1, rel=1e-6)


@pytest.mark.parametrize("n", [1, 255, 257, 311297])
def test_mean_squared_error(lib, n):
    import torch
    a, b, g = make(1, n), make(2, n), make(3, n)
    loss = torch.zeros(1, device="cuda", dtype=torch.float64)
    assert lib.lbm_nn_mse(a.data_ptr(), b.data_ptr(), g.data_ptr(), loss.data_ptr(), n, None) == 0
    d = a.double() - b.double()
    assert abs(float(loss) - float((d * d).mean())) <= 1e-6 * float((d * d).mean())  # float32 differences
    close(g, 2 * d / n, (a.double().abs() + b.double().abs()) * 2 / n)
