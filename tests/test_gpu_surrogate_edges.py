"""The surrogate's lift, head and reduction kernels where their dispatch and
their blocks end: positions short of a block, one past one, and past the
size at which a thread takes two; every output and feature count; channel
counts off the vector path; tensors off the vectors' alignment.

Tolerances: float32 products and sums, 1e-5 of the sum of the terms'
magnitudes (a few thousand terms at unit roundoff 6e-8, summed in blocks);
bfloat16 results half an ulp (2^-9) more, and 2^-10 for the hardware tanh."""
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


@pytest.mark.parametrize("n", [1, 255, 257, 311297])
def test_mean_squared_error(lib, n):
    import torch
    a, b, g = make(1, n), make(2, n), make(3, n)
    loss = torch.zeros(1, device="cuda", dtype=torch.float64)
    assert lib.lbm_nn_mse(a.data_ptr(), b.data_ptr(), g.data_ptr(), loss.data_ptr(), n, None) == 0
    d = a.double() - b.double()
    assert abs(float(loss) - float((d * d).mean())) <= 1e-6 * float((d * d).mean())  # float32 differences
    close(g, 2 * d / n, (a.double().abs() + b.double().abs()) * 2 / n)
