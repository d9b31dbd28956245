"""The 16-byte forms of the ReLU and bias gradients (csrc/nn.cu) against torch on channel slices that allow them (strides
and offsets in eighths) and on ones that take the general kernels, with odd voxel counts."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    _build.build()
    from paper_1501_04840_gb300 import nn
    nn.lib()
    return nn


@pytest.mark.parametrize("C,gs,go,ys,yo", [(16, 16, 0, 16, 0), (24, 64, 8, 32, 8), (8, 8, 0, 8, 0), (48, 56, 4, 48, 0),
                                           (5, 16, 3, 8, 1)])
@pytest.mark.parametrize("M", [1, 1027])
def test_relu_grad(K, M, C, gs, go, ys, yo):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(C + M)
    g = torch.randn((M, gs), generator=gen, device="cuda").bfloat16()
    y = torch.randn((M, ys), generator=gen, device="cuda").bfloat16()
    y[::3, yo] = 0.0
    y[-1, yo] = float("nan")
    want = g.clone()
    part = want[:, go:go + C]
    part[~(y[:, yo:yo + C] > 0)] = 0
    K.relu_grad(K.Slice(g, go, C), K.Slice(y, yo, C))
    torch.cuda.synchronize()
    assert torch.equal(g.view(torch.int16), want.view(torch.int16))


@pytest.mark.parametrize("cout,dys,dyo", [(16, 16, 0), (48, 64, 8), (48, 64, 4), (64, 64, 0)])
def test_bias_gradient(K, cout, dys, dyo):
    import torch
    vol = (2, 3, 5, 37)
    gen = torch.Generator(device="cuda").manual_seed(cout + dyo)
    x = torch.randn(vol + (16,), generator=gen, device="cuda").bfloat16()
    dy = torch.randn(vol + (dys,), generator=gen, device="cuda").bfloat16()
    dw = torch.zeros((cout, 27, 16), device="cuda")
    db = torch.ones(cout, device="cuda")
    K.conv3d_wgrad(vol, K.whole(x), K.Slice(dy, dyo, cout), dw, db)
    torch.cuda.synchronize()
    flat = dy[..., dyo:dyo + cout].double().flatten(0, 3)
    # FP32 sums of 1110 terms in a few levels: 1e-6 of the sum of magnitudes
    assert torch.all((db.double() - 1 - flat.sum(0)).abs() <= 1e-6 * (flat.abs().sum(0) + 1))
