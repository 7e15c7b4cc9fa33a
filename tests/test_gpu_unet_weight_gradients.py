"""Weight gradients of the 3x3x3 convolutions keep every bit of the plain tensor-core product.

A weight gradient is D[(tap, ci), co] = sum_v a(v + tap, ci) g(v, co) over the voxels v.  Its value
depends on how the FP32 sum is cut into chains, so the cut is part of the result: the voxels in
memory order, in ranges of at least 256 (a multiple of 64) that fill two blocks per SM, the ranges'
sums added in order.  The network below has operands that are known exactly: its last convolution
sees a(v, c) = bf16(relu(w_c x(v) + b_c)) through identity weights and the skip connection, and,
with zero weights and bias one, the gradient g(v, co) = bf16(head_co gpred(v)).  The same ranges go
through unet_gemm, and the sums have to agree in every bit.  The bias gradient, an FP32 sum of V terms
in another order than the reference's, agrees to 1e-6 of the sum of magnitudes (V terms over 256
blocks of 256 threads: chains of a few terms and two trees, fewer than 16 roundings of 2^-24).
"""
import numpy as np
import pytest

from oracle import unet as U

pytestmark = pytest.mark.gpu

SMS = 152


@pytest.mark.parametrize("c,shape", [(16, (40, 24, 34)), (32, (20, 26, 18)), (64, (12, 20, 34)), (128, (12, 20, 10))])
def test_weight_gradient_keeps_the_bits_of_the_product(c, shape):
    import torch
    from paper_1808_07150_gb300 import learned
    spec = U.UNetSpec((c, 16))
    gen = torch.Generator().manual_seed(c)
    x = (torch.rand(shape, generator=gen) + 0.1).bfloat16().float()
    gpred = torch.randn(shape, generator=gen)
    w0 = torch.randn(c, generator=gen).bfloat16().float()
    b0 = torch.randn(c, generator=gen)
    head = torch.randn(c, generator=gen)
    p = {k: np.zeros(s, np.float32) for k, s in U.layer_shapes(spec)}
    eye = np.eye(c, dtype=np.float32)
    p["enc0a.W"][:, 0, 1, 1, 1] = w0
    p["enc0a.b"][:] = b0
    p["enc0b.W"][:, :, 1, 1, 1] = eye
    p["dec0a.W"][:, c:, 1, 1, 1] = eye      # [up, skip]
    p["dec0b.b"][:] = 1.0
    p["head.W"][...] = head.numpy().reshape(p["head.W"].shape)
    with learned.UNet(shape, spec.channels) as net:
        net.set_params(np.concatenate([p[k].ravel() for k, _ in U.layer_shapes(spec)]))
        net.forward(x.reshape(-1).cuda(), 1.0)
        net.backward(gpred=gpred.reshape(-1).cuda(), want_loss=False)
        grads, q = net.get_grads(), 0
        assert learned.device_error() == 0
    g = {}
    for k, s in U.layer_shapes(spec):
        n = int(np.prod(s))
        g[k] = grads[q:q + n].reshape(s)
        q += n

    a = torch.relu(x[..., None] * w0 + b0).bfloat16()                     # (ny, nx, nz, c)
    gv = (gpred[..., None] * head).bfloat16().reshape(-1, c)
    pad = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1, 1, 1))
    ny, nx, nz = shape
    cols = torch.cat([pad[ty:ty + ny, tx:tx + nx, tz:tz + nz].reshape(-1, c)
                      for ty in range(3) for tx in range(3) for tz in range(3)], dim=1).contiguous()  # (V, 27 c)
    V = cols.shape[0]
    tiles = (27 * c + 127) // 128
    splits = max(1, min((2 * SMS + tiles - 1) // tiles, (V + 255) // 256))
    per = ((V + splits - 1) // splits + 63) // 64 * 64
    total = torch.zeros(27 * c, c, device="cuda")
    for k in range(0, V, per):
        part = torch.empty(27 * c, c, device="cuda")
        learned.gemm(cols[k:k + per].cuda().contiguous(), gv[k:k + per].cuda().contiguous(), part, 3)
        total += part
    torch.cuda.synchronize()
    ref = total.cpu().numpy().reshape(3, 3, 3, c, c).transpose(4, 3, 0, 1, 2)
    np.testing.assert_array_equal(g["dec0b.W"], ref)
    gd = gv.double().numpy()
    assert np.abs(g["dec0b.b"] - gd.sum(0)).max() <= 1e-6 * np.abs(gd).sum(0).max()
