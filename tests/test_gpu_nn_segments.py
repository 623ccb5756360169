"""The persistent convolution blocks where one takes several tiles and plane segments, so that the input ring, the
accumulator ring and its wrap carry over from one to the next (csrc/vofp_nn.cu): single layers against a plain FP64
product, and a forward pass, whose pooled, upsampled and output tensors come out of the convolutions' epilogues,
against the layers applied one by one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import nn_ref as R
from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _planar(a):
    """(nz, ny, nx, C) channels-last -> chunk-planar (C/8, voxels, 8)."""
    nz, ny, nx, C = a.shape
    return a.reshape(nz * ny * nx, C // 8, 8).permute(1, 0, 2).contiguous().reshape(-1)


def _unplanar(flat, shape):
    n = shape[0] * shape[1] * shape[2]
    return flat.reshape(-1, n, 8).permute(1, 0, 2).reshape(*shape, -1)


def _conv(x, W):
    """sum over taps of x[v + tap - 1] W[tap]^T in FP64 (zero padding)."""
    nz, ny, nx, _ = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    out = torch.zeros(nz, ny, nx, W.shape[1], dtype=torch.float64, device=x.device)
    for t in range(27):
        k, j, i = t // 9, t // 3 % 3, t % 3
        out += xp[k:k + nz, j:j + ny, i:i + nx] @ W[t].T
    return out


@pytest.mark.parametrize("layer", range(10))
def test_conv_layer_over_several_segments_per_block(layer):
    """20 x 404 x 250 voxels: 832 tiles in the plane (ragged in x and y), more than there are blocks, and more planes than
    the accumulator ring has column blocks at 16 channels.  BF16 outputs within one unit (2^-8) and 1e-5 of the
    largest, as FP32 sums of BF16 products rounded once."""
    from paper_1410_1937_gb300 import vofp
    shape = (20, 404, 250)
    cin, cout = R.LAYERS[layer]
    net = vofp.Network(seed=3)
    W, b = R.unpack(net.get_params().astype(np.float64))[0][layer]
    Wb = torch.from_numpy(R.bf16_round(W)).cuda()
    g = torch.Generator(device="cuda").manual_seed(40 + layer)
    x = torch.randn(*shape, cin, generator=g, device="cuda").to(torch.bfloat16)
    dy = torch.randn(*shape, cout, generator=g, device="cuda").to(torch.bfloat16)
    for grad, src in ((False, x), (True, dy)):
        got = _unplanar(net.conv_apply(layer, _planar(src), shape, data_grad=grad), shape).double()
        if grad:   # taps mirrored, channels transposed
            ref = _conv(src.double(), Wb.flip(0).transpose(1, 2))
        else:
            ref = (_conv(src.double(), Wb) + torch.from_numpy(np.asarray(b, dtype=np.float64)).cuda()).clamp(min=0.0)
        bad = (got - ref).abs() > 2.0 ** -8 * ref.abs() + 1e-5 * ref.abs().max()
        assert not bool(bad.any()), (layer, grad, int(bad.sum()), float((got - ref).abs().max()))


@pytest.mark.parametrize("shape", [(44, 40, 24), (264, 324, 12)])
def test_forward_equals_its_layers(shape):
    """Output within 1e-2 in the norm (BF16 through ten layers; the input's scale is rounded once more here)."""
    from paper_1410_1937_gb300 import vofp
    nx, ny, nz = shape
    p = I.config1(shape=shape)
    ctx, t = vofp.context_for(p)
    net = vofp.Network(seed=7)
    net.bind(ctx, t["F"])
    geo, mask = net.export_geometry()
    r = torch.randn(p.n, generator=torch.Generator(device="cuda").manual_seed(5), device="cuda") * mask
    got = net.forward(r)
    _, hw, hb = R.unpack(net.get_params().astype(np.float64))
    rms = float(torch.sqrt((r.double() ** 2).sum() / mask.double().sum()))
    s1, s2, s4 = (nz, ny, nx), (nz // 2, ny // 2, nx // 2), (nz // 4, ny // 4, nx // 4)
    x = torch.zeros(*s1, 16, dtype=torch.bfloat16, device="cuda")
    x[..., :8] = geo.view(torch.bfloat16).reshape(*s1, 8)
    x[..., 7] = (r / rms).reshape(s1).to(torch.bfloat16)

    def conv(layer, a, s):
        return _unplanar(net.conv_apply(layer, _planar(a), s), s)

    def pool(a):
        z, y, w, c = a.shape
        return a.float().reshape(z // 2, 2, y // 2, 2, w // 2, 2, c).mean(dim=(1, 3, 5)).to(torch.bfloat16)

    def up(a):
        return a.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)

    cin0 = R.LAYERS[0][0]
    k1 = conv(1, conv(0, x[..., :cin0].contiguous(), s1), s1)
    k2 = conv(3, conv(2, pool(k1), s2), s2)
    k3 = conv(5, conv(4, pool(k2), s4), s4)
    d2 = conv(7, conv(6, torch.cat([up(k3), k2], -1), s2), s2)
    d1 = conv(9, conv(8, torch.cat([up(d2), k1], -1), s1), s1)
    ref = (d1.double() @ torch.from_numpy(hw).cuda() + float(hb)).reshape(-1) * mask.double() * rms
    assert float((got.double() - ref).norm()) <= 1e-2 * float(ref.norm())
