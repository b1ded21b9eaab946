"""FP32 training products of the proposal network against torch's float64
autograd on the CPU, at batches whose positions end inside a tile.  Bounds, as
for the oracle: outputs 2e-4 of their scale, loss 1e-5 relative, gradient 1e-3
in relative L2 norm per parameter block (FP32 sums of up to B 4096 products;
an activation within rounding of zero can change sides)."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
CH, HID = synth.CNN_CHANNELS, synth.CNN_HIDDEN


@pytest.fixture(scope="module")
def px():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_11313_gb300 as px
    px.load()
    return px


def _blocks(flat, k):
    shapes = []
    for i in range(5):
        shapes += [(CH[i + 1], CH[i], 3, 3), (CH[i + 1],)]
    shapes += [(HID, CH[5]), (HID,), (6 * k, HID), (6 * k,)]
    out, o = [], 0
    for s in shapes:
        n = int(np.prod(s))
        out.append(flat[o:o + n].reshape(s))
        o += n
    assert o == flat.numel()
    return out


def _operators():
    ops = []
    for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        for sg in range(8):
            m = torch.zeros(3, 3, dtype=torch.float64)
            for j in range(3):
                m[j, p[j]] = 1 - 2 * ((sg >> j) & 1)
            if torch.det(m) > 0:
                ops.append(m)
    return torch.stack(ops)


def _reference(params, imgs, q, k):
    blocks = [b.clone().requires_grad_() for b in _blocks(torch.from_numpy(params).double(), k)]
    x = torch.from_numpy(imgs).double()
    x = ((x - x.mean((1, 2), keepdim=True)) / x.std((1, 2), keepdim=True, unbiased=False))[:, None]
    for i in range(5):
        x = torch.relu(torch.nn.functional.conv2d(x, blocks[2 * i], blocks[2 * i + 1], stride=2, padding=1))
    out = torch.relu(x.mean((2, 3)) @ blocks[10].T + blocks[11]) @ blocks[12].T + blocks[13]
    a = out.reshape(-1, k, 2, 3)
    b1 = torch.nn.functional.normalize(a[:, :, 0], dim=-1)
    b2 = torch.nn.functional.normalize(a[:, :, 1] - (b1 * a[:, :, 1]).sum(-1, keepdim=True) * b1, dim=-1)
    R = torch.stack([b1, b2, torch.cross(b1, b2, dim=-1)], dim=-1)
    w, x_, y, z = torch.from_numpy(q).unbind(-1)
    Rg = torch.stack([1 - 2 * (y * y + z * z), 2 * (x_ * y - w * z), 2 * (x_ * z + w * y),
                      2 * (x_ * y + w * z), 1 - 2 * (x_ * x_ + z * z), 2 * (y * z - w * x_),
                      2 * (x_ * z - w * y), 2 * (y * z + w * x_), 1 - 2 * (x_ * x_ + y * y)], -1).reshape(-1, 3, 3)
    t = _operators()[None] @ Rg[:, None]
    d = ((R[:, :, None] - t[:, None]) ** 2).sum((3, 4)).flatten(1)
    loss, win = d.min(1)
    loss.mean().backward()
    return out.detach().numpy(), loss.mean().item(), win.numpy() // 24, [b.grad.numpy() for b in blocks]


@pytest.mark.parametrize("B,k", [(1, 1), (2, 8), (3, 5), (5, 64), (17, 8), (33, 3)])
def test_loss_and_gradient_match_float64_autograd(px, B, k):
    rng = np.random.default_rng(B)
    imgs = (rng.standard_normal((B, 128, 128)) * 3 + 20).astype(np.float32)
    q, params = synth.random_quaternions(B, B + 1), synth.cnn_init_params(k, B)
    out, loss, head, grads = _reference(params, imgs, q, k)
    ctx = px.Context()
    net = px.xcf_net_create(ctx, k, torch.from_numpy(params).cuda())
    x = torch.from_numpy(imgs).cuda()
    got = px.xcf_net_forward(ctx, net, x).cpu().numpy()
    np.testing.assert_allclose(got, out, rtol=0, atol=2e-4 * np.abs(out).max())
    l, g, w = px.xcf_net_loss_grad(ctx, net, x, torch.from_numpy(q).cuda(), want_grad=True, want_winners=True)
    np.testing.assert_allclose(l.item(), loss, rtol=1e-5)
    assert (w.cpu().numpy()[:, 0] == head).all()
    for i, (a, b) in enumerate(zip(_blocks(g.cpu().double(), k), grads)):
        assert np.linalg.norm(a.numpy() - b) <= 1e-3 * np.linalg.norm(b) + 1e-12, i
    net.close()
    ctx.close()
