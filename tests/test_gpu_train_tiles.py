"""The training kernels' tiles: 64 rows a tile, several tiles a CTA once there are more tiles than resident CTAs,
and a valid-row count read 16 bytes at a time from any alignment; against autograd in 64 bits."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = ((64, 40), (64,), (64, 64), (64,), (64,), (1,))


def _reference(theta, x, y, valid):
    """(loss, gradient, the gradient with every term's absolute value: the scale of its rounding errors)"""
    w = theta.bfloat16().double()
    parts, at = [], 0
    for s in SHAPES:
        parts.append(w[at:at + math.prod(s)].view(s).clone().requires_grad_(True))
        at += math.prod(s)
    W1, b1, W2, b2, w3, b3 = parts
    x, y, v = x.double(), y.double(), valid.ne(0).double()
    m = v.sum().clamp(min=1.0)
    p1 = x @ W1.t() + b1
    h1 = torch.relu(p1)
    p2 = h1 @ W2.t() + b2
    h2 = torch.relu(p2)
    d = (h2 @ w3 + b3 - y) * v
    loss = (d * d).sum() / m
    loss.backward()
    grad = torch.cat([p.grad.reshape(-1) for p in parts])
    with torch.no_grad():
        dy = ((h2.abs() @ w3.abs() + b3.abs() + y.abs()) * v * 2 / m)[:, None]
        d2 = dy * w3.abs() * (p2 > 0)
        d1 = (d2 @ W2.abs()) * (p1 > 0)
        H1 = x.abs() @ W1.abs().t() + b1.abs()
        H2 = H1 @ W2.abs().t() + b2.abs()
        scale = torch.cat([(d1.t() @ x.abs()).reshape(-1), d1.sum(0), (d2.t() @ H1).reshape(-1), d2.sum(0),
                           (dy * H2).sum(0), dy.sum(0)])
        lscale = (dy[:, 0] * (h2.abs() @ w3.abs() + b3.abs() + y.abs())).sum()
    return loss.detach(), grad, scale, lscale


# a row, one short of a tile, a tile, one over, and more tiles than two CTAs on each of 160 SMs hold
@pytest.mark.parametrize("n", [1, 63, 64, 65, 20545])
@pytest.mark.parametrize("shift", [0, 3])
def test_gradient_tiles(n, shift):
    import paper_2206_14503_gb300 as vdi

    g = torch.Generator(device="cuda").manual_seed(1000 + n)
    x = torch.rand((n, 40), generator=g, device="cuda") * 2 - 0.5
    y = torch.randn(n, generator=g, device="cuda")
    buf = (torch.rand(n + 16, generator=g, device="cuda") > 0.2).to(torch.uint8) * 200
    valid = buf[shift:shift + n]
    model = torch.zeros(vdi.vdi_model_bytes(), dtype=torch.uint8, device="cuda")
    vdi.check(vdi.vdi_model_init(model.data_ptr(), 5), "init")
    theta = model[:4 * vdi.vdi_model_nparams()].view(torch.float32).clone()
    ws = vdi.Workspace(vdi.vdi_mlp_train_workspace(n))
    grad = torch.zeros(vdi.vdi_model_nparams(), device="cuda")
    loss = torch.zeros(1, device="cuda")
    vdi.check(vdi.vdi_mlp_grad(model.data_ptr(), x.data_ptr(), y.data_ptr(), valid.data_ptr(), n, grad.data_ptr(),
                               loss.data_ptr(), ws.ptr, ws.nbytes), "grad")
    torch.cuda.synchronize()
    ref_loss, ref, scale, lscale = _reference(theta, x, y, valid)
    # a chain of at most 40 + 64 + 64 forward and backward terms, 64 rows a tile for a few tiles and the partial
    # sums: under 500 roundings of 2^-24 on the terms' absolute sums; and, among many rows, one activation whose
    # sign its rounding decides
    tol = 500 * 2.0 ** -24 + (1.0 / n if n > 1000 else 0.0)
    assert float((loss[0].double() - ref_loss).abs()) <= tol * float(lscale)
    assert bool(((grad.double() - ref).abs() <= tol * scale + 1e-30).all())
