"""The training pass's count of valid rows, read 16 bytes at a time from any alignment, and its rows, tile by tile: with
all weights 0 the loss is the mean of y^2 over the valid rows, in which one row more or less shows."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def rounding_bound(n):
    # y^2 is exact, its quotient one rounding; a chain over a CTA's rows (at most 304 CTAs), 38 partial sums, 8 groups
    rows = 64 * -(-(-(-n // 64)) // 304)
    return (1 + rows + 38 + 8) * 2.0 ** -24


# less than a word, a word and its neighbours, a tile, more tiles than CTAs with a last tile of one row, two tiles a CTA
@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 65, 4097, 20545, 38912])
@pytest.mark.parametrize("shift", [0, 1, 8, 15])
def test_every_valid_row_counts_once(n, shift):
    import paper_2206_14503_gb300 as vdi

    g = torch.Generator(device="cuda").manual_seed(n + shift)
    buf = (torch.rand(n + 32, generator=g, device="cuda") > 0.2).to(torch.uint8)
    buf *= torch.randint(1, 256, (n + 32,), generator=g, device="cuda").to(torch.uint8)  # any value but 0 is valid
    valid = buf[shift:shift + n]
    valid[0] = valid[-1] = 1
    y = torch.full((n,), 2.0, device="cuda")
    y[-1] = 64.0
    x = torch.rand((n, 40), generator=g, device="cuda")
    model = torch.zeros(vdi.vdi_model_bytes(), dtype=torch.uint8, device="cuda")
    ws = vdi.Workspace(vdi.vdi_mlp_train_workspace(n))
    grad, loss = torch.zeros(vdi.vdi_model_nparams(), device="cuda"), torch.zeros(1, device="cuda")
    vdi.check(vdi.vdi_mlp_grad(model.data_ptr(), x.data_ptr(), y.data_ptr(), valid.data_ptr(), n, grad.data_ptr(),
                               loss.data_ptr(), ws.ptr, ws.nbytes), "grad")
    torch.cuda.synchronize()
    v = valid.ne(0).double()
    m = float(v.sum())
    tol = rounding_bound(n)
    # a row of y = 2 more or less in the sum, or one in the count, is well beyond the bound
    assert 2 * tol * float((y.double() ** 2 * v).sum()) < 4.0 and 2 * tol * m < 1.0
    want = float((y.double() ** 2 * v).sum()) / m
    assert abs(float(loss) - want) <= tol * want
    db = -2.0 * float((y.double() * v).sum()) / m
    assert abs(float(grad[-1]) - db) <= tol * abs(db)
    assert not grad[:-1].any()
