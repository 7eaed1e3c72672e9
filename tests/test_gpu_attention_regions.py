"""Bf16 attention at the edges of its kernels: the last short key range at head
dim 64 and the first long one, tiles that just fill or overflow, one and two
tiles per item on CTAs with several items, and rows whose max grows from tile
to tile, so that the reference moves after P was formed, with the items of
a partial last wave whole and, with a workspace, split along their keys."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DEV = "cuda"


@pytest.fixture(scope="module")
def acid():
    import __graft_entry__ as g

    g.build()
    from paper_2607_12358_gb300 import acid as a

    return a


@pytest.mark.parametrize("nq,nk,heads,hd", [
    (1, 1, 2, 64), (130, 63, 3, 64), (257, 65, 2, 64), (3000, 64, 30, 64), (700, 448, 4, 64), (700, 449, 4, 64),
    (129, 512, 3, 64), (5000, 513, 10, 64), (900, 1000, 2, 64), (2600, 2600, 16, 64),
    (3000, 128, 14, 128), (5000, 129, 9, 128), (1300, 1025, 3, 128), (2600, 2600, 16, 128)])
@pytest.mark.parametrize("grow", [0.0, 60.0])
def test_attention_regions(acid, nq, nk, heads, hd, grow):
    g = torch.Generator(device=DEV).manual_seed(nq + nk)
    q, k, v = (torch.randn(n, heads * hd, device=DEV, generator=g, dtype=torch.float32).to(torch.bfloat16)
               for n in (nq, nk, nk))
    if grow:  # scores of the even rows rise by `grow` nats along the keys, those of the odd rows fall
        sign = 1.0 - 2.0 * (torch.arange(nq, device=DEV, dtype=torch.float32) % 2)
        q.view(nq, heads, hd)[:, :, 0] = (sign * hd ** 0.5)[:, None].to(torch.bfloat16)
        ramp = torch.linspace(0.0, grow, nk, device=DEV, dtype=torch.float32)
        k.view(nk, heads, hd)[:, :, 0] = ramp[:, None].to(torch.bfloat16)
    ws = torch.empty(acid.attention_workspace_size(hd), dtype=torch.uint8, device=DEV)
    outs = [acid.acid_attention_forward(q, k, v, heads, workspace=w).double() for w in (None, ws)]
    acid.check_device_error()
    for h in (0, heads - 1):  # the last head's items are in the last wave
        c = slice(h * hd, (h + 1) * hd)
        w = torch.softmax(q[:, c].double() @ k[:, c].double().T / hd ** 0.5, dim=1)
        ref = w @ v[:, c].double()
        # weights round to bf16 (2^-9) before P V; fp32 scores of magnitude up to
        # grow + 10 carry 2^-24 of it into the exponent; the output rounds once more
        tol = (2.0 ** -8 + (grow + 10.0) * 2.0 ** -20) * (w @ v[:, c].double().abs()) + 2.0 ** -8 * ref.abs() + 1e-6
        for got in outs:
            assert torch.all((got[:, c] - ref).abs() <= tol)
