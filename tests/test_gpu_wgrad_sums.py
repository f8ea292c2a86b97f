"""Weight gradients whose partial sums are added by warps (few elements, many splits) and by a thread
per element (few splits, or many elements)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beta", [False, True])
@pytest.mark.parametrize("Cin,Cout,B,side,KS", [(32, 32, 1, 8, 3), (32, 32, 16, 128, 3), (64, 32, 16, 64, 1), (128, 128, 2, 32, 3),
                                                (256, 256, 1, 16, 3), (128, 128, 16, 64, 3)])
def test_partial_sums(lbm, Cin, Cout, B, side, KS, beta):
    import torch
    from paper_2408_01081_gb300 import nn as K
    gen = torch.Generator(device="cuda").manual_seed(3)
    f32 = dict(dtype=torch.float32, device="cuda", generator=gen)
    x, dy = torch.randn((B, side, side, Cin), **f32), torch.randn((B, side, side, Cout), **f32)
    dw = torch.randn((Cout, KS, KS, Cin), **f32)
    ref = dw.double() if beta else torch.zeros_like(dw, dtype=torch.float64)
    for ky in range(KS):
        for kx in range(KS):
            xs = torch.roll(x, (KS // 2 - ky, KS // 2 - kx), (1, 2)).double()
            ref[:, ky, kx] += torch.einsum("byxo,byxi->oi", dy.double(), xs)
    ws = torch.empty(K.wgrad_workspace_bytes(Cin, Cout, B, side, side, KS) // 4 + 4, dtype=torch.float32, device="cuda")
    K.conv_backward_weight(dy, Cout, x, Cin, None, 0, B, side, side, KS, dw, ws, beta=beta)
    # BF16 halves of both operands without the product of the low ones: 2^-16 of each, as the other tests allow
    assert ((dw.double() - ref).norm() / ref.norm()).item() < 2e-5
