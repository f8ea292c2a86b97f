"""Length of the addition chains of the one-pass ReLU mask and bias gradient."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [32, 256, 320, 512, 1024])
def test_wide_layers_add_in_short_chains(lbm, C):
    """One block's 32 pixels: 1, then halves of the unit in the last place of 1, each lost where it is
    added to that 1 alone.  In chains of 8 no more than 7 of them are, as in lbm_nn_bias_grad."""
    import torch
    from paper_2408_01081_gb300 import nn as K
    P = 32
    dy = torch.full((P, C), 2.0 ** -24, dtype=torch.float32, device="cuda")
    dy[0] = 1.0
    y = torch.ones_like(dy)
    db = torch.empty(C, dtype=torch.float32, device="cuda")
    ws = torch.empty(K.bias_grad_workspace_bytes(P, C) // 4 + 4, dtype=torch.float32, device="cuda")
    K.relu_bias_backward(dy, y, P, C, db, ws)
    lost = (1.0 + 31 * 2.0 ** -24 - db.double()) * 2.0 ** 24
    assert torch.all(lost >= 0) and torch.all(lost <= 7), lost.max().item()
