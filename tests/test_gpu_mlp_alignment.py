"""BF16 weights that do not start on a 4-byte word are loaded one at a time, not by word copies."""
import pytest

from paper_2105_01722_gb300 import gdg, learned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 2, 17, 64])
def test_weights_on_an_odd_halfword(rows):
    """Forward, backward and Adam: the bits of aligned weights."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(3)
    X = torch.randn(rows, gdg.MLP_IN, device="cuda", generator=g)
    T = torch.randn(rows, gdg.MLP_OUT, device="cuda", generator=g)
    out = []
    for shift in (0, 1):
        net = gdg.Mlp(learned.glorot_params(7))
        room = torch.zeros(gdg.MLP_NWEIGHT + 2, dtype=torch.int16, device="cuda")
        weights = room[shift : shift + gdg.MLP_NWEIGHT]
        weights.copy_(net.wbf16)
        net.wbf16 = weights
        assert weights.data_ptr() % 4 == 2 * shift
        Y = torch.empty(rows, gdg.MLP_OUT, device="cuda")
        net.forward(X, Y)
        loss = net.backward(X, T).clone()
        net.adam(1e-3)
        assert int(room[0]) == 0 or shift == 0        # nothing written before the weights, or behind them
        assert int(room[-1]) == 0
        out.append([Y, loss, net.grad, net.params, net.wbf16.clone()])
    for a, b in zip(*out):
        assert torch.equal(a, b)
