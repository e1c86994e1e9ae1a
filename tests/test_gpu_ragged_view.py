"""A single ragged sequence is compressed in place: blocks that end inside a row, a
tile or a 64-row step, sequences shorter than a row.  X is followed by NaN, which
must reach no output or gradient."""
import pytest
import torch

import paper_2608_23463_gb300 as pf
import pf_synth as S
from oracle import layer as OL
from paper_2608_23463_gb300.layer import ProxyLayer, to_device
from tests._util import assert_close, assert_grad_close

pytestmark = pytest.mark.gpu

SPECS = {
    "one_token": S.LayerSpec(batch=1, L=1, d=64, n_heads=1, P=4),
    "shorter_than_a_row": S.LayerSpec(batch=1, L=5, d=128, n_heads=2, P=16),
    "row_and_one": S.LayerSpec(batch=1, L=17, d=128, n_heads=2, P=16),
    "whole_rows_partial_block": S.LayerSpec(batch=1, L=1016, d=128, n_heads=2, P=32, levels=2,
                                            k1=8, k2=4),
    "row_128_ends_late": S.LayerSpec(batch=1, L=129 * 8 - 1, d=64, n_heads=1, P=8),
    "tokens_of_64": S.LayerSpec(batch=1, L=2003, d=512, n_heads=8, P=64, d_fine=64),
    "sliced_k": S.LayerSpec(batch=1, L=9001, d=512, n_heads=8, P=64),
    "pairs": S.LayerSpec(batch=1, L=20003, d=1024, n_heads=16, P=64, levels=2, k1=8, k2=8),
}


@pytest.mark.parametrize("name", list(SPECS))
def test_ragged_sequence_in_place(name):
    spec = SPECS[name]
    inp = S.make_layer_inputs(spec, 20 + len(name))
    lay = ProxyLayer(spec, inp)
    src, G = to_device(inp["X"], torch.bfloat16), to_device(inp["G"], torch.bfloat16)
    n = src.numel()
    buf = torch.full((n + 256 * spec.P * 64,), float("nan"), dtype=torch.bfloat16, device="cuda")
    X = buf[:n].view(src.shape)
    X.copy_(src)
    H = lay.empty_proxy()
    Xo = lay.forward(X, H_out=H)
    dX = lay.backward(X, G)
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    f = lambda t: t.float().cpu().numpy()
    rX, rH = OL.layer_fwd(spec, inp, inp["X"])
    rdX, _, grads = OL.layer_bwd(spec, inp, inp["X"], inp["G"])
    assert_close("H_out", f(H), rH)
    assert_grad_close("X_out", f(Xo), rX)
    assert_grad_close("dX", f(dX), rdX)
    assert_grad_close("W_c1", f(lay.grads["W_c1"]), grads["W_c1"])
