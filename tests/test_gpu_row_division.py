"""Fused epilogues find each row's place by multiplications instead of divisions:
divisors that are 1, powers of two, odd, and one past a power of two, against the
places that the layer's output must have."""
import pytest
import torch

import paper_2608_23463_gb300 as pf
import pf_synth as S
from oracle import layer as OL
from paper_2608_23463_gb300.layer import ProxyLayer, to_device
from tests._util import assert_grad_close

pytestmark = pytest.mark.gpu

SPECS = {
    # blocks per sequence m, level-2 rows k2: 1, 33, 17, 65 with 1, 3, 4, 5
    "m1_k1": S.LayerSpec(batch=9, L=6, d=64, n_heads=1, P=8),
    "m33_k3": S.LayerSpec(batch=3, L=33 * 12 - 5, d=64, n_heads=1, P=12, levels=2, k1=4, k2=3),
    "m17_k5": S.LayerSpec(batch=2, L=17 * 10, d=192, n_heads=3, P=10, levels=2, k1=2, k2=5),
    "m65_k4": S.LayerSpec(batch=4, L=65 * 8 - 7, d=64, n_heads=1, P=8, levels=2, k1=2, k2=4),
}


@pytest.mark.parametrize("name", list(SPECS))
def test_rows_land_in_their_tokens(name):
    spec = SPECS[name]
    inp = S.make_layer_inputs(spec, 70 + len(name))
    lay = ProxyLayer(spec, inp)
    X, G = to_device(inp["X"], torch.bfloat16), to_device(inp["G"], torch.bfloat16)
    Xo = lay.forward(X)
    dX = lay.backward(X, G)
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    ref, _ = OL.layer_fwd(spec, inp, inp["X"])
    rdX, _, _ = OL.layer_bwd(spec, inp, inp["X"], inp["G"])
    assert_grad_close("X_out", Xo.float().cpu().numpy(), ref)
    assert_grad_close("dX", dX.float().cpu().numpy(), rdX)
