"""The row handling of the fused injection and dX epilogues and of the injection
backward: every token of X_out and dX is written exactly where it belongs, at
sizes where rows and columns end inside tiles.  Block 0 of a causal sequence
receives nothing, so there X_out equals X bit for bit, and a canary after the
last token must stay as it was; the rest is held to the layer's usual bars."""
import pytest
import torch

import paper_2608_23463_gb300 as pf
import pf_synth as S
from oracle import layer as OL
from paper_2608_23463_gb300.layer import ProxyLayer, to_device
from tests._util import assert_grad_close

pytestmark = pytest.mark.gpu

SPECS = {
    # one row; rows end inside an 8-row group, a 32-row warp and a 128-row tile
    "one_block": S.LayerSpec(batch=1, L=16, d=64, n_heads=1, P=16),
    "b3_ragged_k1_8": S.LayerSpec(batch=3, L=333, d=64, n_heads=1, P=32, levels=2, k1=8, k2=4),
    "b5_last_block_one_token": S.LayerSpec(batch=5, L=8 * 13 + 1, d=128, n_heads=2, P=8),
    # 192 columns: of the second 128-column tile only one half of the warps has any
    "narrow_tokens": S.LayerSpec(batch=2, L=77, d=128, n_heads=2, P=3, d_fine=64),
    # 256-wide tiles on CTA pairs, two ragged sequences, the row count not a multiple of 256
    "pairs_b2_ragged": S.LayerSpec(batch=2, L=9001, d=1024, n_heads=16, P=64, levels=2, k1=8, k2=8),
    "pairs_add_bidir": S.LayerSpec(batch=1, L=12000, d=1024, n_heads=16, P=64, levels=2, k1=8, k2=8,
                                   mode=S.BIDIR_1D, inject=S.INJ_ADD),
    # 320 and 448 columns of 256-wide tiles: the last tile's warps find 64 columns of 256, or
    # one half whole and the other half of theirs, and fetch the next tile's rows past that
    "pairs_last_64": S.LayerSpec(batch=1, L=99998, d=64, n_heads=1, P=5, interact=S.F_IDENTITY),
    "pairs_last_192": S.LayerSpec(batch=2, L=70000, d=64, n_heads=1, P=7, mode=S.BIDIR_1D,
                                  inject=S.INJ_ADD, interact=S.F_IDENTITY),
}


@pytest.mark.parametrize("name", list(SPECS))
def test_rows_of_x_out_and_dx(name):
    spec = SPECS[name]
    inp = S.make_layer_inputs(spec, 40 + len(name))
    lay = ProxyLayer(spec, inp)
    X, G = to_device(inp["X"], torch.bfloat16), to_device(inp["G"], torch.bfloat16)
    n = X.numel()
    bufs = [torch.full((n + 4096,), float("nan"), dtype=torch.bfloat16, device="cuda")
            for _ in range(2)]
    for b in bufs:
        b[n:] = 7.0
    Xo, dX = (b[:n].view(X.shape) for b in bufs)
    lay.forward(X, X_out=Xo)
    lay.backward(X, G, dX=dX)
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    for b in bufs:
        assert bool((b[n:] == 7.0).all())
    if spec.mode == S.CAUSAL_1D:
        assert torch.equal(Xo[:, :spec.P], X[:, :spec.P])
    ref, _ = OL.layer_fwd(spec, inp, inp["X"])
    rdX, _, _ = OL.layer_bwd(spec, inp, inp["X"], inp["G"])
    assert_grad_close("X_out", Xo.float().cpu().numpy(), ref)
    assert_grad_close("dX", dX.float().cpu().numpy(), rdX)
