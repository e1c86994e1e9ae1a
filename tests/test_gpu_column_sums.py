"""Bias and gate gradients, which are column sums over row chunks: row counts on
both sides of every split of the sum over chunks, threads and warps."""
import numpy as np
import pytest
import torch

import paper_2608_23463_gb300 as pf
import pf_synth as S
from oracle import layer as OL
from paper_2608_23463_gb300.layer import ProxyLayer, to_device
from tests._util import assert_grad_close

pytestmark = pytest.mark.gpu

# blocks: 16 | 17 and 256 | 257 change the warps per column, 256 | 257 the passes
ROWS = [1, 16, 17, 33, 256, 257, 1100]


# 2048 columns: by registers | streamed, 64 rows to each of 304 chunks, then ragged.  Slices
# of 2048 columns: 64 fill 256 of 304 places, by registers; 76 fill all, streamed
@pytest.mark.parametrize("rows,P", [(r, 8) for r in ROWS] +
                         [(19455, 32), (19456, 32), (19500, 32), (257, 2048), (255, 2432),
                          (256, 2432), (257, 2432)])
def test_bias_gradient_is_the_exact_sum(rows, P):
    """Add injection: the gradient of b_d1 at token t of a block is the sum of G over
    the blocks.  G holds whole numbers of at most 8, so the sum is exact."""
    spec = S.LayerSpec(batch=1, L=P * rows, d=64, n_heads=1, P=P, mode=S.BIDIR_1D,
                       inject=S.INJ_ADD)
    inp = S.make_layer_inputs(spec, rows)
    G = np.random.default_rng(rows).integers(-8, 9, (1, spec.L, 64)).astype(np.float32)
    lay = ProxyLayer(spec, inp)
    X = to_device(inp["X"], torch.bfloat16)
    lay.forward(X)
    lay.backward(X, to_device(G, torch.bfloat16))
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    want = G.reshape(rows, P * 64).sum(0)
    assert np.array_equal(lay.grads["b_d1"].cpu().numpy().ravel(), want)


@pytest.mark.parametrize("rows", ROWS[1:])
def test_gate_and_bias_gradients_match_oracle(rows):
    # 192 token columns a block: 1.5 warps of the widest column group
    spec = S.LayerSpec(batch=1, L=3 * rows - 1, d=128, n_heads=2, P=3, d_fine=64)
    inp = S.make_layer_inputs(spec, 60 + rows)
    lay = ProxyLayer(spec, inp)
    X, G = to_device(inp["X"], torch.bfloat16), to_device(inp["G"], torch.bfloat16)
    lay.forward(X)
    lay.backward(X, G)
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    _, _, grads = OL.layer_bwd(spec, inp, inp["X"], inp["G"])
    for k in ("b_d1", "b_c1", "w_x", "w_dlt", "b_g"):
        assert_grad_close("grad " + k, lay.grads[k].float().cpu().numpy(), grads[k])
