"""2D layer at sizes where its token and timestep kernels end inside a warp's or
a CTA's share: token counts that are not a multiple of a warp's tokens, patches
that are not a multiple of a CTA's, widths that fill part of a warp's lanes,
rectangular grids, 1 x 1 patches."""
import numpy as np
import pytest
import torch

import paper_2608_23463_gb300 as pf
import pf_synth as S
from oracle import layer as OL
from paper_2608_23463_gb300.layer import ProxyLayer, to_device
from tests._util import assert_grad_close, rms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,gh,gw,d,patch", [(1, 5, 7, 128, 1), (3, 6, 10, 384, 2),
                                                  (2, 66, 34, 256, 2), (1, 8, 24, 512, 8)])
def test_layer2d_edge_sizes(batch, gh, gw, d, patch):
    spec = S.LayerSpec(batch=batch, L=gh * gw, d=d, n_heads=d // 64, P=patch * patch,
                       mode=S.BIDIR_2D, inject=S.INJ_AFFINE, grid_h=gh, grid_w=gw, patch=patch)
    inp = S.make_layer_inputs(spec, 300 + gh)
    lay = ProxyLayer(spec, inp)
    X, G = to_device(inp["X"], torch.bfloat16), to_device(inp["G"], torch.bfloat16)
    t = to_device(inp["t"], torch.float32)
    Xo = lay.forward(X, None, t)
    dX = lay.backward(X, G, None, t)
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    ref, _ = OL.layer_fwd(spec, inp, inp["X"], None, inp["t"])
    rdX, _, rg = OL.layer_bwd(spec, inp, inp["X"], inp["G"], None, inp["t"])
    assert_grad_close("X_out", Xo.float().cpu().numpy(), ref)
    assert_grad_close("dX", dX.float().cpu().numpy(), rdX)
    # W_t2's gradient is sum_b dgb_b u_b^T: an error of dgb within the bar's 1e-1 RMS comes
    # out of it times |u_i| / RMS(u), and likewise W_t1's times |e_k| / RMS(e)
    tcs = [OL.adaln_params(float(tb), inp)[2] for tb in inp["t"]]
    peak = {f: max(abs(c[f]).max() for c in tcs) / rms(np.stack([c[f] for c in tcs]))
            for f in ("u", "e")}
    for k, f in (("b_d1", 1.0), ("W_t1", peak["e"]), ("b_t1", 1.0), ("W_t2", peak["u"]),
                 ("b_t2", 1.0)):
        assert_grad_close("grad " + k, lay.grads[k].cpu().numpy(), rg[k], max_tol=1e-1 * f)
