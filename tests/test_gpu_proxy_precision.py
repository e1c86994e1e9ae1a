"""The proxies of a one-level compression against float64: their inputs are exact, so
what the sum over K loses is all of the error.  Each MMA adds 16 products and cuts the
sum off at the accumulator's last bit, half a unit on average, so that a slice of n
MMAs loses at most n 2^-25 of its largest partial sum.  The slices may be no deeper
than those that fill 152 SMs with 128 x 128 tiles, at sizes where larger tiles on
fewer slices would be cheaper."""
import pytest
import torch

import paper_2608_23463_gb300 as pf
import pf_synth as S
from paper_2608_23463_gb300.layer import ProxyLayer, to_device

pytestmark = pytest.mark.gpu

SPECS = {  # MMAs of the deepest slice: rows x width tiles, K = P d in blocks of 64
    # 3360 x 256: 54 tiles on 14 slices, 256 blocks
    "d256": (S.LayerSpec(batch=1, L=3360 * 64, d=256, n_heads=4, P=64), 4 * 19),
    # 3624 x 512: 116 tiles on 13 slices, 256 blocks; ragged
    "d512": (S.LayerSpec(batch=1, L=3624 * 32 - 5, d=512, n_heads=8, P=32), 4 * 20),
    # 2565 x 384: 63 tiles on 12 slices, 384 blocks; the image layer's patches
    "image": (S.LayerSpec(batch=3, L=152 * 360, d=384, n_heads=6, P=64, mode=S.BIDIR_2D,
                          inject=S.INJ_AFFINE, grid_h=152, grid_w=360, patch=8), 4 * 32),
}


@pytest.mark.parametrize("name", list(SPECS))
def test_proxies_against_float64(name):
    spec, mmas = SPECS[name]
    inp = S.make_layer_inputs(spec, 7)
    lay = ProxyLayer(spec, inp)
    X = to_device(inp["X"], torch.bfloat16)
    t = to_device(inp["t"], torch.float32) if spec.patch else None
    H = lay.empty_proxy()
    lay.forward(X, None, t, H_out=H, train=False)
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    p, B, P, d = spec.patch, spec.batch, spec.P, spec.d
    if p:
        blocks = X.view(B, spec.grid_h // p, p, spec.grid_w // p, p, d).transpose(2, 3)
    else:
        blocks = torch.nn.functional.pad(X, (0, 0, 0, spec.m * P - spec.L))
    ref = blocks.reshape(B * spec.m, P * d).double() @ lay.params["W_c1"].double().T
    ref += lay.params["b_c1"].double()
    err = ((H.view_as(ref).double() - ref).norm() / ref.norm()).item()
    assert err <= mmas * 2.0 ** -25, err
