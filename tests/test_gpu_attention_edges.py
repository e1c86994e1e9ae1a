"""Attention forward and backward at proxy and token counts around its 128-row tiles and
128-column steps: one row, one short of, at and past a tile, several tiles; causal
and bidirectional proxies, and tokens against proxies (cross injection) where
block boundaries fall inside tiles and steps."""
import pytest
import torch

import paper_2608_23463_gb300 as pf
import pf_synth as S
from oracle import layer as OL
from paper_2608_23463_gb300.layer import ProxyLayer, to_device
from tests._util import BF16_MAX_TOL, BF16_TOL, CROSS_MAX_TOL, CROSS_TOL, assert_grad_close

pytestmark = pytest.mark.gpu


def _check(spec, seed, tol, max_tol):
    inp = S.make_layer_inputs(spec, seed, with_h_in=True)
    lay = ProxyLayer(spec, inp)
    X, G = to_device(inp["X"], torch.bfloat16), to_device(inp["G"], torch.bfloat16)
    H_in = to_device(inp["H_in"], torch.float32)
    dH = lay.empty_proxy()
    lay.forward(X, H_in)
    dX = lay.backward(X, G, H_in, dH_in=dH)
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    rdX, rdH, rg = OL.layer_bwd(spec, inp, inp["X"], inp["G"], inp["H_in"])
    assert_grad_close("dX", dX.float().cpu().numpy(), rdX, tol, max_tol)
    assert_grad_close("dH_in", dH.cpu().numpy(), rdH, tol, max_tol)
    for k in ("W_qkv",) + (("W_qa", "W_kvx") if spec.inject == S.INJ_CROSS else ()):
        assert_grad_close("grad " + k, lay.grads[k].cpu().numpy(), rg[k], tol, max_tol)


@pytest.mark.parametrize("mode", [S.CAUSAL_1D, S.BIDIR_1D])
@pytest.mark.parametrize("m", [2, 127, 128, 129, 300])
def test_proxy_attention_backward_edges(m, mode):
    # two proxies: rounding the oracle's intermediates to bf16 moves the gradient of W_qkv by
    # 1.0e-2 (RMS) and 1.1e-1 (max), past the layer's bars' margin; the cross injection's are
    # about twice that.  From 127 proxies on it is 8.5e-3 and 7.5e-2 in any gradient.
    spec = S.LayerSpec(batch=2, L=4 * m - 1, d=128, n_heads=2, P=4, mode=mode)
    if m == 2:
        _check(spec, m, CROSS_TOL, CROSS_MAX_TOL)
    else:
        _check(spec, m, BF16_TOL, BF16_MAX_TOL)


@pytest.mark.parametrize("L,P,mode", [(129, 1, S.CAUSAL_1D), (257, 3, S.CAUSAL_1D),
                                      (1000, 7, S.CAUSAL_1D), (520, 130, S.CAUSAL_1D),
                                      (385, 3, S.BIDIR_1D)])
def test_cross_attention_backward_edges(L, P, mode):
    spec = S.LayerSpec(batch=2, L=L, d=128, n_heads=2, P=P, mode=mode, inject=S.INJ_CROSS)
    _check(spec, L, CROSS_TOL, CROSS_MAX_TOL)


# one sequence ends inside a tile and another follows it: no row may spill over
@pytest.mark.parametrize("train", [True, False])
@pytest.mark.parametrize("L,P,inject", [(4 * 129 - 1, 4, S.INJ_GATED), (4 * 256, 4, S.INJ_GATED),
                                        (129, 1, S.INJ_CROSS), (391, 3, S.INJ_CROSS),
                                        (520, 130, S.INJ_CROSS), (100, 101, S.INJ_CROSS)])
def test_attention_forward_edges(L, P, inject, train):
    spec = S.LayerSpec(batch=3, L=L, d=128, n_heads=2, P=P, inject=inject)
    inp = S.make_layer_inputs(spec, L)
    lay = ProxyLayer(spec, inp)
    Xo = lay.forward(to_device(inp["X"], torch.bfloat16), train=train)
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    ref, _ = OL.layer_fwd(spec, inp, inp["X"])
    assert_grad_close("X_out", Xo.float().cpu().numpy(), ref)


# 64 proxies and 192 tokens: a 128-row step ends in the sequence that follows
@pytest.mark.parametrize("mode", [S.CAUSAL_1D, S.BIDIR_1D])
@pytest.mark.parametrize("L,P,inject", [(256, 4, S.INJ_GATED), (192, 3, S.INJ_CROSS)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_sequence_keeps_its_gradients_beside_a_bad_one(L, P, inject, mode, bad):
    spec = S.LayerSpec(batch=2, L=L, d=128, n_heads=2, P=P, mode=mode, inject=inject)
    inp = S.make_layer_inputs(spec, 31)
    lay = ProxyLayer(spec, inp)
    X, G = to_device(inp["X"], torch.bfloat16), to_device(inp["G"], torch.bfloat16)
    lay.forward(X)
    got = []
    for fill in (None, bad):
        if fill is not None:
            G[1] = fill
        dH = lay.empty_proxy()
        got.append((lay.backward(X, G, dH_in=dH), dH))
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    for clean, dirty in zip(*got):
        assert torch.equal(clean[0], dirty[0])
        assert not torch.isfinite(dirty[1]).all()


# token tau sees none of the proxies from block n on: block 0 sees none (n = 0), block 128 those of
# the first 128-key tile only
@pytest.mark.parametrize("L,P,tau,n", [(1144, 200, 0, 0), (1144, 200, 130, 0), (1144, 200, 199, 0),
                                       (14000, 100, 12810, 128), (14000, 100, 12899, 128)])
def test_a_bad_token_leaves_the_proxies_it_does_not_see(L, P, tau, n):
    spec = S.LayerSpec(batch=1, L=L, d=128, n_heads=2, P=P, inject=S.INJ_CROSS,
                       interact=S.F_IDENTITY)
    inp = S.make_layer_inputs(spec, 37)
    lay = ProxyLayer(spec, inp)
    X, G = to_device(inp["X"], torch.bfloat16), to_device(inp["G"], torch.bfloat16)
    lay.forward(X)
    got = []
    for bad in (False, True):
        if bad:
            G[0, tau] = float("nan")
        dH = lay.empty_proxy()
        lay.backward(X, G, dH_in=dH)
        got.append(dH[0, n:])
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    assert torch.equal(*got)
