"""Split contractions: weight gradients and compressions whose output is a few
tiles and whose K is long run in K slices on CTA pairs or single CTAs, with as
many slices as their scratch allows.  Weight gradients and proxies are held to the
oracle, also where the allocation-free entry's fixed scratch leaves fewer slices than
the cheapest plan wants."""
import pytest
import torch

import paper_2608_23463_gb300 as pf
import pf_synth as S
from oracle import layer as OL
from paper_2608_23463_gb300.layer import ProxyLayer, to_device
from tests._util import assert_close, assert_grad_close

pytestmark = pytest.mark.gpu

# K = P d for the compression (M = L / P rows), K = L / k1 for the weight gradients
SPECS = {
    # M = 47 rows x N = 192: single CTAs, ragged N tile; K = 24576
    "few_rows": S.LayerSpec(batch=1, L=47 * 128, d=192, n_heads=3, P=128),
    # pairs with a ragged M tile (300 rows), K = 32768 for the compression
    "pairs_ragged_m": S.LayerSpec(batch=1, L=300 * 64, d=512, n_heads=8, P=64),
    # long K (rows) for the weight gradients, the last K block partly filled
    "long_k": S.LayerSpec(batch=3, L=8191, d=256, n_heads=4, P=4, levels=2, k1=2, k2=2),
}


@pytest.mark.parametrize("name", list(SPECS))
def test_split_contractions(name):
    spec = SPECS[name]
    inp = S.make_layer_inputs(spec, 90 + len(name))
    lay = ProxyLayer(spec, inp)
    X, G = to_device(inp["X"], torch.bfloat16), to_device(inp["G"], torch.bfloat16)
    H = lay.empty_proxy()
    Xo = lay.forward(X, H_out=H)
    dX = lay.backward(X, G)
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    ref, rH = OL.layer_fwd(spec, inp, inp["X"])
    rdX, _, rg = OL.layer_bwd(spec, inp, inp["X"], inp["G"])
    assert_close("H_out", H.cpu().numpy(), rH)
    assert_grad_close("X_out", Xo.float().cpu().numpy(), ref)
    assert_grad_close("dX", dX.float().cpu().numpy(), rdX)
    for k, v in rg.items():
        assert_grad_close("grad " + k, lay.grads[k].cpu().numpy(), v)


# layers whose other buffers leave less scratch than their plans want: their workspace is
# the limit to the byte (14.8 to 16.0 MiB with the fewest slices)
CUT = {
    "cut_mlp": S.LayerSpec(batch=1, L=1029, d=1024, n_heads=16, P=2, mode=S.BIDIR_1D, d_fine=64,
                           interact=S.F_MLP),
    "cut_add_2lvl": S.LayerSpec(batch=3, L=1158, d=640, n_heads=10, P=48, levels=2, k1=1, k2=48,
                                mode=S.BIDIR_1D, inject=S.INJ_ADD, d_fine=64),
    "cut_identity": S.LayerSpec(batch=1, L=1408, d=640, n_heads=10, P=128, inject=S.INJ_ADD,
                                interact=S.F_IDENTITY),
    "cut_gated_2lvl": S.LayerSpec(batch=3, L=1106, d=640, n_heads=10, P=32, levels=2, k1=1, k2=32,
                                  d_fine=64),
}
ROOMY = {f"roomy_d{d}_P{P}": S.LayerSpec(batch=2, L=L, d=d, n_heads=d // 64, P=P)
         for L, P, d in [(1000, 16, 128), (4000, 16, 64), (900, 8, 192), (300, 64, 256)]}


@pytest.mark.parametrize("name", list(ROOMY) + list(CUT))
def test_small_layers_still_fit_the_fixed_scratch(name):
    """The split scratch of a backward gives way to the allocation-free entry's limit, and
    its products take the slices that are left."""
    spec = {**ROOMY, **CUT}[name]
    need = pf.proxy_layer_workspace_size(pf.layer_desc(spec), 1)
    if name in CUT:
        assert need == pf.PF_NOALLOC_SCRATCH_BYTES
    else:
        assert need < pf.PF_NOALLOC_SCRATCH_BYTES
    inp = S.make_layer_inputs(spec, 5)
    lay = ProxyLayer(spec, inp)
    X, G = to_device(inp["X"], torch.bfloat16), to_device(inp["G"], torch.bfloat16)
    st = torch.cuda.current_stream().cuda_stream
    lay.forward(X)
    dX = lay.backward(X, G)
    ref = {k: v.clone() for k, v in lay.grads.items()}
    dX2 = torch.empty_like(dX)
    pf.proxy_layer_bwd_noalloc(lay.desc, lay.p_struct, X, None, None, lay.saved, G, None, dX2, None,
                               lay.g_struct, st)
    pf.pf_sync_check(st)
    assert torch.equal(dX, dX2)
    assert all(torch.equal(ref[k], lay.grads[k]) for k in ref)
    if name in CUT:
        _, _, rg = OL.layer_bwd(spec, inp, inp["X"], inp["G"])
        for k, v in rg.items():
            assert_grad_close("grad " + k, lay.grads[k].cpu().numpy(), v)
