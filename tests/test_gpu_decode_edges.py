"""The merge of a decode step's partials at the edges of its register windows (64
open keys, 64 splits) and key passes (32 keys)."""
import pytest
import torch

import paper_2608_23463_gb300 as pf
import pf_synth as S
from oracle import decode as OD
from paper_2608_23463_gb300.decode import ProxyKVCache
from tests._util import assert_close, assert_grad_close

pytestmark = pytest.mark.gpu


# one sequence of 1040 rows: 65 splits; three of 300: at most 18
@pytest.mark.parametrize("dh", [64, 128])
@pytest.mark.parametrize("capacity,n_proxy,n_open", [
    (1040, [1040], [255]), (1024, [1024], [63]), (300, [0, 1, 17], [0, 31, 32]),
    (300, [300, 299, 0], [62, 64, 200])])
def test_step_at_window_edges(dh, capacity, n_proxy, n_open):
    B = len(n_proxy)
    spec = S.DecodeSpec(batch=B, d=384, n_heads=384 // dh, P=256, capacity=capacity)
    prm = S.make_decode_params(spec, 11)
    st = S.make_decode_state(spec, 12, n_proxy, n_open)
    y = ProxyKVCache(spec, prm, st).step(torch.from_numpy(st["x"]).to("cuda", torch.bfloat16))
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    ref, _ = OD.decode_step(spec, prm, st)
    y = y.float().cpu().numpy()
    assert_close("y", y, ref)
    assert_grad_close("y - x", y - st["x"], ref - st["x"])
