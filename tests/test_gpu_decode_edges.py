"""The merge of a decode step's partials at the edges of its register windows (64
open keys, 64 splits) and key passes (32 keys), and the K/V rows of an append and a
prefill around 8 rows to a pass and 16 rows to the tiled product."""
import numpy as np
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


@pytest.mark.parametrize("batch", [1, 8, 9, 16, 17])
def test_append_rows(batch):
    """Every second sequence has no full block: it is flagged and its cache stays."""
    spec = S.DecodeSpec(batch=batch, d=192, n_heads=3, P=4, capacity=5)
    prm = S.make_decode_params(spec, 13)
    n_open = [4 if b % 2 == 0 else 1 for b in range(batch)]
    st = S.make_decode_state(spec, 14, [b % 5 for b in range(batch)], n_open)
    cache = ProxyKVCache(spec, prm, st)
    before = {k: cache.s[k].clone() for k in ("K_proxy", "V_proxy")}
    H = np.random.default_rng(15).standard_normal((batch, 192)).astype(np.float32)
    cache.append(torch.from_numpy(H).cuda())
    if batch == 1:
        pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    else:
        with pytest.raises(pf.ProxyFormerError):
            pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    full = [b for b in range(batch) if n_open[b] == 4]
    ref = OD.kv_append(spec, prm, {k: (v[full] if k != "x" else v) for k, v in st.items()}, H[full])
    for k in ("K_proxy", "V_proxy"):
        for i, b in enumerate(full):
            row = b % 5
            assert_close(k, cache.s[k][b, row].float().cpu().numpy(), ref[k][i, row])
            before[k][b, row] = cache.s[k][b, row]
        assert torch.equal(before[k], cache.s[k])


@pytest.mark.parametrize("r", [1, 8, 9, 16, 17, 255])
def test_prefill_open_rows(r):
    spec = S.DecodeSpec(batch=2, d=192, n_heads=3, P=256, capacity=3)
    prm = S.make_decode_params(spec, 16)
    cache = ProxyKVCache(spec, prm, S.make_decode_state(spec, 17, [1, 2], [3, 4]))
    before = {k: cache.s[k][:, r:].clone() for k in ("X_open", "K_open", "V_open")}
    X = S.round_bf16(np.random.default_rng(18).standard_normal((2, r, 192)).astype(np.float32))
    cache.prefill(torch.from_numpy(X).to("cuda", torch.bfloat16))
    pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
    ref = OD.kv_prefill(spec, prm, X, None)
    for k in ("X_open", "K_open", "V_open"):
        assert_close(k, cache.s[k][:, :r].float().cpu().numpy(), ref[k][:, :r])
        assert torch.equal(before[k], cache.s[k][:, r:])
    assert cache.s["n_open"].tolist() == [r, r] and cache.s["n_proxy"].tolist() == [0, 0]


@pytest.mark.parametrize("batch", [1, 8, 9, 16, 17])
def test_append_kv_is_one_launch(batch):
    """However many rows it has: a short append is bound by its launches."""
    spec = S.DecodeSpec(batch=batch, d=192, n_heads=3, P=4, capacity=5)
    cache = ProxyKVCache(spec, S.make_decode_params(spec, 13),
                         S.make_decode_state(spec, 14, [0] * batch, [4] * batch))
    pf.pf_timing_enable(True)
    try:
        cache.append()
        pf.pf_sync_check(torch.cuda.current_stream().cuda_stream)
        launches = pf.pf_timing_collect()["append_kv"]["launches"]
    finally:
        pf.pf_timing_enable(False)
    assert launches == 1
