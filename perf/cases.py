"""Performance cases of the ProxyFormer library: what a program that uses it has it do.

``listed()`` names the measured calls, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes what a
program holds before the call (weights, inputs, caches, buffers), ``run`` is one pass through the public entry
points, ``work`` the bytes and FLOPs the pass cannot do without, ``exact`` the same pass in plain float64 torch
and ``tolerance`` how far two correct bf16 (or fp32) implementations differ.

Kinds: "layer" (1D layer, training step or inference forward, every option of the descriptor), "image" (2D
layer), "fp32" (fp32 layer, inference), "decode" (one token per sequence on the proxy cache, called directly or
replayed as a graph), "append" (a full open block becomes a cached proxy), "stack" (prefill of a stack of layers
with all their caches).
"""
import math
from types import SimpleNamespace

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_2608_23463_gb300 as pf
from paper_2608_23463_gb300.decode import ProxyKVCache
from paper_2608_23463_gb300.layer import ProxyLayer
from paper_2608_23463_gb300.stack import ProxyStack

BF, F32, F64 = torch.bfloat16, torch.float32, torch.float64
MODES = {"causal": pf.PF_CAUSAL_1D, "bidir": pf.PF_BIDIR_1D, "2d": pf.PF_BIDIR_2D}
INJECTS = {"add": pf.PF_INJ_ADD, "gated": pf.PF_INJ_GATED, "affine": pf.PF_INJ_AFFINE, "cross": pf.PF_INJ_CROSS}
INTERACTS = {"attention": pf.PF_F_ATTENTION, "identity": pf.PF_F_IDENTITY, "mlp": pf.PF_F_MLP}
TEMB = 256  # width of the timestep embedding


def _layer(name, batch, L, d, P, k1=0, d_fine=0, mode="causal", inject="gated", interact="attention", rope=0,
           train=True, carry=False):
    """A 1D layer; k1 > 0: two levels k1 x P/k1; carry: with an incoming proxy state and its gradients."""
    c = dict(kind="layer", batch=batch, L=L, d=d, P=P, k1=k1, d_fine=d_fine, mode=mode, inject=inject,
             interact=interact, rope=rope, train=train, carry=carry)
    return dict(c, name=name) if name else c


def _image(name, batch, gh, gw, d, patch, train=True):
    c = dict(kind="image", batch=batch, gh=gh, gw=gw, d=d, patch=patch, train=train)
    return dict(c, name=name) if name else c


def _fp32(name, batch, L, d, P, k1=0, mode="causal"):
    c = dict(kind="fp32", batch=batch, L=L, d=d, P=P, k1=k1, mode=mode)
    return dict(c, name=name) if name else c


def _decode(name, batch, d, dh, P, capacity, fill, graph):
    """fill: share of the cache that the longest sequence uses (the others hold less)."""
    c = dict(kind="decode", batch=batch, d=d, dh=dh, P=P, capacity=capacity, fill=fill, graph=graph)
    return dict(c, name=name) if name else c


def _append(name, batch, d, dh, P, k1):
    c = dict(kind="append", batch=batch, d=d, dh=dh, P=P, k1=k1)
    return dict(c, name=name) if name else c


def _stack(name, L, d, P0, P1):
    """Three layers with block sizes P0, P0, P1 (the second takes the first one's proxy state)."""
    c = dict(kind="stack", L=L, d=d, P0=P0, P1=P1)
    return dict(c, name=name) if name else c


def listed():
    return [
        # training step of the long-context layer: 256K tokens, two-level 8 x 8 compression
        _layer("layer_train_256k", 1, 262144, 1024, 64, 8),
        # training step with one-level compression: weights of 64K columns, 64K tokens
        _layer("layer_train_64k_1level", 1, 65536, 1024, 64),
        # training step of a small layer (ragged, carried proxy state): latency and launches
        _layer("layer_train_small", 2, 1000, 128, 16, 4, carry=True),
        # inference forward over two prompts of a few thousand tokens, ragged
        _layer("layer_infer_5k", 2, 5000, 1024, 64, 8, train=False),
        # training step with gated cross-attention injection: every token attends to the proxies
        _layer("cross_train_128k", 1, 131072, 1024, 64, 8, inject="cross"),
        # training step of the language model's history layer: narrow tokens, 16384 proxies
        _layer("history_train_1m", 1, 1048576, 512, 64, d_fine=64),
        # training step of the image layer: four 512 x 512 grids, 8 x 8 patches
        _image("image_train_512", 4, 512, 512, 512, 8),
        # fp32 inference forward, 4K tokens
        _fp32("fp32_infer_4k", 1, 4096, 256, 64),
        # one generated token for each of 8 sequences with 1M-token histories, called directly
        _decode("decode_b8_16k", 8, 2048, 128, 64, 16384, 1.0, False),
        # one generated token of a single sequence with a short history, replayed as a CUDA graph
        _decode("decode_graph_b1_1k", 1, 1024, 64, 64, 1024, 0.9, True),
        # a full block of 8 sequences compressed and appended to their caches
        _append("append_b8", 8, 2048, 128, 64, 0),
        # prefill of a short stack: forward over a ragged history and all caches filled
        _stack("stack_prefill_32k", 32760, 1024, 16, 64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer"] * 5 + ["cross", "image", "fp32", "decode", "decode", "append", "stack"])
    if kind == "layer":
        while True:
            d = 64 * rng.choice([1, 2, 3, 4, 6, 8, 12, 16])
            P = rng.choice([8, 16, 32, 64, 64, 128, 256])
            k1 = rng.choice([0, 1 << math.ceil(math.log2(P) / 2)])
            df = rng.choice([0, 0, 0, 64, 128])
            batch, L = rng.choice([1, 1, 2, 3]), _log(rng, 300, 262144)
            if rng.random() < 0.4:
                L -= L % P
            m = -(-L // P)
            if batch * L * (df or d) <= 2 ** 27 and (k1 or P) * (df or d) * d <= 2 ** 26 and m >= 2 and m <= 16384:
                break
        interact = rng.choice(["attention"] * 5 + ["identity", "mlp"])
        return _layer("", batch, L, d, P, k1, 0 if df == d else df, rng.choice(["causal", "causal", "causal", "bidir"]),
                      rng.choice(["gated", "gated", "add"]), interact,
                      int(interact == "attention" and rng.random() < 0.25), rng.random() < 0.7, rng.random() < 0.4)
    if kind == "cross":
        P = rng.choice([16, 32, 64, 128])
        L = _log(rng, 500, 65536 if P >= 32 else 32768)
        return _layer("", rng.choice([1, 2]) if L < 20000 else 1, L, 64 * rng.choice([2, 4, 8, 16]), P,
                      rng.choice([0, 8]) if P != 128 else 16, inject="cross",
                      mode=rng.choice(["causal", "causal", "bidir"]), train=rng.random() < 0.7)
    if kind == "image":
        p, d = rng.choice([2, 4, 8]), 128 * rng.choice([1, 2, 3, 4])
        while True:
            gh, gw = p * _log(rng, 3, 64), p * _log(rng, 3, 64)
            batch = rng.choice([1, 2, 3, 4])
            if batch * gh * gw * d <= 2 ** 27 and gh * gw // (p * p) <= 4096:
                return _image("", batch, gh, gw, d, p, rng.random() < 0.8)
    if kind == "fp32":
        P = rng.choice([8, 16, 32, 64])
        return _fp32("", rng.choice([1, 2]), _log(rng, 200, 16384), 64 * rng.choice([1, 2, 4, 6, 8]), P,
                     rng.choice([0, 8 if P >= 32 else 4]), rng.choice(["causal", "causal", "bidir"]))
    if kind == "decode":
        dh = rng.choice([64, 128])
        return _decode("", rng.choice([1, 2, 3, 5, 8, 12]), dh * rng.choice([2, 4, 6, 8, 16, 16]), dh,
                       rng.choice([16, 32, 64]), _log(rng, 16, 16384), round(rng.uniform(0.2, 1.0), 2),
                       rng.random() < 0.4)
    if kind == "append":
        dh = rng.choice([64, 128])
        P = rng.choice([16, 32, 64])
        return _append("", rng.choice([1, 2, 3, 5, 8, 16]), dh * rng.choice([2, 4, 8, 12, 16]), dh, P,
                       rng.choice([0, 8 if P >= 32 else 4]))
    P0 = rng.choice([16, 32])
    return _stack("", _log(rng, 1000, 32768), 64 * rng.choice([4, 8, 16]), P0, P0 * rng.choice([2, 4]))


# ------------------------------------------------------------------ inputs
def _spec(c, L=None, P=None, k1=None):
    """The layer descriptor's fields (an object with the attributes that the library's classes read)."""
    P = P or c.get("P") or c["patch"] ** 2
    k1 = c.get("k1", 0) if k1 is None else k1
    d, image = c["d"], c["kind"] == "image"
    L = L or (c["gh"] * c["gw"] if image else c["L"])
    return SimpleNamespace(
        batch=c.get("batch", 1), L=L, d=d, n_heads=d // 64, P=P, levels=2 if k1 else 1, k1=k1 or P,
        k2=P // k1 if k1 else 1, mode=MODES["2d" if image else c.get("mode", "causal")],
        inject=INJECTS["affine" if image else c.get("inject", "gated")],
        dtype=pf.PF_F32 if c["kind"] == "fp32" else pf.PF_BF16, grid_h=c.get("gh", 0), grid_w=c.get("gw", 0),
        patch=c.get("patch", 0), d_fine=c.get("d_fine", 0), interact=INTERACTS[c.get("interact", "attention")],
        rope=c.get("rope", 0), m=-(-L // P))


def _draws(seed):
    """Draw functions on a generator of this seed: Xavier-uniform matrices, small vectors, N(0, 1) activations."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def mat(o, i, dt, rows=None):
        b = math.sqrt(6.0 / (i + (rows or o)))
        return torch.empty(o, i, device="cuda").uniform_(-b, b, generator=g).to(dt)

    def vec(n, at=0.0):
        return torch.empty(n, device="cuda").uniform_(-0.1, 0.1, generator=g) + at

    def act(*shape, dt=BF):
        return torch.empty(shape, device="cuda", dtype=dt).normal_(generator=g)

    return mat, vec, act, g


def _params(s, mat, vec, dt):
    """One layer's parameters, drawn in a fixed order (as tensors of the layer's types)."""
    d, df = s.d, s.d_fine or s.d
    p = {"W_c1": mat(d, s.k1 * df, dt), "b_c1": vec(d)}
    if s.levels == 2:
        p.update(W_c2=mat(d, s.k2 * d, dt), b_c2=vec(d))
    if s.interact == pf.PF_F_ATTENTION:
        p.update(W_qkv=mat(3 * d, d, dt, d), W_o=mat(d, d, dt))
    elif s.interact == pf.PF_F_MLP:
        p.update(W_m1=mat(4 * d, d, dt), b_m1=vec(4 * d), W_m2=mat(d, 4 * d, dt), b_m2=vec(d))
    if s.inject == pf.PF_INJ_CROSS:
        p.update(W_qa=mat(d + s.n_heads, d, dt, d), b_a=vec(s.n_heads), W_kvx=mat(2 * d, d, dt, d),
                 W_ox=mat(d, d, dt))
        return p
    w = 2 * d if s.inject == pf.PF_INJ_AFFINE else df
    if s.levels == 2:
        p.update(W_d2=mat(s.k2 * d, d, dt), b_d2=vec(s.k2 * d))
    p.update(W_d1=mat(s.k1 * w, d, dt), b_d1=vec(s.k1 * w))
    if s.inject == pf.PF_INJ_GATED:
        p.update(w_x=vec(df), w_dlt=vec(df), b_g=vec(df))
    if s.mode == pf.PF_BIDIR_2D:
        p.update(W_t1=mat(d, TEMB, dt), b_t1=vec(d), W_t2=mat(2 * d, d, dt), b_t2=vec(2 * d))
    return p


def _layer_inputs(c, seed):
    s = _spec(c)
    mat, vec, act, g = _draws(seed)
    dt = F32 if c["kind"] == "fp32" else BF
    p = _params(s, mat, vec, dt)
    df = s.d_fine or s.d
    x = {"X": act(s.batch, s.L, df, dt=dt)}
    if c.get("carry"):
        x["H_in"] = act(s.batch, s.m, s.d, dt=F32)
    if c["kind"] == "image":
        x["t"] = torch.rand(s.batch, device="cuda", generator=g)
    if c.get("train"):
        x["G"] = act(s.batch, s.L, df, dt=dt)
        if c.get("carry"):
            x["dH_out"] = act(s.batch, s.m, s.d, dt=F32)
    return s, p, x


def _np(p):
    return {k: v.float().cpu().numpy() for k, v in p.items()}


def _decode_spec(batch, d, dh, P, k1, capacity):
    return SimpleNamespace(batch=batch, d=d, n_heads=d // dh, P=P, levels=2 if k1 else 1, k1=k1 or P,
                           k2=P // k1 if k1 else 1, capacity=capacity)


def _decode_params(s, mat, vec):
    d, h = s.d, s.d // 8
    p = {"W_qkv": mat(3 * d, d, BF, d), "W_o": mat(d, d, BF), "rms_w": vec(d, 1.0), "W_a1": mat(h, d, BF),
         "b_a1": vec(h), "W_a2": mat(s.n_heads, h, BF), "b_a2": vec(s.n_heads), "W_c1": mat(d, s.k1 * d, BF),
         "b_c1": vec(d)}
    if s.levels == 2:
        p.update(W_c2=mat(d, s.k2 * d, BF), b_c2=vec(d))
    p["W_kvh"] = mat(2 * d, d, BF, d)
    return p


def _cache(s, p):
    """An empty cache (int8 zeros: its constructor converts what it is given on the device)."""
    z = lambda rows: np.zeros((s.batch, rows, s.d), np.int8)  # noqa: E731
    st = {"K_proxy": z(s.capacity), "V_proxy": z(s.capacity), "X_open": z(s.P), "K_open": z(s.P), "V_open": z(s.P),
          "n_proxy": np.zeros(s.batch, np.int32), "n_open": np.zeros(s.batch, np.int32)}
    return ProxyKVCache(s, _np(p), st)


def _decode_inputs(c, seed):
    # the weights of the append are not used by a step: one-token blocks keep them small
    s = _decode_spec(c["batch"], c["d"], c["dh"], c["P"], 0, c["capacity"])
    mat, vec, act, _ = _draws(seed)
    p = _decode_params(SimpleNamespace(**{**vars(s), "k1": 1}), mat, vec)
    B, d, P, cap = s.batch, s.d, s.P, s.capacity
    top = max(1, int(c["fill"] * cap))
    n_proxy = torch.tensor([max(0, top - (top * 3 * b) // (4 * B)) if c["fill"] < 1 else cap for b in range(B)],
                           dtype=torch.int32, device="cuda")
    n_open = torch.tensor([(seed + 5 * b) % (P - 1) for b in range(B)], dtype=torch.int32, device="cuda")
    x = {"x": act(B, d), "K_proxy": act(B, cap, d), "V_proxy": act(B, cap, d), "X_open": act(B, P, d),
         "K_open": act(B, P, d), "V_open": act(B, P, d), "n_proxy": n_proxy, "n_open": n_open}
    return s, p, x


def _append_inputs(c, seed):
    s = _decode_spec(c["batch"], c["d"], c["dh"], c["P"], c["k1"], 8)
    mat, vec, act, _ = _draws(seed)
    p = _decode_params(s, mat, vec)
    B = s.batch
    x = {"X_open": act(B, s.P, s.d), "H_in": act(B, s.d, dt=F32),
         "n_proxy": torch.tensor([b % 3 for b in range(B)], dtype=torch.int32, device="cuda")}
    return s, p, x


def _stack_inputs(c, seed):
    mat, vec, act, _ = _draws(seed)
    lay, specs = [], []
    for P in (c["P0"], c["P0"], c["P1"]):
        s = _spec(dict(c, kind="layer"), P=P, k1=1 << math.ceil(math.log2(P) / 2))
        specs.append(s)
        p = _params(s, mat, vec, BF)
        cs = _decode_spec(1, s.d, 64, P, s.k1, s.L // P + 8)
        q = _decode_params(SimpleNamespace(**{**vars(cs), "k1": 1, "k2": 1}), mat, vec)
        q.update({k: p[k] for k in ("W_c1", "b_c1", "W_c2", "b_c2")}, W_kvh=p["W_qkv"][s.d:])
        lay.append((cs, p, q))
    return specs, lay, act(1, c["L"], c["d"])


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("layer", "image", "fp32"):
        s, p, x = _layer_inputs(c, seed)
        layer = ProxyLayer(s, _np(p))
        st = dict(x, layer=layer, train=c.get("train", False), X_out=layer.empty_act(), H_out=layer.empty_proxy())
        if st["train"]:
            st.update(dX=layer.empty_act(), dH_in=layer.empty_proxy())
        return st
    if kind == "decode":
        s, p, x = _decode_inputs(c, seed)
        cache = _cache(s, p)
        for k in ("K_proxy", "V_proxy", "X_open", "K_open", "V_open", "n_proxy", "n_open"):
            cache.s[k].copy_(x[k])
        st = dict(cache=cache, x=x["x"], y=torch.zeros_like(x["x"]), n_open=x["n_open"], graph=None)
        if c["graph"]:
            cache.step(st["x"], st["y"])
            cache.s["n_open"].copy_(x["n_open"])
            torch.cuda.synchronize()
            st["graph"] = cache.capture_step(st["x"], st["y"])
        return st
    if kind == "append":
        s, p, x = _append_inputs(c, seed)
        cache = _cache(s, p)
        cache.s["X_open"].copy_(x["X_open"])
        return dict(cache=cache, H_in=x["H_in"], n_proxy=x["n_proxy"],
                    n_open=torch.full((s.batch,), s.P, dtype=torch.int32, device="cuda"))
    specs, lay, X = _stack_inputs(c, seed)
    return dict(stack=ProxyStack(specs, [_np(p) for _, p, _ in lay]), X=X,
                caches=[_cache(cs, q) for cs, _, q in lay])


# --------------------------------------------------------------------- run
def run(state):
    st = state
    if "layer" in st:
        lay, H_in, t = st["layer"], st.get("H_in"), st.get("t")
        lay.forward(st["X"], H_in, t, X_out=st["X_out"], H_out=st["H_out"], train=st["train"])
        out = {"X_out": st["X_out"], "H_out": st["H_out"]}
        if st["train"]:
            lay.backward(st["X"], st["G"], H_in, t, dH_out=st.get("dH_out"), dX=st["dX"], dH_in=st["dH_in"])
            out.update(dX=st["dX"], dH_in=st["dH_in"], **{"grad_" + k: v for k, v in lay.grads.items()})
        return out
    if "stack" in st:
        out = {"X_out": st["stack"].prefill(st["X"], st["caches"])}
        for l, cache in enumerate(st["caches"]):
            out.update({"%s%d" % (k, l): cache.s[k] for k in
                        ("K_proxy", "V_proxy", "X_open", "K_open", "V_open", "n_proxy", "n_open")})
        return out
    cache = st["cache"]
    if "x" in st:
        # a token at the same place again, as a decoder that discards a draft token has it
        cache.s["n_open"].copy_(st["n_open"])
        if st["graph"] is not None:
            st["graph"].replay()
        else:
            cache.step(st["x"], st["y"])
        return {"y": st["y"], "X_open": cache.s["X_open"], "K_open": cache.s["K_open"], "V_open": cache.s["V_open"],
                "n_open": cache.s["n_open"]}
    cache.s["n_open"].copy_(st["n_open"])  # the block is full again, its proxy is written at the same row
    cache.s["n_proxy"].copy_(st["n_proxy"])
    cache.append(st["H_in"])
    return {"K_proxy": cache.s["K_proxy"], "V_proxy": cache.s["V_proxy"], "n_proxy": cache.s["n_proxy"],
            "n_open": cache.s["n_open"]}


# -------------------------------------------------------------------- work
def _layer_work(s, train, carry):
    """FLOPs: the contractions (backward: twice the linear ones, 2.5 times the attention).  Bytes: inputs,
    weights and outputs once; proxy states and gradients fp32."""
    B, L, d, df, m, P = s.batch, s.L, s.d, s.d_fine or s.d, s.m, s.P
    e = 4 if s.dtype == pf.PF_F32 else 2
    causal = s.mode == pf.PF_CAUSAL_1D
    R = B * m
    lin = 2.0 * R * P * df * d + (2.0 * R * s.k2 * d * d if s.levels == 2 else 0.0)
    w = d * s.k1 * df + (d * s.k2 * d if s.levels == 2 else 0)
    att = 0.0
    if s.interact == pf.PF_F_ATTENTION:
        lin += 8.0 * R * d * d
        w += 4 * d * d
        att += 4.0 * d * B * (m * (m + 1) / 2.0 if causal else float(m) * m)
    elif s.interact == pf.PF_F_MLP:
        lin += 16.0 * R * d * d
        w += 8 * d * d
    if s.inject == pf.PF_INJ_CROSS:
        lin += 2.0 * B * L * d * (d + s.n_heads) + 4.0 * R * d * d + 2.0 * B * L * d * d
        w += d * (d + s.n_heads) + 3 * d * d
        n = sum(min(P, L - i * P) * i for i in range(m)) if causal else L * m
        att += 4.0 * d * B * n
    else:
        wide = 2 * df if s.inject == pf.PF_INJ_AFFINE else df
        lin += 2.0 * R * P * wide * d + (2.0 * R * s.k2 * d * d if s.levels == 2 else 0.0)
        w += d * s.k1 * wide + (d * s.k2 * d if s.levels == 2 else 0)
    if s.mode == pf.PF_BIDIR_2D:
        w += d * TEMB + 2 * d * d
    tok, prox = B * L * df * e, R * d * 4
    by = 2 * tok + w * e + prox * (2 if carry else 1)
    fl = lin + att
    if train:
        by += 2 * tok + 4 * w + prox * (2 if carry else 1)
        fl += 2 * lin + 2.5 * att
    return by, fl


def work(case):
    c, kind = case, case["kind"]
    if kind in ("layer", "image", "fp32"):
        by, fl = _layer_work(_spec(c), c.get("train", False), c.get("carry", False))
        return {"bytes": by, "flops": fl}
    if kind == "decode":
        B, d, P, cap, h = c["batch"], c["d"], c["P"], c["capacity"], c["d"] // 8
        top = max(1, int(c["fill"] * cap))
        n = sum(max(0, top - (top * 3 * b) // (4 * B)) if c["fill"] < 1 else cap for b in range(B))
        w = 4 * d * d + h * d + h * d // c["dh"]
        return {"bytes": 4.0 * d * (n + B * P / 2.0) + 2.0 * w + 12.0 * B * d,
                "flops": 2.0 * B * w + 4.0 * d * (n + B * P / 2.0)}
    if kind == "append":
        B, d, P, k1 = c["batch"], c["d"], c["P"], c["k1"]
        w = (k1 or P) * d * d + (P // k1 * d * d if k1 else 0) + 2 * d * d
        return {"bytes": 2.0 * w + 2.0 * B * P * d + 8.0 * B * d,
                "flops": 2.0 * B * (P * d * d + (P // k1 * d * d if k1 else 0) + 2 * d * d)}
    by = fl = 0.0
    for P in (c["P0"], c["P0"], c["P1"]):
        s = _spec(dict(c, kind="layer"), P=P, k1=1 << math.ceil(math.log2(P) / 2))
        b, f = _layer_work(s, False, False)
        r = s.L % P
        by += b + 4.0 * (s.L // P) * s.d + 6.0 * r * s.d
        fl += f + 4.0 * r * s.d * s.d
    return {"bytes": by, "flops": fl}


def tolerance(case):
    # about four times what the library was off float64 (largest relative error of any output): fp32 4e-7; a step,
    # a forward 2e-3; an append 2.3e-3; the third layer's cache rows of a stack 5e-3; gradients 1.2e-2 (bf16 storage
    # of every activation gradient; four times that is over what one can tell apart, 3e-2 is taken)
    if case["kind"] == "fp32":
        return {"rel": 5e-6, "max": 5e-4}
    if case["kind"] == "append":
        return {"rel": 0.01, "max": 0.1}
    if case["kind"] == "stack":
        return {"rel": 0.02, "max": 0.3}
    if case.get("train"):
        return {"rel": 0.03, "max": 0.6}
    return {"rel": 0.008, "max": 0.1}


# ------------------------------------------------------------------- exact
def _attend(q, k, v, vis):
    """softmax(q k^T / sqrt(dh)) v over the visible pairs (vis None: all); every row sees something."""
    s = (q @ k.T) * (1.0 / math.sqrt(q.shape[1]))
    if vis is not None:
        s = s.masked_fill(~vis, -math.inf)
    return torch.softmax(s, 1) @ v


def _rope(z, nh):
    m, d = z.shape
    ang = torch.arange(m, device=z.device, dtype=F64)[:, None] * \
        10000.0 ** (-torch.arange(0, 64, 2, device=z.device, dtype=F64) / 64)[None, :]
    cs, sn = ang.cos()[:, None, :], ang.sin()[:, None, :]
    a, b = z.view(m, nh, 32, 2).unbind(-1)
    return torch.stack((a * cs - b * sn, a * sn + b * cs), -1).reshape(m, d)


def _ln(x):
    return (x - x.mean(-1, keepdim=True)) / (x.var(-1, unbiased=False, keepdim=True) + 1e-6).sqrt()


def _layer64(s, p, X, H_in=None, t=None):
    """The layer in float64: (X_out, H, H's keys, H's values) from float64 parameters and inputs."""
    B, L, df = X.shape
    d, m, P, k1, k2, nh = s.d, s.m, s.P, s.k1, s.k2, s.n_heads
    if s.mode == pf.PF_BIDIR_2D:
        q = s.patch
        cut = lambda z: z.view(B, s.grid_h // q, q, s.grid_w // q, q, -1).permute(  # noqa: E731
            0, 1, 3, 2, 4, 5).reshape(B, m, P, -1)
        back = lambda z: z.reshape(B, s.grid_h // q, s.grid_w // q, q, q, -1).permute(  # noqa: E731
            0, 1, 3, 2, 4, 5).reshape(B, L, -1)
    else:
        cut = lambda z: torch.nn.functional.pad(z, (0, 0, 0, m * P - L)).view(B, m, P, -1)  # noqa: E731
        back = lambda z: z.reshape(B, m * P, -1)[:, :L]  # noqa: E731
    C = cut(X).reshape(B, m, k2, k1 * df) @ p["W_c1"].T + p["b_c1"]
    C = C.reshape(B, m, k2 * d) @ p["W_c2"].T + p["b_c2"] if s.levels == 2 else C.reshape(B, m, d)
    H = C if H_in is None else H_in + C
    Hq = H
    if s.mode == pf.PF_BIDIR_2D:
        w = 10000.0 ** (-torch.arange(128, device=X.device, dtype=F64) / 128)
        a = 1000.0 * t[:, None] * w
        e = torch.cat((a.cos(), a.sin()), 1)
        gb = torch.nn.functional.silu(e @ p["W_t1"].T + p["b_t1"]) @ p["W_t2"].T + p["b_t2"]
        Hq = (1.0 + gb[:, None, :d]) * _ln(H) + gb[:, None, d:]
    causal = s.mode == pf.PF_CAUSAL_1D
    K = V = None
    if s.interact == pf.PF_F_IDENTITY:
        Hbar = Hq
    elif s.interact == pf.PF_F_MLP:
        Hbar = torch.nn.functional.silu(Hq @ p["W_m1"].T + p["b_m1"]) @ p["W_m2"].T + p["b_m2"]
    else:
        Q, K, V = (Hq @ p["W_qkv"].T).split(d, -1)
        vis = torch.ones(m, m, dtype=torch.bool, device=X.device).tril() if causal else None
        rows = []
        for b in range(B):
            qb, kb = (_rope(Q[b], nh), _rope(K[b], nh)) if s.rope else (Q[b], K[b])
            rows.append(torch.cat([checkpoint(_attend, qb[:, h:h + 64], kb[:, h:h + 64], V[b][:, h:h + 64], vis,
                                              use_reentrant=False) for h in range(0, d, 64)], 1))
        Hbar = torch.stack(rows) @ p["W_o"].T
    if s.inject == pf.PF_INJ_CROSS:
        Qx, al = X @ p["W_qa"][:d].T, torch.sigmoid(X @ p["W_qa"][d:].T + p["b_a"])
        Kx, Vx = (Hbar @ p["W_kvx"].T).split(d, -1)
        n0 = min(P, L) if causal else 0  # the first block's tokens see no proxy
        vis = (torch.arange(m, device=X.device)[None, :] <
               (torch.arange(n0, L, device=X.device) // P)[:, None]) if causal else None
        rows = []
        for b in range(B):
            heads = [checkpoint(_attend, Qx[b, n0:, h:h + 64], Kx[b][:, h:h + 64], Vx[b][:, h:h + 64], vis,
                                use_reentrant=False) for h in range(0, d, 64)] if n0 < L else []
            a = torch.cat(heads, 1) if heads else X.new_zeros(0, d)
            rows.append(torch.cat((X.new_zeros(n0, d), a)))
        A = torch.stack(rows) * al.repeat_interleave(64, dim=2)
        return X + A @ p["W_ox"].T, H, K, V
    Z = Hbar
    if s.levels == 2:
        Z = Z @ p["W_d2"].T + p["b_d2"]
    D = (Z.reshape(B, m, k2, d) @ p["W_d1"].T + p["b_d1"]).reshape(B, m, P, -1)
    if causal:  # a block receives the proxy before it
        D = torch.cat((torch.zeros_like(D[:, :1]), D[:, :-1]), 1)
    D = back(D)
    if s.inject == pf.PF_INJ_ADD:
        return X + D, H, K, V
    if s.inject == pf.PF_INJ_AFFINE:
        return (1.0 + D[..., :d]) * _ln(X) + D[..., d:], H, K, V
    return X + torch.sigmoid(p["w_x"] * X + p["w_dlt"] * D + p["b_g"]) * D, H, K, V


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("layer", "image", "fp32"):
        s, p, x = _layer_inputs(c, seed)
        train = c.get("train", False)
        p = {k: v.to(F64).requires_grad_(train) for k, v in p.items()}
        G, dH = x.pop("G", None), x.pop("dH_out", None)
        x = {k: v.to(F64) for k, v in x.items()}
        X = x["X"].requires_grad_(train)
        H_in = x.get("H_in")
        if H_in is not None:
            H_in.requires_grad_(train)
        with torch.set_grad_enabled(train):
            Xo, H, _, _ = _layer64(s, p, X, H_in, x.get("t"))
        out = {"X_out": Xo.detach(), "H_out": H.detach()}
        if train:
            # dH_in is the gradient of H itself (H = H_in + C), whether or not H_in is given
            H.retain_grad()
            torch.autograd.backward([Xo] + ([H] if dH is not None else []),
                                    [G.to(F64)] + ([dH.to(F64)] if dH is not None else []))
            out.update(dX=X.grad, dH_in=H.grad, **{"grad_" + k: v.grad for k, v in p.items()})
        return out
    if kind == "decode":
        s, p, x = _decode_inputs(c, seed)
        p, y = {k: v.to(F64) for k, v in p.items()}, {k: v for k, v in x.items()}
        d, nh, dh = s.d, s.n_heads, s.d // s.n_heads
        xs = x["x"].to(F64)
        q, k, v = (xs @ p["W_qkv"].T).split(d, 1)
        o = {n: y[n].to(F64) for n in ("X_open", "K_open", "V_open")}
        rn = xs / (xs.square().mean(1, keepdim=True) + 1e-6).sqrt() * p["rms_w"]
        u = torch.nn.functional.silu(rn @ p["W_a1"].T + p["b_a1"])
        al = torch.sigmoid(u @ p["W_a2"].T + p["b_a2"])
        A = torch.zeros_like(xs)
        for b in range(s.batch):
            n, no = int(x["n_proxy"][b]), int(x["n_open"][b])
            o["X_open"][b, no], o["K_open"][b, no], o["V_open"][b, no] = xs[b], k[b], v[b]
            Kp, Vp = x["K_proxy"][b, :n].to(F64), x["V_proxy"][b, :n].to(F64)
            for h in range(nh):
                cs = slice(h * dh, (h + 1) * dh)
                A[b, cs] = _attend(q[b:b + 1, cs], o["K_open"][b, :no + 1, cs], o["V_open"][b, :no + 1, cs], None)[0]
                if n:
                    A[b, cs] += al[b, h] * _attend(q[b:b + 1, cs], Kp[:, cs], Vp[:, cs], None)[0]
        return dict(y=xs + A @ p["W_o"].T, **o, n_open=None)
    if kind == "append":
        s, p, x = _append_inputs(c, seed)
        p = {k: v.to(F64) for k, v in p.items()}
        C = x["X_open"].to(F64).reshape(s.batch, s.k2, s.k1 * s.d) @ p["W_c1"].T + p["b_c1"]
        C = C.reshape(s.batch, s.k2 * s.d) @ p["W_c2"].T + p["b_c2"] if s.levels == 2 else C.reshape(s.batch, s.d)
        kv = (x["H_in"].to(F64) + C) @ p["W_kvh"].T
        out = {n: torch.zeros(s.batch, s.capacity, s.d, device="cuda", dtype=F64) for n in ("K_proxy", "V_proxy")}
        for b in range(s.batch):
            out["K_proxy"][b, int(x["n_proxy"][b])] = kv[b, :s.d]
            out["V_proxy"][b, int(x["n_proxy"][b])] = kv[b, s.d:]
        return dict(out, n_proxy=None, n_open=None)
    specs, lay, X = _stack_inputs(c, seed)
    X, H, out = X.to(F64), None, {}
    with torch.no_grad():
        for l, (s, (cs, p, q)) in enumerate(zip(specs, lay)):
            p = {k: v.to(F64) for k, v in p.items()}
            m, r, d = s.L // s.P, s.L % s.P, s.d
            zero = lambda n: torch.zeros(1, n, d, device="cuda", dtype=F64)  # noqa: E731
            o = {"K_proxy": zero(cs.capacity), "V_proxy": zero(cs.capacity), "X_open": zero(s.P),
                 "K_open": zero(s.P), "V_open": zero(s.P)}
            tail, w = X[:, m * s.P:], q["W_qkv"].to(F64)
            o["X_open"][:, :r], o["K_open"][:, :r], o["V_open"][:, :r] = tail, tail @ w[d:2 * d].T, tail @ w[2 * d:].T
            X, H, K, V = _layer64(s, p, X, H if l and specs[l - 1].P == s.P else None)
            o["K_proxy"][:, :m], o["V_proxy"][:, :m] = K[:, :m], V[:, :m]
            out.update({"%s%d" % (k, l): v for k, v in o.items()}, **{"n_proxy%d" % l: None, "n_open%d" % l: None})
    return dict(out, X_out=X)
