"""What this library is timed on: the calls a decoding program makes, from one small projection
to whole decode steps, through the public entry points.

A case is a dict of plain values; its "kind" says which part of the library it exercises:

  operator  afx_select_gemv: selection + sparse GEMV of one projection in one call
  list      afx_select_active (+ afx_diff_active against a predicted set) + afx_sparse_gemv: the
            same operator as separate calls, for programs that keep or ship the active list
  mlp       DecoderModel.mlp_block: the MLP of a layer on a given input, threshold or top-k
  decode    DecoderModel.decode_step / decode_step_q4: whole decode steps of a Llama-shaped stack
            at consecutive positions of a filled KV cache, every step with another hidden state
  moe       afx_moe_block: router + chosen experts of mixture-of-experts layers
  cached    afx_select_active + afx_cache_fetch + afx_sparse_gemv: an operator whose weights live in
            pinned host memory behind the hot-channel cache; a pass is a few steps of one sequence

Inputs are random: weights N(0, 0.02^2) for single operators; in decode stacks N(0, 1 / inputs), the
projections that add to the residual stream a twentieth of that (a block then changes the residual
by a percent or two, as in deep trained models; where every block outweighs the residual, one rounding that tips
grows from layer to layer until no two summation orders agree); activations Laplace, hidden states
Laplace with a persistent lognormal scale per channel; N(0, 1) KV caches.  "sparsity" is the
percentage of input channels left out.
"""
import math

import numpy as np
import torch

from paper_2504_08378_b200 import afx, synth
from paper_2504_08378_b200.model import DecoderModel

TORCH = {"f16": torch.float16, "bf16": torch.bfloat16}


# ---- cases --------------------------------------------------------------------------------------

def _operator(K, N, T=1, dtype="bf16", mode="topk", sparsity=50, steps=1, hint=False):
    return dict(kind="operator", K=K, N=N, T=T, dtype=dtype, mode=mode, sparsity=sparsity, steps=steps, hint=hint)


def _list(K, N, T=1, dtype="bf16", sparsity=50, predict=False):
    return dict(kind="list", K=K, N=N, T=T, dtype=dtype, sparsity=sparsity, predict=predict)


def _mlp(hidden, mlp, T=1, dtype="f16", mode="threshold", sparsity=50, layers=4):
    return dict(kind="mlp", hidden=hidden, mlp=mlp, T=T, dtype=dtype, mode=mode, sparsity=sparsity, layers=layers)


def _decode(hidden, heads, kv_heads, mlp, layers, past, T=1, dtype="bf16", sparsity=50, xl="bookkeep", q4=False, steps=4):
    return dict(kind="decode", hidden=hidden, heads=heads, kv_heads=kv_heads, mlp=mlp, layers=layers, past=past, T=T,
                dtype=dtype, sparsity=sparsity, xl=xl, q4=q4, steps=steps)


def _moe(hidden, mlp, experts, top, layers, dtype="bf16", sparsity=50):
    return dict(kind="moe", hidden=hidden, mlp=mlp, experts=experts, top=top, layers=layers, dtype=dtype, sparsity=sparsity)


def _cached(K, N, dtype="bf16", sparsity=50, cache_percent=30, steps=4):
    return dict(kind="cached", K=K, N=N, dtype=dtype, sparsity=sparsity, cache_percent=cache_percent, steps=steps)


def listed():
    return [
        # the smallest call: one projection of a small model, all of it in L2; latency and host cost
        dict(_operator(512, 1376, dtype="f16"), name="projection_small"),
        # a projection whose sizes fit no tile, a few tokens at once (speculative or parallel decoding)
        dict(_operator(5003, 7208, T=3, sparsity=60), name="projection_ragged_3_tokens"),
        # the largest operator of a 70B-shaped layer as separate selection, set difference and GEMV
        dict(_list(8192, 57344, predict=True), name="list_70b_gate_up"),
        # a 13B-shaped gate|up for the most tokens a call takes, the list kept by the caller
        dict(_list(5120, 27648, T=8, sparsity=60), name="list_13b_gate_up_8_tokens"),
        # the 7B-shaped MLP block with calibrated thresholds, the run-time form of the method
        dict(_mlp(4096, 11008), name="mlp_7b_threshold"),
        # one sequence decoding on a small grouped-query model that reuses predicted sets: launch-bound
        dict(_decode(1024, 16, 4, 2816, 8, 300, dtype="f16", xl="reuse"), name="decode_small_reuse"),
        # the headline workload: 7B-shaped stack, one sequence, top 50 %, cross-layer bookkeeping
        dict(_decode(4096, 32, 32, 11008, 32, 2048), name="decode_7b"),
        # the same stack over 4-bit weights, the storage type the method is deployed with
        dict(_decode(4096, 32, 32, 11008, 32, 2048, q4=True), name="decode_7b_q4"),
        # four sequences decoded together on a 13B-shaped stack
        dict(_decode(5120, 40, 40, 13824, 40, 2048, T=4, sparsity=60, xl="off", steps=2), name="decode_13b_4_tokens"),
        # a long context on 70B-shaped layers: eight query heads per KV head, attention counts
        dict(_decode(8192, 64, 8, 28672, 8, 8000, steps=2), name="decode_70b_long"),
        # mixture-of-experts layers of the 8 x 7B shape, two experts per token
        dict(_moe(4096, 14336, 8, 2, 2), name="moe_8x7b"),
        # an operator that does not fit the device: pinned host memory behind a 30 % cache
        dict(_cached(8192, 8192), name="cached_70b_o"),
    ]


def _log_int(rng, lo, hi, step=1):
    return max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step)


def draw(rng):
    kind = rng.choice(["operator", "operator", "list", "mlp", "decode", "decode", "decode", "moe", "cached"])
    dtype = rng.choice(["f16", "bf16"])
    sparsity = rng.choice([0, rng.randint(10, 40), rng.randint(40, 60), 50, rng.randint(60, 90)])
    T = rng.choice([1, 1, 1, rng.randint(2, 4), rng.randint(5, 8)])
    if kind == "operator":
        return _operator(_log_int(rng, 256, 16384), _log_int(rng, 256, 32768, 8), T, dtype, rng.choice(["topk", "threshold"]),
                         sparsity, rng.randint(1, 4), rng.random() < 0.5)
    if kind == "list":
        return _list(_log_int(rng, 512, 16384), _log_int(rng, 1024, 57344, 8), T, dtype, sparsity, rng.random() < 0.5)
    if kind == "mlp":
        return _mlp(_log_int(rng, 512, 8192, 8), _log_int(rng, 1024, 16384, 8), T, dtype, rng.choice(["topk", "threshold"]),
                    sparsity, rng.randint(1, 4))
    if kind == "decode":
        q4 = rng.random() < 0.25
        kv, rep = rng.choice([(8, 1), (16, 1), (32, 1), (40, 1), (4, 2), (16, 2), (8, 4), (8, 8), (2, 4)])
        hidden = _log_int(rng, 512, 8192, 32 if q4 else 8)
        mlp = _log_int(rng, 1024, 28672, 32 if q4 else 8)
        per_layer = hidden * (rep * kv + 2 * kv) * 128 + rep * kv * 128 * hidden + 3 * hidden * mlp
        layers = max(1, min(rng.randint(2, 12), 2_000_000_000 // per_layer))
        return _decode(hidden, kv * rep, kv, mlp, layers, _log_int(rng, 16, 8000), 1 if q4 else T, dtype, sparsity,
                       rng.choice(["off", "bookkeep", "reuse"]), q4, rng.randint(1, 4))
    if kind == "moe":
        return _moe(_log_int(rng, 512, 4096, 8), _log_int(rng, 1024, 14336, 8), rng.randint(4, 12), rng.randint(1, 3),
                    rng.randint(1, 2), dtype, sparsity)
    return _cached(_log_int(rng, 1024, 8192), _log_int(rng, 1024, 8192, 8), dtype, max(sparsity, 30),
                   rng.randint(20, 50), rng.randint(2, 6))


# ---- inputs -------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + 17)
    return g


def _normal(g, shape, dtype, sigma):
    """N(0, sigma^2) rounded to a 16-bit type, as int16 bit patterns."""
    n = math.prod(shape)
    out = torch.empty(n, dtype=TORCH[dtype], device="cuda")
    for o in range(0, n, 1 << 26):
        m = min(1 << 26, n - o)
        out[o:o + m] = torch.randn(m, generator=g, device="cuda").mul_(sigma)
    return out.view(torch.int16).view(*shape)


def _laplace(g, shape):
    u = torch.rand(shape, generator=g, device="cuda", dtype=torch.float64).sub_(0.5)
    return (-torch.sign(u) * torch.log1p(-2.0 * u.abs())).float()


def _bits(a, dtype):
    return a.to(TORCH[dtype]).view(torch.int16)


def _tau(sparsity):
    return synth.laplace_tau(sparsity / 100.0)  # inputs are Laplace(0, 1)


def _prepare_operator(c, seed):
    g = _gen(seed)
    K, N, T = c["K"], c["N"], c["T"]
    return dict(c=c, W=_normal(g, (K, N), c["dtype"], 0.02), x=_bits(_laplace(g, (c["steps"], T, K)), c["dtype"]),
                k=synth.keep_count(K, c["sparsity"]), tau=_tau(c["sparsity"]),
                y=torch.zeros((c["steps"], T, N), device="cuda"),
                idx=torch.zeros((c["steps"], K), dtype=torch.int32, device="cuda"),
                count=torch.zeros((c["steps"], 1), dtype=torch.int32, device="cuda"),
                hint=torch.zeros(1, dtype=torch.int32, device="cuda") if c["hint"] else None)


def _run_operator(s):
    c = s["c"]
    mode = afx.MODE_TOPK if c["mode"] == "topk" else afx.MODE_THRESHOLD
    for i in range(c["steps"]):
        afx.afx_select_gemv(s["W"], c["dtype"], c["K"], c["N"], c["N"], s["x"][i], c["T"], mode, s["k"], s["tau"], s["y"][i], 0,
                            s["idx"][i], s["count"][i], kth_hint=s["hint"])
    return s["y"], s["idx"], s["count"]


def _prepare_list(c, seed):
    g = _gen(seed)
    K, N, T = c["K"], c["N"], c["T"]
    shared = _laplace(g, (T, K))  # what this layer's input has in common with the predicting layer's
    mix = lambda: _bits(shared + 0.4 * _laplace(g, (T, K)), c["dtype"])
    s = dict(c=c, W=_normal(g, (K, N), c["dtype"], 0.02), x=mix(), k=synth.keep_count(K, c["sparsity"]),
             y=torch.zeros((T, N), device="cuda"))
    for name, n in (("idx", K), ("count", 1), ("miss", K), ("miss_count", 1), ("hit_count", 1), ("bitmap", (K + 31) // 32)):
        s[name] = torch.zeros(n, dtype=torch.int32, device="cuda")
    if c["predict"]:
        afx.afx_select_active(mix(), c["dtype"], K, T, afx.MODE_TOPK, s["k"], 0.0, s["idx"], s["count"], s["bitmap"])
        s["idx"].zero_()
    return s


def _run_list(s):
    c = s["c"]
    afx.afx_select_active(s["x"], c["dtype"], c["K"], c["T"], afx.MODE_TOPK, s["k"], 0.0, s["idx"], s["count"])
    if c["predict"]:
        afx.afx_diff_active(s["idx"], s["count"], s["bitmap"], c["K"], s["miss"], s["miss_count"], s["hit_count"])
    afx.afx_sparse_gemv(s["W"], c["dtype"], c["K"], c["N"], c["N"], s["x"], c["T"], s["idx"], s["count"], None, s["y"], 0)
    return s["y"], s["idx"], s["count"], s["miss"], s["miss_count"], s["hit_count"]


def _prepare_mlp(c, seed):
    g = _gen(seed)
    H, M, T, dt = c["hidden"], c["mlp"], c["T"], c["dtype"]
    k = [0, 0, synth.keep_count(H, c["sparsity"]), synth.keep_count(M, c["sparsity"])]
    calibration = _laplace(g, (16, H)).to(TORCH[dt])
    layers = []
    for _ in range(c["layers"]):
        w_gu, w_down = _normal(g, (H, 2 * M), dt, 0.02), _normal(g, (M, H), dt, 0.02)
        tau_down = -1.0
        if c["sparsity"]:  # the magnitude below which that share of the down inputs of other tokens falls
            gu = (calibration @ w_gu.view(TORCH[dt])).float().view(16, M // 8, 2, 8)
            hm = (torch.nn.functional.silu(gu[:, :, 0]) * gu[:, :, 1]).abs().flatten()
            tau_down = float(hm.sort().values[hm.numel() * c["sparsity"] // 100])
        one = torch.ones(H, device="cuda")
        layers.append(dict(w_gu=w_gu, w_down=w_down, g_attn=one, g_mlp=one, k=k, tau=[0.0, 0.0, _tau(c["sparsity"]), tau_down]))
    m = DecoderModel(dt, H, 1, 1, M, 8, layers, T=T,
                     select_mode=afx.MODE_TOPK if c["mode"] == "topk" else afx.MODE_THRESHOLD)
    return dict(c=c, m=m, x=_bits(_laplace(g, (c["layers"], T, H)), dt), y=torch.zeros((c["layers"], T, H), device="cuda"))


def _run_mlp(s):
    for layer in range(s["c"]["layers"]):
        s["m"].mlp_block(layer, s["x"][layer], s["y"][layer])
    return s["y"]


def _prepare_decode(c, seed):
    g = _gen(seed)
    H, M, T, NL, dt, kv = c["hidden"], c["mlp"], c["T"], c["layers"], c["dtype"], c["kv_heads"]
    n_attn, n_qkv, max_seq = c["heads"] * 128, (c["heads"] + 2 * kv) * 128, c["past"] + c["steps"]
    k = [synth.keep_count(K, c["sparsity"]) for K in (H, n_attn, H, M)]
    cache = _normal(g, (2, NL, T, max_seq, kv, 128), "f16", 1.0)
    one = torch.ones(H, device="cuda")
    layers = []
    for l in range(NL):
        L = dict(g_attn=one, g_mlp=one, k=k, k_cache=cache[0, l], v_cache=cache[1, l])
        shapes = [("w_qkv", H, n_qkv, H ** -0.5), ("w_o", n_attn, H, 0.05 * n_attn ** -0.5), ("w_gu", H, 2 * M, H ** -0.5),
                  ("w_down", M, H, 0.05 * M ** -0.5)]
        if c["q4"]:
            L["q4"] = [synth.device_q4_weight(seed, 10 * l + i, K, N, sigma) for i, (_, K, N, sigma) in enumerate(shapes)]
        else:
            for name, K, N, sigma in shapes:
                L[name] = _normal(g, (K, N), dt, sigma)
        layers.append(L)
    xl = {"off": afx.XL_OFF, "bookkeep": afx.XL_BOOKKEEP, "reuse": afx.XL_REUSE}[c["xl"]]
    m = DecoderModel(dt, H, c["heads"], kv, M, max_seq, layers, T=T, select_mode=afx.MODE_TOPK,
                     xl_depth=0 if c["xl"] == "off" else 3, xl_mode=xl)
    channel = torch.exp(0.5 * torch.randn(H, generator=g, device="cuda"))
    new = slice(c["past"], max_seq)
    return dict(c=c, m=m, h=m.h, h_in=_laplace(g, (c["steps"], T, H)) * channel,
                h_out=torch.zeros((c["steps"], T, H), device="cuda"), new_kv=cache.view(torch.float16)[:, :, :, new])


def _run_decode(s):
    c, m = s["c"], s["m"]
    step = m.decode_step_q4 if c["q4"] else m.decode_step
    for i in range(c["steps"]):
        s["h"].copy_(s["h_in"][i])
        step(c["past"] + i)
        s["h_out"][i].copy_(s["h"])
    return s["h_out"], s["new_kv"]


def _prepare_moe(c, seed):
    g = _gen(seed)
    H, M, E, dt = c["hidden"], c["mlp"], c["experts"], c["dtype"]
    descs, keep = [], []
    for _ in range(c["layers"]):
        gu = [_normal(g, (H, 2 * M), dt, 0.02) for _ in range(E)]
        down = [_normal(g, (M, H), dt, 0.02) for _ in range(E)]
        router = _normal(g, (H, E), dt, 0.05)
        tables = [torch.tensor([t.data_ptr() for t in ts], dtype=torch.int64, device="cuda") for ts in (gu, down)]
        keep.append((gu, down, router, tables))
        descs.append(afx.MoeDesc(dtype=afx.DTYPES[dt], hidden=H, mlp=M, n_experts=E, top=c["top"], select_mode=afx.MODE_TOPK,
                                 k_gu=synth.keep_count(H, c["sparsity"]), k_down=synth.keep_count(M, c["sparsity"]),
                                 tau_gu=0.0, tau_down=0.0, w_router=router.data_ptr(), ld_router=E,
                                 w_gu_table=tables[0].data_ptr(), w_down_table=tables[1].data_ptr()))
    n = afx.afx_moe_workspace_bytes(descs[0])
    return dict(c=c, descs=descs, keep=keep, n=n, workspace=torch.zeros(n, dtype=torch.uint8, device="cuda"),
                x=_bits(_laplace(g, (c["layers"], H)), dt), y=torch.zeros((c["layers"], H), device="cuda"))


def _run_moe(s):
    for layer, desc in enumerate(s["descs"]):
        afx.afx_moe_block(desc, s["x"][layer], s["y"][layer], 0, s["workspace"], s["n"])
    return s["y"]


class _Cache:
    """A cache handle that is given back with the state that holds it."""

    def __init__(self, desc):
        self.handle = afx.afx_cache_create(desc)

    def __del__(self):
        try:
            torch.cuda.synchronize()
            afx.afx_cache_destroy(self.handle)
        except Exception:
            pass


def _prepare_cached(c, seed):
    g = _gen(seed)
    K, N, dt, steps = c["K"], c["N"], c["dtype"], c["steps"]
    k, capacity = synth.keep_count(K, c["sparsity"]), max(1, K * c["cache_percent"] // 100)
    host = torch.empty((K, N), dtype=torch.int16, pin_memory=True)
    host.copy_(_normal(g, (K, N), dt, 0.02))
    rows = torch.zeros((capacity + k, N), dtype=torch.int16, device="cuda")
    # channel popularity r^-1.1 over a random order, shared by the steps of the sequence
    rank = torch.empty(K, device="cuda")
    rank[torch.randperm(K, generator=g, device="cuda")] = torch.arange(1, K + 1, device="cuda", dtype=torch.float32)
    u = torch.rand((steps, K), generator=g, device="cuda").clamp_(1e-7, 1 - 1e-7)
    sign = torch.where(torch.rand((steps, K), generator=g, device="cuda") < 0.5, -1.0, 1.0)
    x = _bits(torch.exp((-1.1 * torch.log(rank) - torch.log(-torch.log(u))) / 4.0) * sign, dt)
    cache = _Cache(afx.CacheDesc(dtype=afx.DTYPES[dt], K=K, N=N, ldw=N, capacity=capacity, staging_rows=k,
                                 host_base=host.data_ptr(), slots=rows.data_ptr()))
    return dict(c=c, k=k, host=host, rows=rows, x=x, cache=cache, y=torch.zeros((steps, N), device="cuda"),
                idx=torch.zeros((steps, K), dtype=torch.int32, device="cuda"),
                count=torch.zeros((steps, 1), dtype=torch.int32, device="cuda"),
                slot=torch.zeros((steps, K), dtype=torch.int32, device="cuda"))


def _run_cached(s):
    c = s["c"]
    K, N, dt = c["K"], c["N"], c["dtype"]
    afx.afx_cache_reset(s["cache"].handle)  # a new sequence
    for i in range(c["steps"]):
        idx, count, slot = s["idx"][i], s["count"][i], s["slot"][i]
        afx.afx_select_active(s["x"][i], dt, K, 1, afx.MODE_TOPK, s["k"], 0.0, idx, count)
        afx.afx_cache_fetch(s["cache"].handle, idx, count, slot)
        afx.afx_sparse_gemv(s["rows"], dt, K, N, N, s["x"][i], 1, idx, count, slot, s["y"][i], 0)
    return s["y"], s["idx"], s["count"], s["slot"]


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def run(state):
    return globals()["_run_" + state["c"]["kind"]](state)


# ---- what a pass cannot do without --------------------------------------------------------------

def _kept(K, sparsity, T):
    """Expected channels in the union of T tokens' active sets (independent tokens)."""
    return K * (1.0 - (sparsity / 100.0) ** T)


def work(case):
    c = case
    kind, sp, T = c["kind"], c["sparsity"], c.get("T", 1)
    if kind in ("operator", "list"):
        n = c.get("steps", 1)
        a = _kept(c["K"], sp, T) * c["N"]
        return {"bytes": n * (2 * a + 2 * T * c["K"] + 4 * T * c["N"]), "flops": n * 2 * T * a}
    if kind == "mlp":
        a = _kept(c["hidden"], sp, T) * 2 * c["mlp"] + _kept(c["mlp"], sp, T) * c["hidden"]
        return {"bytes": c["layers"] * (2 * a + 6 * T * c["hidden"]), "flops": c["layers"] * 2 * T * a}
    if kind == "decode":
        H, M, n_attn, n_kv = c["hidden"], c["mlp"], c["heads"] * 128, c["kv_heads"] * 128
        a = (_kept(H, sp, T) * (n_attn + 2 * n_kv) + _kept(n_attn, sp, T) * H + _kept(H, sp, T) * 2 * M + _kept(M, sp, T) * H)
        weight_bytes = 0.5625 if c["q4"] else 2
        per_layer = weight_bytes * a + T * 4 * n_kv * (c["past"] + 1)
        flops = 2 * T * a + 4 * T * n_attn * (c["past"] + 1)
        return {"bytes": c["steps"] * (c["layers"] * per_layer + 8 * T * H), "flops": c["steps"] * c["layers"] * flops}
    if kind == "moe":
        a = c["top"] * (_kept(c["hidden"], sp, 1) * 2 * c["mlp"] + _kept(c["mlp"], sp, 1) * c["hidden"])
        router = c["hidden"] * c["experts"]
        return {"bytes": c["layers"] * (2 * a + 2 * router + 6 * c["hidden"]), "flops": c["layers"] * 2 * (a + router)}
    # cached: the active columns once from the cache rows (what crosses the host link depends on the hits)
    a = _kept(c["K"], sp, 1) * c["N"]
    return {"bytes": c["steps"] * (2 * a + 2 * c["K"] + 4 * c["N"]), "flops": c["steps"] * 2 * a}


def tolerance(case):
    kind = case["kind"]
    if kind in ("operator", "list", "cached"):
        # fp32 sums (measured against fp64: 1e-7 on the fp32 pipe, 3e-6 on the tensor cores); lists,
        # counts and slots are whole numbers and exact
        return {"rel": 1e-5, "max": 4e-5}
    if kind in ("mlp", "moe"):
        # rounding of the 16-bit intermediate that tips, and now and then a channel at the boundary of
        # the active set (measured between two summation orders: up to 1.5e-4)
        return {"rel": 1e-3, "max": 4e-3}
    # the same through every layer of the stack (measured with the hidden states moved by one fp32
    # rounding, on 32 layers in bf16: 5e-3 to 1e-2)
    return {"rel": 3e-2}
