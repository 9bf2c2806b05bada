"""GPU parity of the decoding-step attention at the edges of its tiles and splits: one query head per kv
head (fp32 pipe) and several (tensor cores), against the oracle on the same q, k, v and cache."""
import numpy as np
import pytest
import torch

import oracle
import oracle.layer as ol
from paper_2504_08378_b200 import afx, synth
from paper_2504_08378_b200.model import DecoderModel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pos", [0, 1, 15, 16, 17, 127, 128, 129, 1100])
@pytest.mark.parametrize("kvh,rep,T", [(3, 1, 2), (13, 1, 3), (5, 2, 1), (2, 3, 3), (1, 8, 1)])
def test_attention_matches_oracle_at_tile_edges(pos, kvh, rep, T):
    dt, heads, scale = "f16", kvh * rep, [1.0, 30.0, 1e-3][pos % 3]
    hidden, mlp, max_seq = 128, 64, pos + 1
    cfg = ol.Config(dt, hidden, heads, kvh, mlp)
    L = synth.layer_weights(41, 0, hidden, heads, kvh, mlp, dt)
    kc0, vc0 = synth.kv_cache(41, 0, T, max_seq, kvh, pos)
    L["k_cache"], L["v_cache"], L["k"] = kc0, vc0, [hidden, heads * 128, hidden, mlp]
    m = DecoderModel(dt, hidden, heads, kvh, mlp, max_seq, [L], T=T)
    qkv = scale * np.random.default_rng(pos).standard_normal(m.qkv.shape).astype(np.float32)
    m.qkv.copy_(torch.from_numpy(qkv).cuda())
    m.layer_kernel(0, pos, afx.STEP_ATTN)
    torch.cuda.synchronize()
    kc, vc = kc0.copy(), vc0.copy()
    ref = oracle.decode(ol.attention_stage(cfg, qkv.astype(np.float64), kc, vc, pos), dt)
    got = oracle.decode(m.bits(afx.BUF_ATTN).cpu().numpy().view(np.uint16), dt)
    # fp32 scores of up to |q||k| / sqrt(128) <~ 30 * 30 carry an absolute error of some 1e-4 into the
    # exponent (and 64 half-ulp steps of a new row tipped in fp16); the result is rounded to fp16
    err = np.abs(got - ref) / np.maximum(np.abs(ref), np.sqrt((ref ** 2).mean()))
    assert err.max() <= 2 * 2.0 ** -11 + 1e-3
    for cache, want, before in ((m.k_cache[0], kc, kc0), (m.v_cache[0], vc, vc0)):
        have = cache.cpu().numpy().view(np.uint16)
        assert np.array_equal(have[:, :pos], before[:, :pos])
        assert np.abs(have[:, pos].astype(np.int32) - want[:, pos].astype(np.int32)).max() <= 1
    m.close()


@pytest.mark.parametrize("kvh,rep,T", [(4, 1, 1), (8, 1, 4), (4, 4, 1), (2, 8, 2)])
def test_attention_calls_in_a_row_see_each_others_rows(kvh, rep, T):
    """The attention kernel of one layer at consecutive (and earlier) positions without any other kernel between: each
    call must read the rows that the calls before it wrote, not what the cache held."""
    dt, heads, start, n = "bf16", kvh * rep, 37, 24
    hidden, mlp, max_seq = 128, 64, start + n
    positions = list(range(start, max_seq)) + [5, max_seq - 1, 3, 6]
    L = synth.layer_weights(43, 0, hidden, heads, kvh, mlp, dt)
    kc0, vc0 = synth.kv_cache(43, 0, T, max_seq, kvh, max_seq)
    L["k_cache"], L["v_cache"], L["k"] = kc0, vc0, [hidden, heads * 128, hidden, mlp]
    m = DecoderModel(dt, hidden, heads, kvh, mlp, max_seq, [L], T=T)
    qkv = torch.from_numpy(np.random.default_rng(7).standard_normal(m.qkv.shape).astype(np.float32)).cuda()
    qkv[:, -kvh * 128:] *= 50  # values of new rows unlike the old ones
    got = []
    for sync in (True, False):
        m.k_cache[0].copy_(torch.from_numpy(kc0.view(np.int16)))
        m.v_cache[0].copy_(torch.from_numpy(vc0.view(np.int16)))
        m.qkv.copy_(qkv)
        torch.cuda.synchronize()
        outs = torch.empty((len(positions), *m.bits(afx.BUF_ATTN).shape), dtype=torch.int16, device="cuda")
        for i, pos in enumerate(positions):
            m.layer_kernel(0, pos, afx.STEP_ATTN)
            if sync:
                torch.cuda.synchronize()
                outs[i] = m.bits(afx.BUF_ATTN)
        if not sync:
            outs[-1] = m.bits(afx.BUF_ATTN)
        got.append((outs[-1].clone(), m.k_cache[0].clone(), m.v_cache[0].clone()))
    assert all(torch.equal(a, b) for a, b in zip(*got))
    # the last call, at position 6, read the rows of the calls at 3 and 5
    q = qkv.double().cpu().numpy()
    kc, vc = (got[0][i].cpu().numpy().view(np.uint16).copy() for i in (1, 2))
    ref = oracle.decode(ol.attention_stage(ol.Config(dt, hidden, heads, kvh, mlp), q, kc, vc, positions[-1]), dt)
    out = oracle.decode(got[0][0].cpu().numpy().view(np.uint16), dt)
    assert np.abs(out - ref).max() <= 2.0 ** -8 * np.abs(ref).max()  # one rounding to bf16
    m.close()


@pytest.mark.parametrize("kvh,rep", [(4, 1), (8, 2), (4, 4), (2, 8)])
@pytest.mark.parametrize("pos", [60, 200])
def test_attention_keeps_32_bit_precision(kvh, rep, pos):
    """Share of fp16 outputs that are not the nearest ones.  An error of e times the sum of p |v| before the last
    rounding tips 2 e sum(p |v|) / ulp of them: with e = 2^-20, ulp ~ 2^-10.5 |out| and sum(p |v|) / |out| ~ 10 at 200
    positions of random values 1.4 %.  Queries or probabilities in a single fp16 number tip a third."""
    dt, heads, T = "f16", kvh * rep, 2
    hidden, mlp, max_seq = 128, 64, pos + 1
    cfg = ol.Config(dt, hidden, heads, kvh, mlp)
    L = synth.layer_weights(47, 0, hidden, heads, kvh, mlp, dt)
    kc, vc = synth.kv_cache(47, 0, T, max_seq, kvh, pos)
    L["k_cache"], L["v_cache"], L["k"] = kc.copy(), vc.copy(), [hidden, heads * 128, hidden, mlp]
    m = DecoderModel(dt, hidden, heads, kvh, mlp, max_seq, [L], T=T)
    qkv = np.random.default_rng(pos).standard_normal(m.qkv.shape).astype(np.float32)
    m.qkv.copy_(torch.from_numpy(qkv).cuda())
    m.layer_kernel(0, pos, afx.STEP_ATTN)
    ref = ol.attention_stage(cfg, qkv.astype(np.float64), kc, vc, pos)
    assert (m.bits(afx.BUF_ATTN).cpu().numpy().view(np.uint16) != ref).mean() <= 0.014
    m.close()


@pytest.mark.parametrize("kvh,rep", [(3, 2), (2, 8)])
@pytest.mark.parametrize("pos", [17, 200])
def test_attention_with_infinities_in_the_cache(kvh, rep, pos):
    """fp16 caches overflow to infinity.  A key that makes every head's score -inf leaves its position out (the only
    past one of a tile among them); an infinite value makes its dimension infinite and nothing else."""
    dt, heads, T = "f16", kvh * rep, 1
    hidden, mlp, max_seq = 128, 64, pos + 1
    cfg = ol.Config(dt, hidden, heads, kvh, mlp)
    L = synth.layer_weights(53, 0, hidden, heads, kvh, mlp, dt)
    kc, vc = synth.kv_cache(53, 0, T, max_seq, kvh, pos)
    qkv = np.random.default_rng(pos).standard_normal((T, (heads + 2 * kvh) * 128)).astype(np.float32)
    rot = np.stack([oracle.rope(qkv[0, h * 128:(h + 1) * 128].reshape(1, 1, 128), np.full(1, pos, np.int32))[0, 0] for h in range(heads)])
    for g in range(kvh):
        d = 127  # a dimension in which all queries of the group are made positive
        for h in range(g * rep, (g + 1) * rep):
            if rot[h, d] <= 0:
                qkv[0, h * 128:(h + 1) * 128] *= -1
        for p in (0, 5, 16):
            kc[0, p, g, d] = 0xFC00  # -inf
        vc[0, 3, g, 10] = 0x7C00
        vc[0, pos - 1 if pos > 17 else 15, g, 77] = 0xFC00  # (200: the row that fills up the last tile)
    L["k_cache"], L["v_cache"], L["k"] = kc.copy(), vc.copy(), [hidden, heads * 128, hidden, mlp]
    m = DecoderModel(dt, hidden, heads, kvh, mlp, max_seq, [L], T=T)
    m.qkv.copy_(torch.from_numpy(qkv).cuda())
    m.layer_kernel(0, pos, afx.STEP_ATTN)
    got = oracle.decode(m.bits(afx.BUF_ATTN).cpu().numpy().view(np.uint16), dt).reshape(heads, 128)
    K, V = (oracle.decode(c.cpu().numpy().view(np.uint16), "f16")[0] for c in (m.k_cache[0], m.v_cache[0]))
    for h in range(heads):
        q = oracle.rope(qkv[0, h * 128:(h + 1) * 128].reshape(1, 1, 128).astype(np.float64), np.full(1, pos, np.int32))[0, 0]
        sc = K[:, h // rep] @ q / np.sqrt(128.0)
        w = np.exp(sc - sc.max())
        want = (w[:, None] * V[:, h // rep]).sum(0) / w.sum()
        fin = np.isfinite(want)
        assert (~fin).sum() >= 1 and np.array_equal(got[h][~fin], want[~fin])
        assert np.abs(got[h][fin] - want[fin]).max() <= 2 * 2.0 ** -11 * np.abs(want[fin]).max()
    m.close()
