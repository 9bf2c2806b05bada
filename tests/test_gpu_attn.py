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
