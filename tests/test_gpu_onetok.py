"""GPU parity of the one-token operator where its dispatch and its slices change: the limits of the
selecting warps, 512 and 1024 threads, one granule, ragged last granules, more slices than SMs, clusters
that share a granule's list."""
import numpy as np
import pytest
import torch

import oracle
import oracle.layer as ol
from paper_2504_08378_b200 import afx, synth
from test_gpu_layer import OPN, check_layer_stages, make, oracle_weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["topk", "threshold"])
@pytest.mark.parametrize("K,N,dt", [
    (1, 8, "bf16"), (127, 40, "f16"), (64, 80000, "bf16"),          # one channel; one granule and a bit; waves of slices
    (4096, 2048, "bf16"), (4096, 2056, "f16"), (4097, 2040, "f16"),  # 512 / 1024 threads, 8 / 16 selecting warps
    (8200, 4104, "bf16"), (12288, 680, "f16"), (12289, 688, "bf16"),  # 6 / 8 slots per lane
    (16384, 4608, "bf16"), (16385, 4608, "f16"), (16385, 2048, "f16"),  # 16 / 32 selecting warps
    (6143, 64, "bf16"), (6144, 64, "bf16"), (6144, 1120, "f16"), (6144, 1160, "f16"),  # clusters that share a list
    (16384, 520, "bf16"), (16385, 264, "bf16"), (32768, 8, "bf16"),
    (32768, 96, "f16"),
])
def test_one_token_operator_at_dispatch_edges(K, N, dt, mode):
    rng = np.random.default_rng(K + N)
    torch_dt = torch.float16 if dt == "f16" else torch.bfloat16
    x = torch.from_numpy(rng.laplace(size=K).astype(np.float32)).to(torch_dt).cuda()
    W = (0.02 * torch.from_numpy(rng.standard_normal((K, N), dtype=np.float32))).to(torch_dt).cuda()
    bits = lambda t: t.view(torch.int16)
    k, tau = synth.keep_count(K, 50), 0.7
    y = torch.zeros(N, device="cuda")
    idx, count = torch.zeros(K, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    hint = torch.zeros(1, dtype=torch.int32, device="cuda")
    xb = bits(x).cpu().numpy().view(np.uint16)
    want = oracle.select_active(xb, dt, oracle.TOPK if mode == "topk" else oracle.THRESHOLD, k=k, tau=tau)
    for _ in range(2):  # without a hint of the k-th key, then with one
        y.zero_()
        afx.afx_select_gemv(bits(W), dt, K, N, N, bits(x), 1, afx.MODE_TOPK if mode == "topk" else afx.MODE_THRESHOLD, k, tau,
                            y, 0, idx, count, kth_hint=hint)
        assert np.array_equal(idx.cpu().numpy()[: int(count)], want)
        a = torch.from_numpy(want.astype(np.int64)).cuda()
        w, xa = W[a].double(), x[a].double()
        # sums of fp32 products in any order: at most K / 2 additions, each within 2^-24 of the running sum
        bound = (len(want) + 2) * 2.0 ** -24 * (w.abs() * xa.abs()[:, None]).sum(0)
        assert bool(((y.double() - (w * xa[:, None]).sum(0)).abs() <= bound).all())


@pytest.mark.parametrize("K,N,keep,dt", [(20000, 64, 20000, "f16"), (8193, 1032, 8193, "bf16"), (64, 80000, 33, "bf16"),
                                         (4096, 2056, 1, "f16"), (4096, 2048, 0, "bf16")])
def test_given_list_at_pass_and_slice_edges(K, N, keep, dt):
    """One token with a given list: more entries than a pass holds, both block sizes, waves of slices, none."""
    rng = np.random.default_rng(K + N)
    torch_dt = torch.float16 if dt == "f16" else torch.bfloat16
    x = torch.from_numpy(rng.standard_normal(K).astype(np.float32)).to(torch_dt).cuda()
    W = (0.02 * torch.from_numpy(rng.standard_normal((K, N), dtype=np.float32))).to(torch_dt).cuda()
    want = np.sort(rng.permutation(K)[:keep]).astype(np.int32)
    idx = torch.zeros(K, dtype=torch.int32, device="cuda")
    idx[:keep] = torch.from_numpy(want).cuda()
    count = torch.tensor([keep], dtype=torch.int32, device="cuda")
    y = torch.full((N,), 0.5, device="cuda")
    afx.afx_sparse_gemv(W.view(torch.int16), dt, K, N, N, x.view(torch.int16), 1, idx, count, None, y, 1)
    a = torch.from_numpy(want.astype(np.int64)).cuda()
    w, xa = W[a].double(), x[a].double()[:, None]
    bound = (keep + 3) * 2.0 ** -24 * ((w.abs() * xa.abs()).sum(0) + 0.5)  # any order of fp32 additions
    assert bool(((y.double() - 0.5 - (w * xa).sum(0)).abs() <= bound).all())


@pytest.mark.parametrize("K", [33, 4096, 4097, 8193, 16385, 32768])
@pytest.mark.parametrize("T", [1, 2, 8])
@pytest.mark.parametrize("dt,mode", [("bf16", "topk"), ("f16", "topk"), ("f16", "threshold")])
def test_selection_of_tokens_at_warp_limits(K, T, dt, mode):
    """Union over tokens with few distinct magnitudes (ties at the boundary), one token all zero."""
    rng = np.random.default_rng(K + T)
    x = np.round(rng.laplace(size=(T, K)) * 4) / 4
    x[-1] *= T == 1
    bits = torch.from_numpy(x.astype(np.float32)).to(torch.float16 if dt == "f16" else torch.bfloat16).view(torch.int16).cuda()
    k, tau = max(1, K // 3), 0.75
    want = oracle.select_active(bits.cpu().numpy().view(np.uint16), dt, oracle.TOPK if mode == "topk" else oracle.THRESHOLD, k=k, tau=tau)
    idx, count = torch.zeros(K, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    bitmap = torch.zeros((K + 31) // 32, dtype=torch.int32, device="cuda")
    afx.afx_select_active(bits, dt, K, T, afx.MODE_TOPK if mode == "topk" else afx.MODE_THRESHOLD, k, tau, idx, count, bitmap)
    assert np.array_equal(idx.cpu().numpy()[: int(count)], want)
    flags = np.unpackbits(bitmap.cpu().numpy().view(np.uint8), bitorder="little")[:K]
    assert np.array_equal(np.flatnonzero(flags), want)


@pytest.mark.parametrize("K,N,dt", [(512, 256, "f16"), (4096, 512, "bf16"), (11008, 1024, "bf16")])
def test_calls_in_a_row_share_a_hint(K, N, dt):
    """The next launch reads the hint while the one before rewrites it, and the hints are far apart: every block
    must search from ONE of the two values, and the lists must not depend on which."""
    rng = np.random.default_rng(K + N)
    torch_dt = torch.float16 if dt == "f16" else torch.bfloat16
    x = torch.from_numpy(rng.laplace(size=(2, K)) * np.array([[1.0], [1.0 / 64]])).to(torch_dt).cuda().view(torch.int16)
    W = (0.02 * torch.from_numpy(rng.standard_normal((K, N), dtype=np.float32))).to(torch_dt).cuda().view(torch.int16)
    k, calls = synth.keep_count(K, 50), 64
    y = torch.zeros((calls, N), device="cuda")
    idx = torch.zeros((calls, K), dtype=torch.int32, device="cuda")
    count = torch.zeros(calls, dtype=torch.int32, device="cuda")
    want = [oracle.select_active(v.cpu().numpy().view(np.uint16), dt, oracle.TOPK, k=k) for v in x]
    hint = torch.zeros(1, dtype=torch.int32, device="cuda")
    for i in range(calls):
        if i % 16 == 0:
            hint.zero_()
        afx.afx_select_gemv(W, dt, K, N, N, x[i % 2], 1, afx.MODE_TOPK, k, 0.0, y[i], 0, idx[i], count[i], kth_hint=hint)
    assert count.tolist() == [k] * calls
    for i in range(calls):
        assert np.array_equal(idx[i, :k].cpu().numpy(), want[i % 2]), i
        assert torch.equal(y[i], y[i % 2])


@pytest.mark.parametrize("K", [1536, 5000])
@pytest.mark.parametrize("N", [8, 264, 1168, 1176, 1184, 2352, 2360, 2368])
def test_one_token_on_slices_of_fewer_pieces(K, N):
    """Slices of one and two 16-byte pieces per row, at the outputs where the next smaller ones begin."""
    g = torch.Generator(device="cuda")
    g.manual_seed(K + N)
    W = torch.randn(K, N, generator=g, device="cuda").mul_(0.02).to(torch.bfloat16)
    x = torch.randn(K, generator=g, device="cuda").to(torch.bfloat16)
    k = K // 2
    want = oracle.select_active(x.view(torch.int16).cpu().numpy().view(np.uint16)[None], "bf16", oracle.TOPK, k=k)
    a = torch.from_numpy(want.astype(np.int64)).cuda()
    w, xa = W[a].double(), x[a].double()[:, None]
    bound = (k + 3) * 2.0 ** -24 * ((w.abs() * xa.abs()).sum(0) + 0.5)  # any order of fp32 additions
    for side in (False, True):
        y = torch.full((N,), 0.5, device="cuda")
        idx, count = torch.zeros(K, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        afx.afx_select_gemv(W.view(torch.int16), "bf16", K, N, N, x.view(torch.int16), 1, afx.MODE_TOPK, k, 0.0, y, 1,
                            idx if side else None, count if side else None)
        assert bool(((y.double() - 0.5 - (w * xa).sum(0)).abs() <= bound).all())
        if side:
            assert int(count) == k and np.array_equal(idx[:k].cpu().numpy(), want)


@pytest.mark.parametrize("dt", ["bf16", "f16"])
@pytest.mark.parametrize("K,N,rows", [(2304, 4096, 256), (4096, 4072, 256), (2304, 5632, 128), (1200, 7272, 128), (8192, 4096, 256)])
def test_one_token_where_all_rows_of_a_thread_are_in_flight(K, N, rows, dt):
    """Lists of six rows per thread, just above, eight, and just above; stored and added."""
    g = torch.Generator(device="cuda")
    g.manual_seed(K + N)
    td = torch.bfloat16 if dt == "bf16" else torch.float16
    W = torch.randn(K, N, generator=g, device="cuda").mul_(0.02).to(td)
    x = torch.randn(K, generator=g, device="cuda").to(td)
    for k in (6 * rows, 6 * rows + 1, 7 * rows - 3, 8 * rows, 8 * rows + 1):
        want = oracle.select_active(x.view(torch.int16).cpu().numpy().view(np.uint16)[None], dt, oracle.TOPK, k=k)
        a = torch.from_numpy(want.astype(np.int64)).cuda()
        w, xa = W[a].double(), x[a].double()
        for accumulate in (0, 1):
            y = torch.full((N,), 0.5, device="cuda")
            idx, count = torch.zeros(K, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
            afx.afx_select_gemv(W.view(torch.int16), dt, K, N, N, x.view(torch.int16), 1, afx.MODE_TOPK, k, 0.0, y, accumulate, idx, count)
            bound = (k + 3) * 2.0 ** -24 * (xa.abs() @ w.abs() + 0.5)  # any order of fp32 additions
            assert bool(((y.double() - 0.5 * accumulate - xa @ w).abs() <= bound).all()), k
            assert int(count) == k and np.array_equal(idx[:k].cpu().numpy(), want), k


@pytest.mark.parametrize("dt,half", [("bf16", 32), ("f16", 128)])
@pytest.mark.parametrize("K", [160, 4096, 12296])
@pytest.mark.parametrize("lo,hi", [(0, 40), (0x3C00, 0x3C90), (0x7F00, 0x7F81)])
def test_hints_at_the_edges_of_the_counted_window(K, dt, half, lo, hi):
    """Keys at the bottom, in the middle and at the top of the range (f16: NaN patterns), many of them equal; the k-th
    key lies at the first and last key of the window around the hint, and just outside."""
    rng = np.random.default_rng(K + lo)
    keys = rng.integers(lo, hi, K)
    x = (keys | (rng.integers(0, 2, K) << 15)).astype(np.uint16)
    k = K // 2
    want = oracle.select_active(x[None], dt, oracle.TOPK, k=k)
    kth = int(np.sort(keys)[::-1][k - 1])
    W = torch.zeros((K, 256), dtype=torch.int16, device="cuda")
    xd, y = torch.from_numpy(x.view(np.int16)).cuda(), torch.zeros(256, device="cuda")
    for off in (0, half - 1, half, half + 1, -half + 1, -half, -half - 1):
        hint = torch.tensor([0x10000 | min(0x7FFF, max(0, kth + off))], dtype=torch.int32, device="cuda")
        idx, count = torch.zeros(K, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        afx.afx_select_gemv(W, dt, K, 256, 256, xd, 1, afx.MODE_TOPK, k, 0.0, y, 0, idx, count, kth_hint=hint)
        assert int(count) == k and np.array_equal(idx[:k].cpu().numpy(), want), off
        assert int(hint) == 0x10000 | kth


@pytest.mark.parametrize("dt,half,near", [("bf16", 32, 49), ("f16", 128, 343)])
@pytest.mark.parametrize("K,zeros", [(160, 0.0), (4096, 0.0), (12296, 0.0), (1000, 0.49), (4096, 0.6)])
def test_hints_whose_window_misses(K, zeros, dt, half, near):
    """The search from the window outwards: the k-th key at, before and behind the first, second and last of the next
    candidates, beyond all of them, and among zeros."""
    rng = np.random.default_rng(K)
    keys = rng.integers(0x1000, 0x6000, K)
    keys[rng.random(K) < zeros] = 0
    x = (keys | (rng.integers(0, 2, K) << 15)).astype(np.uint16)
    k = K // 2
    want = oracle.select_active(x[None], dt, oracle.TOPK, k=k)
    kth = int(np.sort(keys)[::-1][k - 1])
    W = torch.zeros((K, 256), dtype=torch.int16, device="cuda")
    xd, y = torch.from_numpy(x.view(np.int16)).cuda(), torch.zeros(256, device="cuda")
    for d in [half + m * near + e for m in (0, 1, 2, 6) for e in (-1, 0, 1, 2)] + [6000, 12000, 24000]:
        for hint in {min(0x7FFF, kth + d), max(0, kth - d)}:
            slot = torch.tensor([0x10000 | hint], dtype=torch.int32, device="cuda")
            idx, count = torch.zeros(K, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
            afx.afx_select_gemv(W, dt, K, 256, 256, xd, 1, afx.MODE_TOPK, k, 0.0, y, 0, idx, count, kth_hint=slot)
            assert int(count) == k and np.array_equal(idx[:k].cpu().numpy(), want), (d, hint)
            assert int(slot) == 0x10000 | kth


@pytest.mark.parametrize("hidden,mlp", [(12296, 2312), (16392, 264), (8192, 64), (2048, 552), (1536, 1192)])
def test_layer_of_very_wide_hidden_state(hidden, mlp):
    """Gains read late (8 slots per lane), normed operators by clusters and by slices, a family of side outputs: two
    layers, the second compared with the first one's sets."""
    dt, pos, T = "bf16", 9, 1
    cfg = ol.Config(dt, hidden, 1, 1, mlp, mode=oracle.TOPK, xl_depth=1, xl_mode=1)
    k = [synth.keep_count(K, 50) for K in (hidden, 128, hidden, mlp)]
    L = synth.layer_weights(59, 0, hidden, 1, 1, mlp, dt, gain_jitter=0.1)
    kc, vc = synth.kv_cache(59, 0, T, 16, 1, pos)
    L["k"], L["k_cache"], L["v_cache"] = k, kc, vc
    m = make(cfg, [L, L], T, afx.MODE_TOPK, xl_depth=1, xl_mode=afx.XL_BOOKKEEP, max_seq=16)
    h = synth.hidden_state(59, 5, T, hidden, scale=4.0, scales_stream=6)
    m.h.copy_(torch.from_numpy(h).cuda())
    sets = []
    for layer in (0, 1):
        h0 = m.h.cpu().numpy().copy()
        m.layer_step(layer, pos)
        torch.cuda.synchronize()
        check_layer_stages(cfg, L, oracle_weights(L, k), m, layer, h0, kc, vc, pos, T)
        stats = m.stats.cpu().numpy()[layer]
        sets.append([m.idx(op).cpu().numpy()[: stats[op][0]].copy() for op in range(4)])
        if layer == 1:
            for op in range(4):
                miss, hit = oracle.diff_active(sets[1][op], sets[0][op], m.K_op[op])
                assert stats[op][1] == hit and stats[op][2] == len(miss), OPN[op]
                assert np.array_equal(m.miss(op).cpu().numpy()[: len(miss)], miss)
    m.close()


@pytest.mark.parametrize("hidden,mlp,E,top", [(8192, 512, 3, 2), (512, 8192, 4, 3), (256, 16392, 2, 1)])
def test_expert_families_by_clusters(hidden, mlp, E, top):
    """Experts whose operators are narrow with long lists, against the same call's own intermediates in fp64."""
    from test_gpu_moe import run_moe
    dt = "bf16"
    ex = [synth.layer_weights(61, e, hidden, 1, 1, mlp, dt) for e in range(E)]
    Wr = synth.weight(61, 99, hidden, E, dt, sigma=0.05)
    x = synth.laplace_bits(61, 7, (1, hidden), dt)
    k_gu, k_down = hidden // 2, mlp // 2
    ids, w, _ = ol.moe_router(x, Wr, dt, top)
    lg, sel, wsel, hm, y = run_moe(dt, hidden, mlp, E, top, ex, Wr, x, k_gu, k_down)
    assert sel.tolist() == ids.tolist()
    ref = np.zeros((1, hidden))
    idx = oracle.select_active(x, dt, oracle.TOPK, k=k_gu)
    for r in range(top):
        e = ex[int(sel[r])]
        g, u = (oracle.sparse_gemv(e[n], dt, mlp, x, idx) for n in ("w_gate", "w_up"))
        want = oracle.decode(oracle.silu_mul(g, u, dt), dt)
        got = oracle.decode(hm[r][None, :], dt)
        assert np.abs(got - want).max() <= 2.0 ** -7 * np.abs(want).max()
        ref += float(wsel[r]) * oracle.sparse_gemv(e["w_down"], dt, hidden, hm[r], oracle.select_active(hm[r], dt, oracle.TOPK, k=k_down))
    assert np.abs(y - ref).max() <= 2e-5 * np.sqrt((ref ** 2).mean()) * 10
