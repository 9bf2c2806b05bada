"""GPU parity of the one-token operator where its dispatch and its slices change: the limits of the
selecting warps, 512 and 1024 threads, one granule, ragged last granules, more slices than SMs."""
import numpy as np
import pytest
import torch

import oracle
from paper_2504_08378_b200 import afx, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["topk", "threshold"])
@pytest.mark.parametrize("K,N,dt", [
    (1, 8, "bf16"), (127, 40, "f16"), (64, 80000, "bf16"),          # one channel; one granule and a bit; waves of slices
    (4096, 2048, "bf16"), (4096, 2056, "f16"), (4097, 2040, "f16"),  # 512 / 1024 threads, 8 / 16 selecting warps
    (8200, 4104, "bf16"), (12288, 680, "f16"), (12289, 688, "bf16"),  # 16 / 32 selecting warps
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
