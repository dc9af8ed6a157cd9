"""The split selection and gather kernels (few instances, long caches) against
the oracle: budgets at the edges of the 256-row chunks, one eviction, both head
sizes, leading rows kept, per-instance lengths, and the same caches through the
fused kernel (a batch large enough for it) bit for bit."""
import pytest
import torch

from paper_2609_04971_gb300.workloads import QWEN3_4B, TINY

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from tests import parity as P


@pytest.mark.parametrize("wl,L,budget,prefix", [
    (TINY, 2777, 1024, 0), (TINY, 1281, 1280, 3), (TINY, 3000, 1025, 0), (TINY, 2049, 2047, 0),
    (QWEN3_4B, 1600, 1279, 0), (QWEN3_4B, 1601, 1600, 4), (QWEN3_4B, 5000, 1536, 0), (QWEN3_4B, 29000, 28673, 0),
], ids=lambda v: getattr(v, "name", str(v))[:8])
def test_split_matches_oracle(wl, L, budget, prefix):
    wl = wl.scaled(name=f"split_{wl.head_dim}_{L}_{budget}", n_layers=1, batch=1, L=L, budget=budget, n_prefix=prefix)
    P.check_run(P.run_gpu(wl, seed=L + budget))


@pytest.mark.parametrize("d", [64, 128])
def test_split_equals_fused(d):
    """The first instances of a batch that takes the fused kernel, compressed alone, take the split one."""
    from paper_2609_04971_gb300 import bkv
    L, budget, W, nb, big = 1500, 1111, 8, 4, 700
    g = torch.Generator(device="cuda").manual_seed(d)
    K, V = (torch.randn(big, 1, 1, L, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    K[:, :, :, 100:140] = K[:, :, :, 60:100]  # tied scores
    q = torch.randn(big, 1, 2, W, d, generator=g, device="cuda").to(torch.bfloat16)
    qi = torch.randn(big, 1, 2, 16, d, generator=g, device="cuda").to(torch.bfloat16)
    lens = torch.randint(budget - 50, L + 1, (big, 1, 1), generator=g, device="cuda", dtype=torch.int32)
    out = {}
    for n in (big, 7):
        for ragged in (False, True):
            bk = bkv.BeaconKV(n_layers=n, batch=1, n_q_heads=2, n_kv_heads=1, head_dim=d, n_beacons=nb, window=W,
                              capacity=L, rope_theta=1e4)
            try:
                bk.init_beacons(qi[:n].contiguous())
                k, v = K[:n].clone(), V[:n].clone()
                pos = [2000 + w for w in range(W)]
                if ragged:
                    kept = bk.compress_ragged(k, v, L=lens[:n].contiguous(), budget=budget, t_pos=[2007],
                                              q_recent=q[:n].contiguous(), recent_pos=[pos])
                else:
                    kept = bk.compress(k, v, L=L, budget=budget, t_pos=2007, q_recent=q[:n].contiguous(), recent_pos=pos)
                bk.sync()
                out[n, ragged] = (kept[:7].clone(), k[:7].clone(), v[:7].clone())
            finally:
                bk.close()
    for ragged in (False, True):
        for a, b in zip(out[big, ragged], out[7, ragged]):
            assert torch.equal(a, b)
