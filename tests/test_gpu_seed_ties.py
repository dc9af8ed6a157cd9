"""Prefill seeding where rows tie exactly: the lowest index wins, and no row is picked twice.

Copies of a row scaled by different powers of two have exactly equal cosines with everything, in fp64 as in
the kernel's double-float arithmetic, and each copy can be told from the others, so the picks themselves are
checked.  Equal rows (repeated tokens, zero rows) cannot be told apart: there no value may be picked more
often than it occurs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from tests import parity as P


def _seed(x, nb):
    from paper_2609_04971_gb300 import bkv
    n_inst, n, d = x.shape
    bk = bkv.BeaconKV(n_layers=n_inst, batch=1, n_q_heads=1, n_kv_heads=1, head_dim=d, n_beacons=nb, window=8,
                      capacity=64)
    try:
        bk.init_beacons(x.view(n_inst, 1, 1, n, d).cuda())
        cent = bk.state()[0].cpu().numpy().reshape(n_inst, nb, d)
        bk.sync()
    finally:
        bk.close()
    return cent


def _picks(rows, cent, tag):
    """The rows that the centroids are copies of, each checked to be left and, in fp64, as far as the farthest
    row left (rows may tie to the last bits of the arithmetic: a row's cosine with its own copy is 1 there)."""
    norm = np.linalg.norm(rows, axis=1, keepdims=True)
    unit = np.divide(rows, norm, out=np.zeros_like(rows), where=norm > 0)
    far = unit @ unit.sum(0) / len(rows)
    left, out = np.ones(len(rows), bool), []
    for k in range(len(cent)):
        same = np.flatnonzero(left & (rows == cent[k]).all(-1))
        assert len(same) > 0, f"{tag}: pick {k} is not one of the rows left"
        r = int(same[0])
        assert far[r] <= far[left].min() + P.ASSIGN_TIE, f"{tag} pick {k}"
        left[r] = False
        cos = unit @ unit[r]
        far = cos if k == 0 else np.maximum(far, cos)
        out.append(r)
    return out


@pytest.mark.parametrize("n,d,nb,m,spread", [
    (12, 128, 8, 3, 1.0), (16, 64, 16, 2, 1.0), (40, 128, 32, 5, 0.0), (100, 64, 20, 7, 0.01), (128, 128, 8, 8, 1.0),
    (200, 128, 16, 13, 0.003), (256, 64, 32, 16, 0.0), (272, 128, 8, 17, 1.0), (720, 128, 12, 45, 0.01),
    (1000, 128, 9, 63, 1.0), (2050, 64, 6, 129, 0.0), (4096, 128, 5, 256, 1.0),
])
def test_scaled_copies_are_picked_by_lowest_index(n, d, nb, m, spread):
    """m directions (spread 0: nearly one), each at up to 16 scales, in a shuffled order."""
    n_inst = 2 if n > 1000 else 6
    rng = np.random.default_rng(n + nb)
    x = np.empty((n_inst, n, d), np.float32)
    for e in range(n_inst):
        base = rng.standard_normal((1, d)) + (spread or 1e-4) * rng.standard_normal((m, d)) if spread < 1 else \
            rng.standard_normal((m, d))
        base = torch.from_numpy(base).to(torch.bfloat16).float().numpy()
        kinds = rng.permutation(n)
        x[e] = base[kinds % m] * 2.0 ** (kinds // m % 17 - 8)[:, None]
    t = torch.from_numpy(x).to(torch.bfloat16)
    cent = _seed(t, nb)
    for e in range(n_inst):
        rows = t[e].double().numpy()
        unit = rows / np.linalg.norm(rows, axis=1, keepdims=True)
        _, kind = np.unique(unit.round(9), axis=0, return_inverse=True)  # copies of one direction
        left = np.ones(n, bool)
        for k, r in enumerate(_picks(rows, cent[e], f"instance {e}")):
            # of one direction's copies the first one left wins
            assert r == np.flatnonzero(left & (kind.ravel() == kind.ravel()[r]))[0], f"instance {e} pick {k}: row {r}"
            left[r] = False


@pytest.mark.parametrize("n,d,nb,kind", [
    (16, 128, 16, "all_equal"), (130, 64, 32, "all_equal"), (256, 128, 8, "all_equal"), (600, 128, 20, "all_equal"),
    (33, 128, 20, "repeated"), (256, 128, 32, "repeated"), (900, 64, 16, "repeated"), (2500, 128, 8, "repeated"),
    (64, 64, 24, "zero_rows"), (256, 128, 32, "zero_rows"), (1200, 128, 10, "zero_rows"),
])
def test_equal_rows_are_picked_as_often_as_they_occur_at_most(n, d, nb, kind):
    n_inst = 4
    rng = np.random.default_rng(7 * n + nb)
    x = rng.standard_normal((n_inst, n, d)).astype(np.float32)
    if kind == "all_equal":
        x[:] = x[:, :1]
    elif kind == "repeated":  # about nb - 3 different rows, so that repeats have to be picked
        x = np.take_along_axis(x, rng.integers(0, max(2, nb - 3), (n_inst, n, 1)), 1)
    else:  # more zero rows than others, fewer others than beacons
        x[rng.random((n_inst, n)) < 1.0 - (nb - 2) / n] = 0.0
    t = torch.from_numpy(x).to(torch.bfloat16)
    cent = _seed(t, nb)
    for e in range(n_inst):
        _picks(t[e].double().numpy(), cent[e], f"instance {e}")


def _time(x, nb):
    from paper_2609_04971_gb300 import bkv
    n_inst, n, d = x.shape
    bk = bkv.BeaconKV(n_layers=n_inst, batch=1, n_q_heads=1, n_kv_heads=1, head_dim=d, n_beacons=nb, window=8,
                      capacity=64)
    q, best = x.view(n_inst, 1, 1, n, d), float("inf")
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for r in range(8):
        e0.record()
        bk.init_beacons(q)
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1)) if r >= 2 else best
    bk.close()
    return best


@pytest.mark.parametrize("kind,times", [("all_equal", 4.0), ("repeated", 3.0), ("zero_rows", 3.5), ("near_equal", 7.5)])
def test_ties_cost_a_few_times_the_time(kind, times):
    """Rows that tie are compared in double-float arithmetic; comparing repeats of one row like others, a row
    at a time from global memory, took 4 to 9 times as long as rows that do not tie."""
    n_inst, n, d, nb = 4608, 256, 128, 8
    g = torch.Generator(device="cuda").manual_seed(3)

    def clusters(n):
        c = torch.randn(n_inst, 8, d, generator=g, device="cuda")
        k = torch.randint(0, 8, (n_inst, n, 1), generator=g, device="cuda").expand(n_inst, n, d)
        return torch.gather(c, 1, k) + 0.15 * torch.randn(n_inst, n, d, generator=g, device="cuda")

    plain = clusters(n)
    if kind == "all_equal":
        x = plain[:, :1].expand_as(plain)
    elif kind == "repeated":
        x = clusters(n // 4).repeat(1, 4, 1)
    elif kind == "zero_rows":
        x = plain.clone()
        x[:, n // 4:] = 0.0
    else:
        x = plain[:, :1] + 0.01 * torch.randn(n_inst, n, d, generator=g, device="cuda")
    t_plain, t = (_time(v.to(torch.bfloat16).contiguous(), nb) for v in (plain, x))
    print(f"{kind}: {1e3 * t:.0f} us, plain {1e3 * t_plain:.0f} us")
    assert t < times * t_plain
