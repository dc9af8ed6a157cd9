"""The batched beacon update (many queries per instance) against the oracle, at
the edges of its tiles, beacon padding and element ranges.

The kernel forms each tile's sums as matrix products of elements split by
magnitude around a per-instance exponent; the value sets below put elements on
both sides of every limit (all scales, outlier columns, columns far below the
rest, zero queries), and the sums must still be the exact ones: the reference
is the fp64 sum of the assigned rows, exact for these inputs.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from tests import parity as P


def _values(kind, shape, g):
    x = torch.randn(shape, generator=g, device="cuda")
    if kind == "scaled_down":
        x *= 2.0 ** -9
    elif kind == "scaled_up":
        x *= 2.0 ** 7
    elif kind == "outlier_columns":  # a few columns 300 times the rest
        x[..., 5::29] *= 300.0
    elif kind == "wide":  # magnitudes over 24 octaves, some exact zeros
        x *= 2.0 ** torch.randint(-18, 6, shape, generator=g, device="cuda").float()
        x[torch.rand(shape, generator=g, device="cuda") < 0.05] = 0.0
    elif kind == "zero_queries":
        x[torch.rand(shape[:-1], generator=g, device="cuda") < 0.2] = 0.0
    elif kind == "all_equal":  # sums of 128 equal rows, the largest the operands can be given
        x = (3.0 + 4.984375 * torch.rand(shape[:1] + (1,) * (len(shape) - 2) + shape[-1:], generator=g,
                                         device="cuda")).expand(shape).contiguous()
    elif kind == "first_small":  # what a CTA has seen first says nothing about what follows
        x[: shape[0] // 2] *= 2.0 ** -8
        x[shape[0] // 2:] *= 2.0 ** 5
    return x.to(torch.bfloat16)


@pytest.mark.parametrize("n_inst,G,n_new,d,nb,kind", [
    (3, 1, 33, 128, 1, "plain"), (2, 4, 16, 64, 8, "plain"), (5, 1, 127, 128, 9, "plain"), (4, 2, 64, 64, 16, "plain"),
    (3, 3, 43, 128, 16, "zero_queries"), (2, 8, 129, 128, 17, "plain"), (400, 4, 10, 128, 8, "plain"),
    (330, 5, 37, 64, 5, "first_small"), (700, 1, 40, 128, 16, "first_small"), (160, 4, 128, 128, 32, "plain"),
    (4, 4, 100, 128, 8, "scaled_down"), (4, 4, 100, 64, 8, "scaled_up"), (6, 4, 70, 128, 16, "outlier_columns"),
    (310, 2, 150, 128, 8, "outlier_columns"), (6, 4, 64, 128, 8, "wide"), (6, 4, 65, 64, 32, "wide"),
    (4, 4, 64, 128, 16, "all_equal"), (3, 8, 1100, 64, 8, "plain"), (2, 4, 2200, 128, 4, "plain"),
    (4, 4, 64, 128, 8, "large_state"), (4, 4, 64, 64, 20, "large_state"),
])
def test_batched_update(n_inst, G, n_new, d, nb, kind, olib):
    from paper_2609_04971_gb300 import bkv
    g = torch.Generator(device="cuda").manual_seed(n_inst * 1000 + n_new)
    nq = G * n_new
    q_init = _values(kind, (n_inst, G, max(nb, 4), d), g)
    bk = bkv.BeaconKV(n_layers=n_inst, batch=1, n_q_heads=G, n_kv_heads=1, head_dim=d, n_beacons=nb, window=4,
                      capacity=64)
    try:
        bk.init_beacons(q_init.view(n_inst, 1, G, -1, d))
        if kind == "large_state":  # sums past 2^13 (rounded to their double's grid) and some off the 2^-40 grid
            cent, sums, counts = bk.state()
            counts += torch.randint(1, 1 << 20, counts.shape, generator=g, device="cuda")
            sums = sums * counts.unsqueeze(-1)
            sums[:, ::3, ::5] *= 1.0 + 2.0 ** -45
            bk.set_state((sums / counts.unsqueeze(-1)).float(), sums, counts)
        states, queries, assigns = [[t.cpu().numpy() for t in bk.state()]], [], []
        for _ in range(2):
            q = _values(kind, (n_inst, G, n_new, d), g)
            assign = torch.full((n_inst, 1, G, n_new), -7, dtype=torch.int32, device="cuda")
            bk.update(q.view(n_inst, 1, G, n_new, d), assign)
            states.append([t.cpu().numpy() for t in bk.state()])
            queries.append(q.view(n_inst, nq, d).cpu())
            assigns.append(assign.view(n_inst, nq).cpu().numpy())
        bk.sync()
    finally:
        bk.close()
    insts = range(n_inst) if n_inst <= 8 else sorted({0, 1, 151, 152, 153, n_inst // 2, n_inst - 2, n_inst - 1})
    for c in range(2):
        x64 = queries[c].double().numpy()
        tiny = np.abs(x64) < 2.0 ** -31  # documented: rounded to multiples of 2^-38
        x64 = np.where(tiny, np.rint(x64 * 2.0 ** 38) * 2.0 ** -38, x64)
        # the oracle adds elements as they are: it gets them as the sums take them (still bf16 values)
        bits = torch.from_numpy(x64).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
        for e in insts:
            pre, post = ({"cent": s[0][e], "sums": s[1][e], "counts": s[2][e]} for s in (states[c], states[c + 1]))
            want = pre["sums"].copy()
            for b in range(nb):
                want[b] += x64[e][assigns[c][e] == b].sum(0)  # exact: at most 53 bits between the largest and the finest
            np.testing.assert_array_equal(post["sums"], want, err_msg=f"call {c} instance {e}: sums")
            P.check_update(bits[e], pre, assigns[c][e], post, olib, tag=f"call {c} instance {e}")
