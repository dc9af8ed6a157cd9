"""The batched beacon update on queries of many scales, with several instances per CTA, so that what a CTA
has seen of its earlier instances decides the exponent of the operands that the later ones are summed with,
and which of their elements are added one by one.  Sums must be the exact ones whatever the scales,
assignments the fp64 argmax; and such queries must not take many times the time of plain ones."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SMS = 152


def _queries(kind, n_inst, G, n, d, g):
    r = dict(generator=g, device="cuda")
    x = torch.randn(n_inst, G, n, d, **r)
    if kind == "wide":  # 24 octaves, element by element
        x *= 2.0 ** torch.randint(-18, 6, x.shape, **r).float()
    elif kind == "lognormal":
        x *= torch.exp(1.5 * torch.randn(x.shape, **r))
    elif kind == "query_scales":
        x *= torch.exp(1.5 * torch.randn(n_inst, G, n, 1, **r))
    elif kind == "columns":  # a few columns 300 times the rest
        x[..., 5::29] *= 300.0
    elif kind == "outlier":  # one query per CTA, in its first instance
        x[:SMS, 0, 0] *= 1000.0
    elif kind == "instances":  # plain and wide instances in turn, six at a time
        turn = (torch.arange(n_inst, device="cuda") // (6 * SMS)) % 2 == 1
        scale = 2.0 ** torch.randint(-22, 3, x.shape, **r).float()
        x = torch.where(turn.view(-1, 1, 1, 1), x * scale, x)
    elif kind == "tiny":  # below what the fixed point holds exactly, and zeros
        x *= 2.0 ** torch.randint(-40, -4, x.shape, **r).float()
        x[torch.rand(x.shape[:-1], **r) < 0.1] = 0.0
    return x.to(torch.bfloat16)


def _context(n_inst, G, d, nb, g):
    from paper_2609_04971_gb300 import bkv
    bk = bkv.BeaconKV(n_layers=n_inst, batch=1, n_q_heads=G, n_kv_heads=1, head_dim=d, n_beacons=nb, window=4,
                      capacity=64)
    cent = torch.randn(n_inst, nb, d, generator=g, device="cuda")
    sums = torch.round(cent.double() * 50 * 65536) / 65536
    bk.set_state((sums / 50).float(), sums, torch.full((n_inst, nb), 50, dtype=torch.int64, device="cuda"))
    return bk


@pytest.mark.parametrize("n_inst,G,n_new,d,nb,kind", [
    (6 * SMS + 3, 4, 64, 128, 8, "wide"), (6 * SMS, 4, 65, 64, 8, "wide"), (9 * SMS, 1, 40, 128, 16, "wide"),
    (16 * SMS, 3, 11, 64, 4, "wide"), (5 * SMS, 4, 33, 128, 32, "wide"), (5 * SMS + 1, 5, 30, 64, 20, "wide"),
    (8 * SMS, 4, 64, 128, 8, "lognormal"), (8 * SMS, 4, 64, 128, 8, "query_scales"), (8 * SMS, 4, 40, 64, 8, "columns"),
    (8 * SMS, 4, 64, 128, 8, "outlier"), (20 * SMS, 2, 48, 128, 8, "instances"), (8 * SMS, 4, 32, 128, 8, "tiny"),
    (3 * SMS + 4, 4, 2250, 64, 4, "wide"), (3 * SMS + 1, 4, 2100, 128, 4, "columns"),
])
def test_sums_are_exact_for_queries_of_any_scale(n_inst, G, n_new, d, nb, kind):
    g = torch.Generator(device="cuda").manual_seed(n_inst + n_new)
    bk = _context(n_inst, G, d, nb, g)
    try:
        for call in range(2):
            q = _queries(kind, n_inst, G, n_new, d, g)
            assign = torch.full((n_inst, 1, G, n_new), -7, dtype=torch.int32, device="cuda")
            cent, sums, counts = bk.state()
            bk.update(q.view(n_inst, 1, G, n_new, d), assign)
            _, got, got_counts = bk.state()
            a = assign.view(n_inst, -1).long()
            for i0 in range(0, n_inst, 128):
                e = slice(i0, min(i0 + 128, n_inst))
                x = q[e].reshape(-1, G * n_new, d).double()
                zero = (x == 0).all(-1)
                assert torch.equal(a[e] < 0, zero) and int(a[e].max()) < nb
                cos = torch.bmm(x, torch.nn.functional.normalize(cent[e].double(), dim=-1).transpose(1, 2))
                picked = cos.gather(2, a[e].clamp_min(0).unsqueeze(-1)).squeeze(-1)
                slack = 1e-12 * x.norm(dim=-1)
                assert bool((picked >= cos.amax(-1) - slack)[~zero].all())
                # documented: elements below 2^-31 are rounded to multiples of 2^-38
                x = torch.where(x.abs() < 2.0 ** -31, torch.round(x * 2.0 ** 38) * 2.0 ** -38, x)
                hot = torch.nn.functional.one_hot(a[e].clamp_min(0), nb).double() * (~zero).unsqueeze(-1)
                # the call's sums take at most 53 bits and are exact in any order; one rounding into the state
                want = sums[e].view(-1, nb, d) + torch.bmm(hot.transpose(1, 2), x)
                assert torch.equal(got[e].view(-1, nb, d), want), f"call {call}, instances from {i0}"
                assert torch.equal(got_counts[e].view(-1, nb), counts[e].view(-1, nb) + hot.sum(1).long())
        bk.sync()
    finally:
        bk.close()


def _time(bk, q):
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for r in range(8):
        e0.record()
        bk.update(q)
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1)) if r >= 2 else best
    return best


@pytest.mark.parametrize("kind,times", [("outlier", 2.0), ("columns", 3.0), ("lognormal", 4.0), ("query_scales", 4.0),
                                        ("wide", 12.0)])
def test_scales_cost_a_few_times_the_time(kind, times):
    """Elements outside the operands' range are added one by one.  With a row of them at a time taken by a
    whole warp, and the exponent left where one outlier had put it, these took 4 to 19 times as long."""
    n_inst, G, n_new, d, nb = 30 * SMS, 4, 128, 128, 8
    g = torch.Generator(device="cuda").manual_seed(5)
    bk = _context(n_inst, G, d, nb, g)
    try:
        plain, other = (_queries(k, n_inst, G, n_new, d, g).view(n_inst, 1, G, n_new, d) for k in ("plain", kind))
        t_plain, t_other = _time(bk, plain), _time(bk, other)
        bk.sync()
    finally:
        bk.close()
    print(f"{kind}: {1e3 * t_other:.0f} us, plain {1e3 * t_plain:.0f} us")
    assert t_other < times * t_plain
