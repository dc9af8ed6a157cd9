"""bkv_sync clears the device error word and the batched update's spill words on the context's own stream:
an update enqueued right after a reported error, on a stream that the legacy default stream does not wait
for, must find them cleared before it starts and not be cleared under it.  The update's values spill more
elements per instance than the in-kernel list holds; its sums must be the exact ones."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_inst,d,nb", [(152, 128, 32), (400, 64, 8)])
def test_update_right_after_a_reported_error(n_inst, d, nb):
    from paper_2609_04971_gb300 import bkv
    G, n_new, cap, rounds = 4, 64, 64, 4
    g = torch.Generator(device="cuda").manual_seed(n_inst)

    def wide(n):  # magnitudes over 24 octaves
        x = torch.randn(n_inst, 1, G, n, d, generator=g, device="cuda")
        return (x * 2.0 ** torch.randint(-18, 6, x.shape, generator=g, device="cuda").float()).to(torch.bfloat16)

    q_init, queries = wide(nb), [wide(n_new) for _ in range(rounds)]
    K = torch.zeros(n_inst, 1, 1, cap, d, dtype=torch.bfloat16, device="cuda")
    V = torch.zeros_like(K)
    q_recent = torch.zeros(n_inst, 1, G, 4, d, dtype=torch.bfloat16, device="cuda")
    kept = torch.empty(n_inst, 1, 1, cap, dtype=torch.int32, device="cuda")
    L = torch.full((n_inst, 1, 1), cap, dtype=torch.int32, device="cuda")
    L[n_inst // 2] = cap + 1
    assign = [torch.empty(n_inst, 1, G, n_new, dtype=torch.int32, device="cuda") for _ in range(rounds)]
    torch.cuda.synchronize()
    side = torch.cuda.Stream()  # non-blocking: not ordered with the legacy default stream
    with torch.cuda.stream(side):
        bk = bkv.BeaconKV(n_layers=n_inst, batch=1, n_q_heads=G, n_kv_heads=1, head_dim=d, n_beacons=nb, window=4,
                          capacity=cap, stream=side)
        try:
            bk.init_beacons(q_init)
            states = [bk.state()]
            for r in range(rounds):
                bk.compress_ragged(K, V, L=L, budget=cap, t_pos=[cap], q_recent=q_recent, recent_pos=[[0, 1, 2, 3]],
                                   kept_out=kept)
                with pytest.raises(bkv.BkvError) as ei:
                    bk.sync()
                assert ei.value.code == bkv.BKV_EINVAL
                bk.update(queries[r], assign[r])
                states.append(bk.state())
            bk.sync()
        finally:
            bk.close()
    for r in range(rounds):
        x = queries[r].view(n_inst, G * n_new, d).double().cpu().numpy()
        x = np.where(np.abs(x) < 2.0 ** -31, np.rint(x * 2.0 ** 38) * 2.0 ** -38, x)
        a = assign[r].view(n_inst, -1).cpu().numpy()
        want = states[r][1].cpu().numpy().reshape(n_inst, nb, d).copy()
        count = states[r][2].cpu().numpy().reshape(n_inst, nb).copy()
        for b in range(nb):
            want[:, b] += np.where((a == b)[:, :, None], x, 0.0).sum(1)  # exact: at most 53 bits in all
            count[:, b] += (a == b).sum(1)
        np.testing.assert_array_equal(states[r + 1][1].cpu().numpy().reshape(n_inst, nb, d), want)
        np.testing.assert_array_equal(states[r + 1][2].cpu().numpy().reshape(n_inst, nb), count)
