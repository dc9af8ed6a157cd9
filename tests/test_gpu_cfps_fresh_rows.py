"""A Continual FPS checkpoint copies whole buffers, rows past a head's size included: in a new context these
are zero, not whatever the device memory held before."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_rows_past_the_size_of_a_new_buffer_are_zero():
    from paper_2609_04971_gb300 import bkv
    layers, batch, q_heads, d, nb, W = 4, 4, 8, 128, 8, 8
    held = [torch.full((1 << 22,), 7.0, device="cuda") for _ in range(64)]  # 1 GiB of 7.0 in what create will take
    torch.cuda.synchronize()
    del held
    torch.cuda.empty_cache()
    for _ in range(3):
        bk = bkv.BeaconKV(n_layers=layers, batch=batch, n_q_heads=q_heads, n_kv_heads=2, head_dim=d, n_beacons=nb,
                          window=W, capacity=64, continual_fps=True)
        try:
            bk.init_beacons(torch.randn(layers, batch, q_heads, 32, d, device="cuda").to(torch.bfloat16))
            buf, sizes = bk.cfps_state()
            bk.sync()
        finally:
            bk.close()
        assert bool((sizes == nb).all())
        assert bool((buf[..., nb:, :].view(torch.int16) == 0).all())
        assert bool((buf[..., :nb, :].float().norm(dim=-1) > 0).all())
