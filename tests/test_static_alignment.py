"""bkv_compress_static takes its centroids from the caller, and its query build reads them 16 bytes at a
time: an address that is not a multiple of 16 is refused on the host, before any CUDA call."""
import ctypes

import pytest

from paper_2609_04971_gb300 import bkv
from paper_2609_04971_gb300.workloads import TINY as wl


@pytest.mark.parametrize("centroids,counts", [(0x10004, 0x20000), (0x10008, 0x20000), (0x10000, 0x20004)])
def test_static_compress_refuses_misaligned_state(centroids, counts):
    fn = bkv.load_library().bkv_compress_static
    cfg = bkv.BkvConfig(wl.n_layers, wl.batch, wl.n_q_heads, wl.n_kv_heads, wl.head_dim, wl.n_beacons, wl.window, 0,
                        wl.capacity, wl.rope_theta, 0)
    pos = (ctypes.c_int64 * wl.window)(*range(wl.L - wl.window, wl.L))
    msg = ctypes.create_string_buffer(200)
    rc = fn(ctypes.byref(cfg), centroids, counts, 0x30000, 0x40000, wl.L, wl.budget, wl.L - 1, 0x50000,
            ctypes.cast(pos, ctypes.c_void_p), 0x60000, None, None, None, msg, ctypes.sizeof(msg))
    assert rc == bkv.BKV_EINVAL and "aligned" in msg.value.decode()
