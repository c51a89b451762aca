"""The tensor-core forward with one to nine point tiles per block of threads and one to three
slot blocks per tile: every position of a tile in the rings of buffers, and every warpgroup as
the one that drains the last tile.  Against the fp64 oracle at the bf16 bar (relative L2 1e-2).
"""
import pytest
import torch

from oracle import flashslice_oracle as orc
from paper_2609_32525_gb300.workloads import make_case

from _parity import error, host, tol, upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G", [40, 128, 200, 384])
@pytest.mark.parametrize("tiles", [1, 2, 3, 4, 5, 7, 9])
def test_tiles_per_block(lib, tiles, G):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N = 128 * sms * tiles - 37  # one head: one split of `tiles` tiles per SM, the last tile ragged
    wl = make_case(1, N, 1, 32, G, dtype="bf16", seed=31 * tiles + G, backward=False)
    dev = upload(wl)
    c = lib.Coupling(1, N, 1, 32, G, torch.bfloat16, wl.eps)
    assert lib.path_for_shape(c.shape) == 1
    out = c.forward(dev["x_mid"], dev["fx"], dev["W_slice"], dev["bias"], dev["tau"], dev["M"])
    torch.cuda.synchronize()
    assert c.device_status() == lib.FS_OK
    ref = orc.forward(wl.x_mid, wl.fx, wl.W_slice, wl.bias, wl.tau, wl.M, eps=wl.eps)
    assert error(host(out), ref["out"], "bf16") <= tol("bf16")
