"""The tensor-core backward with one to nine point tiles per block of threads and one to four
slot blocks: every position of a tile in the rings of buffers of the slot, point and row passes,
and every warpgroup as the one that drains the last tile.  Against the fp64 oracle at the bf16
bar (relative L2 1e-2).
"""
import pytest
import torch

from paper_2609_32525_gb300.workloads import make_case

from _parity import error, host, oracle_backward, tol, upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G", [40, 200, 512])
@pytest.mark.parametrize("tiles", [1, 2, 3, 5, 9])
def test_tiles_per_block(lib, tiles, G):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N = 128 * sms * tiles - 37  # one head: one split of `tiles` tiles per SM, the last tile ragged
    wl = make_case(1, N, 1, 32, G, dtype="bf16", seed=37 * tiles + G, backward=True)
    dev = upload(wl)
    c = lib.Coupling(1, N, 1, 32, G, torch.bfloat16, wl.eps, backward=True)
    assert lib.backward_path_for_shape(c.shape) == 1
    c.forward(dev["x_mid"], dev["fx"], dev["W_slice"], dev["bias"], dev["tau"], dev["M"])
    got = c.backward(dev["x_mid"], dev["fx"], dev["W_slice"], dev["bias"], dev["tau"], dev["M"], dev["dout"])
    torch.cuda.synchronize()
    assert c.device_status() == lib.FS_OK
    _check(wl, got)


def _check(wl, got):
    ref = oracle_backward(wl)
    for k in ("dx_mid", "dfx", "dW", "dbias", "dtau", "dM"):
        assert error(host(got[k]), ref[k], "bf16") <= tol("bf16"), k


@pytest.mark.parametrize("G", [256, 512, 513, 640, 1024, 1025])
def test_one_and_two_rows_passes(lib, G):
    """Slot ranges of up to 512 take one rows pass for both parts, ranges of 640 (G = 513 to
    640 and 1025) one for each; G = 1024 adds two ranges up."""
    wl = make_case(2, 700, 2, 32, G, dtype="bf16", seed=41 + G, backward=True)
    dev = upload(wl)
    c = lib.Coupling(2, 700, 2, 32, G, torch.bfloat16, wl.eps, backward=True)
    assert lib.backward_path_for_shape(c.shape) == 1
    c.forward(dev["x_mid"], dev["fx"], dev["W_slice"], dev["bias"], dev["tau"], dev["M"])
    got = c.backward(dev["x_mid"], dev["fx"], dev["W_slice"], dev["bias"], dev["tau"], dev["M"], dev["dout"])
    torch.cuda.synchronize()
    assert c.device_status() == lib.FS_OK
    _check(wl, got)
