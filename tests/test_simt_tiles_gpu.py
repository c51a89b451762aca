"""The tiled fp32 passes (128 points x 32 or 64 slots per tile) at the edges of their tiles,
against the fp64 oracle: one point, one below, at and above a tile of points; slot counts
around the narrow tile (32), the wide tile (64) and two tiles; every head width and point
type.  fs_deslice_bwd + fs_slice_bwd (the separate modes) and fs_coupling_bwd (both parts).

Bars as for the SIMT path everywhere: fp32 normwise max relative 1e-4, bf16 relative L2 1e-2.
"""
import numpy as np
import pytest
import torch

from oracle import flashslice_oracle as orc
from paper_2609_32525_gb300.workloads import make_case

from _parity import error, host, tol, upload

pytestmark = pytest.mark.gpu

SHAPES = [(1, 2, 2, 32, 1, "f32"), (1, 127, 2, 16, 31, "f32"), (2, 128, 1, 32, 32, "f32"), (1, 129, 3, 32, 33, "f32"),
          (1, 300, 2, 64, 32, "f32"), (2, 257, 2, 64, 64, "bf16"), (1, 1000, 2, 16, 65, "bf16"),
          (1, 130, 2, 16, 130, "f32"), (3, 511, 2, 64, 129, "f32"), (1, 4097, 1, 32, 63, "f32")]


@pytest.mark.parametrize("fused", [True, False], ids=["fused", "separate"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "B{}N{}H{}d{}G{}{}".format(*s))
def test_tile_edges(lib, shape, fused):
    B, N, H, d, G, dt = shape
    wl = make_case(B, N, H, d, G, dtype=dt, seed=77 + N + G, backward=True)
    dev = upload(wl)
    c = lib.Coupling(B, N, H, d, G, dev["x_mid"].dtype, wl.eps, backward=True)
    assert lib.path_for_shape(c.shape) == 0 and lib.backward_path_for_shape(c.shape) == 0
    a = [dev[k] for k in ("x_mid", "fx", "W_slice", "bias", "tau", "M")]
    out = c.forward(*a)
    g = c.backward(*a, dev["dout"], fused=fused)
    torch.cuda.synchronize()
    assert c.device_status() == lib.FS_OK
    p = (wl.x_mid, wl.fx, wl.W_slice, wl.bias, wl.tau, wl.M)
    rf, rb = orc.forward(*p, eps=wl.eps), orc.backward(*p, wl.dout, eps=wl.eps)
    for name, got, ref in [("out", out, rf["out"])] + [(k, g[k], rb[k]) for k in g]:
        if G == 1 and name in ("dx_mid", "dW", "dbias", "dtau"):
            # one slot: every weight is 1 and these gradients are exactly 0
            assert np.abs(host(got)).max() <= 1e-4 * np.abs(host(g["dfx"])).max()
            continue
        e = error(host(got), ref, dt)
        assert e <= tol(dt), f"{name}: {e:.3e}"


def test_masked_slots(lib):
    """Slots masked with a bias of -inf (whole runs of a thread's slots): the forward equals
    the problem without them."""
    wl = make_case(1, 300, 2, 16, 100, dtype="f32", seed=5, backward=False)
    keep = np.r_[3:5, 70:81]
    bias = np.full_like(wl.bias, -np.inf)
    bias[:, keep] = wl.bias[:, keep]
    dev = upload(wl)
    dev["bias"] = torch.from_numpy(bias).cuda()
    M = torch.eye(100, device="cuda").expand(2, 100, 100).contiguous()
    c = lib.Coupling(1, 300, 2, 16, 100, torch.float32, wl.eps)
    out = c.forward(dev["x_mid"], dev["fx"], dev["W_slice"], dev["bias"], dev["tau"], M)
    torch.cuda.synchronize()
    eye = np.broadcast_to(np.eye(len(keep)), (2, len(keep), len(keep)))
    ref = orc.forward(wl.x_mid, wl.fx, wl.W_slice[:, :, keep], wl.bias[:, keep], wl.tau, eye, eps=wl.eps)
    assert error(host(out), ref["out"], "f32") <= tol("f32")
