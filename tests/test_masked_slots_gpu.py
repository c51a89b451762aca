"""Slots masked with a bias of -inf, or with the lowest float32 (which overflows in the scaling by
log2(e) / tau): forward and backward equal those of the problem without the slots, on every path.
Bars as everywhere: fp32 normwise max relative 1e-4, bf16 relative L2 1e-2.
"""
import numpy as np
import pytest
import torch

from oracle import flashslice_oracle as orc
from paper_2609_32525_gb300.workloads import make_case

from _parity import error, host, tol, upload

pytestmark = pytest.mark.gpu

# (B, N, H, d, G, dtype), forward path, backward path
CASES = [((1, 300, 2, 16, 100, "f32"), 0, 0), ((2, 257, 2, 64, 64, "bf16"), 0, 0), ((1, 500, 2, 32, 33, "f32"), 0, 0),
         ((2, 1000, 2, 32, 100, "bf16"), 1, 1), ((1, 700, 1, 32, 1100, "bf16"), 0, 1),
         ((1, 84000, 2, 32, 100, "f32"), 1, 0)]


@pytest.mark.parametrize("mask", [-np.inf, np.finfo(np.float32).min], ids=["inf", "lowest"])
@pytest.mark.parametrize("shape,fwd,bwd", CASES, ids=lambda s: "B{}N{}H{}d{}G{}{}".format(*s) if isinstance(s, tuple) else "")
def test_masked(lib, shape, fwd, bwd, mask):
    B, N, H, d, G, dt = shape
    wl = make_case(B, N, H, d, G, dtype=dt, seed=91 + N + G, backward=True)
    keep = np.sort(np.random.default_rng(5).permutation(G)[:G // 3])
    bias = np.full_like(wl.bias, mask)
    bias[:, keep] = wl.bias[:, keep]
    dev = upload(wl)
    dev["bias"] = torch.from_numpy(bias).cuda()
    c = lib.Coupling(B, N, H, d, G, dev["x_mid"].dtype, wl.eps, backward=True)
    assert lib.path_for_shape(c.shape) == fwd and lib.backward_path_for_shape(c.shape) == bwd
    p = (wl.x_mid, wl.fx, wl.W_slice[:, :, keep], wl.bias[:, keep], wl.tau, wl.M[:, keep][:, :, keep])
    rf, rb = orc.forward(*p, eps=wl.eps), orc.backward(*p, wl.dout, eps=wl.eps)
    a = [dev[k] for k in ("x_mid", "fx", "W_slice", "bias", "tau", "M")]
    out = c.forward(*a)
    assert error(host(out), rf["out"], dt) <= tol(dt)
    for fused in (True, False):
        g = {k: host(v) for k, v in c.backward(*a, dev["dout"], fused=fused).items()}
        assert c.device_status() == lib.FS_OK
        masked = np.setdiff1d(np.arange(G), keep)
        assert not g["dW"][:, :, masked].any() and not g["dbias"][:, masked].any()
        g["dW"], g["dbias"], g["dM"] = g["dW"][:, :, keep], g["dbias"][:, keep], g["dM"][:, keep][:, :, keep]
        for k in g:
            e = error(g[k], rb[k], dt)
            assert e <= tol(dt), f"{'fused' if fused else 'separate'} {k}: {e:.3e}"
