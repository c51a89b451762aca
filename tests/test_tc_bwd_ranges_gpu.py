"""The tensor-core backward over several slot ranges with two to nine point tiles per block of
threads: the rows pass of both parts added up over ranges (G = 1024), one rows pass for each part
(640, and two ranges of it: 1100), the point pass over two to five ranges, the slot pass's token
gradient past the forward's 1024 slots.  The fused call and the separate ones, against the same
sums in 64 bits at the bf16 bar (relative L2 1e-2).
"""
import pytest
import torch

from paper_2609_32525_gb300.workloads import make_case

from _parity import TOL_BF16_RELL2, upload

pytestmark = pytest.mark.gpu


def _gradients(x, fx, W, bias, tau, M, dout, eps):
    """One batch, one head, in 64 bits: x, fx, dout [N, d], W [d, G]."""
    x, fx, W, bias, M, dout = (v.double() for v in (x, fx, W, bias, M, dout))
    t, G, d = tau.double(), W.shape[1], W.shape[0]
    parts = x.split(16384)
    log_w = [torch.log_softmax((p @ W + bias) / t, 1) for p in parts]
    U, S, dzm = (torch.zeros(*s, dtype=torch.float64, device="cuda") for s in ((G, d), (G,), (G, d)))
    for lw, f, o in zip(log_w, fx.split(16384), dout.split(16384)):
        w = lw.exp()
        U, S, dzm = U + w.T @ f, S + w.sum(0), dzm + w.T @ o
    z = U / (S + eps)[:, None]
    zm, dz = M @ z, M.T @ dzm
    dU, dS = dz / (S + eps)[:, None], -(dz * z).sum(1) / (S + eps)
    dx, dfx, dW, db, dt = [], [], 0.0, 0.0, 0.0
    for lw, p, f, o in zip(log_w, parts, fx.split(16384), dout.split(16384)):
        w = lw.exp()
        dw = o @ zm.T + f @ dU.T + dS
        da = w * (dw - (w * dw).sum(1, keepdim=True))
        dx.append(da @ W.T / t)
        dfx.append(w @ dU)
        dW, db, dt = dW + p.T @ da / t, db + da.sum(0) / t, dt - (da * lw).sum() / t
    return {"dx_mid": torch.cat(dx), "dfx": torch.cat(dfx), "dW": dW, "dbias": db, "dtau": dt, "dM": dzm @ z.T}


@pytest.mark.parametrize("G", [640, 1024, 1100])
@pytest.mark.parametrize("tiles", [2, 3, 5, 9])
def test_tiles_per_block_and_ranges(lib, tiles, G):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N = 128 * sms * tiles - 37  # one head: one split of `tiles` tiles per SM, the last tile ragged
    wl = make_case(1, N, 1, 32, G, dtype="bf16", seed=53 * tiles + G, backward=True)
    dev = upload(wl)
    c = lib.Coupling(1, N, 1, 32, G, torch.bfloat16, wl.eps, backward=True)
    assert lib.backward_path_for_shape(c.shape) == 1
    a = [dev[k] for k in ("x_mid", "fx", "W_slice", "bias", "tau", "M")]
    ref = _gradients(a[0][0, :, 0], a[1][0, :, 0], *(v[0] for v in a[2:]), dev["dout"][0, :, 0], wl.eps)
    c.forward(*a)
    for fused in (True, False):
        got = c.backward(*a, dev["dout"], fused=fused)
        torch.cuda.synchronize()
        assert c.device_status() == lib.FS_OK
        for k, r in ref.items():
            e = float((got[k].double().reshape(r.shape) - r).norm() / r.norm())
            assert e <= TOL_BF16_RELL2, f"{'fused' if fused else 'separate'} {k}: {e:.3e}"
