"""Sums over long ranges on the tensor cores: their fp32 accumulation drops up to 2^-24 of the
running sum per step of 16 points, always towards zero, so a chain of n such steps drifts by
about n 2^-26 relative (2^-25 a step on average, of a sum that is half of its last value on
average; with split products each of a half's steps counts twice).  The passes restart or split
their chains so that this stays small; the separate backward calls and the fused one are held to
it here, against 64 bits.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _inputs(B, N, H, G, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)

    def randn(*s):
        return torch.randn(*s, device="cuda", generator=g)

    x, fx, dout = (randn(B, N, H, 32).bfloat16() for _ in range(3))
    W, bias, tau = randn(H, 32, G) / 32**0.5, randn(H, G) * 0.1, torch.full((H,), 0.5, device="cuda")
    M = torch.eye(G, device="cuda") + 0.1 * randn(H, G, G) / G**0.5
    return x, fx, W, bias, tau, M, dout


@pytest.mark.parametrize("B,N,G", [(1, 262144, 1024), (2, 131072, 512)])
def test_deslice_bwd_long_ranges(lib, B, N, G):
    """d z' of fs_deslice_bwd.  Ranges of 13,800 and 6,900 points: 1.3e-5 and 6.5e-6; the other
    errors (split weights and logits) are below 6e-6.  Ranges of 37,400 and 18,700 points, as
    fewer splits would give, drift by 3.5e-5 and 1.8e-5."""
    H, h = 8, 3
    x, fx, W, bias, tau, M, dout = _inputs(B, N, H, G, 7 + G)
    c = lib.Coupling(B, N, H, 32, G, torch.bfloat16, backward=True)
    assert lib.backward_path_for_shape(c.shape) == 1
    c.forward(x, fx, W, bias, tau, M)
    lib.fs_deslice_bwd(c.shape, x, W, bias, tau, c.tokens_mixed, c.lse, dout, c.d_tokens_mixed, c.dx_mid, c.dW, c.dbias,
                       c.dtau, False, c.ws_dbwd)
    torch.cuda.synchronize()
    assert c.device_status() == lib.FS_OK
    ref = torch.zeros(G, 32, dtype=torch.float64, device="cuda")
    for n in range(0, N, 65536):
        a = torch.addmm(bias[h].double(), x[0, n:n + 65536, h].double(), W[h].double()) / tau[h].double()
        ref += torch.softmax(a, 1).T @ dout[0, n:n + 65536, h].double()
    e = float((c.d_tokens_mixed[0, h].double() - ref).norm() / ref.norm())
    assert e <= (1.3e-5 if G == 1024 else 6.5e-6) + 6e-6, e


@pytest.mark.parametrize("G", [256, 512, 1024])
def test_fused_backward_keeps_the_balance_of_da(lib, G):
    """sum_g da_ng is 0 for every point, so sum_g dbias_hg is 0 but for the error of delta_n, which
    has one sign; with dout = out, delta_n is |out_n|^2 (the slice's part sums to 0).  The fused
    call forms delta from chains as long as the separate calls' (half of a range's slots each),
    so its imbalance is theirs; chains twice as long would double it."""
    B, N, H = 1, 65536, 4
    x, fx, W, bias, tau, M, _ = _inputs(B, N, H, G, 3 + G)
    fx = fx + 2
    c = lib.Coupling(B, N, H, 32, G, torch.bfloat16, backward=True)
    out = c.forward(x, fx, W, bias, tau, M).clone()
    scale = (out.double() ** 2).sum((0, 1, 3)) / tau.double()
    off = {}
    for fused in (True, False):
        g = c.backward(x, fx, W, bias, tau, M, out, fused=fused)
        off[fused] = float((g["dbias"].double().sum(1) / scale).abs().mean())
    torch.cuda.synchronize()
    assert c.device_status() == lib.FS_OK
    assert off[True] <= 1.4 * off[False], off
