"""fs_*_launch_count against the kernels that the calls launch, counted as the nodes of a captured
graph (every node a kernel: the calls issue no memsets or copies)."""
import ctypes

import pytest
import torch

from paper_2609_32525_gb300.workloads import make_case

from _parity import upload

pytestmark = pytest.mark.gpu

# (B, N, H, d, G, dtype): tensor cores with one and several slot ranges, G past the forward's
# 1024, a single point, fp32 split products, SIMT.
SHAPES = [(1, 700, 2, 32, 100, "bf16"), (1, 700, 2, 32, 600, "bf16"), (1, 700, 2, 32, 1024, "bf16"),
          (1, 700, 1, 32, 1500, "bf16"), (1, 1, 2, 32, 64, "bf16"), (1, 131072, 2, 32, 64, "f32"),
          (1, 32768, 1, 32, 600, "f32"), (1, 500, 2, 32, 64, "f32"), (1, 500, 2, 64, 64, "bf16")]


def _nodes(fn):
    rt = ctypes.CDLL("libcudart.so.13")
    stream = torch.cuda.Stream()
    h, graph, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    with torch.cuda.stream(stream):
        assert rt.cudaStreamBeginCapture(h, 2) == 0
        try:
            fn()
        finally:
            assert rt.cudaStreamEndCapture(h, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return n.value


@pytest.mark.parametrize("dot", [0, 1], ids=["bf16", "bf16x2"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "B{}N{}H{}d{}G{}{}".format(*s))
def test_counts(lib, shape, dot):
    B, N, H, d, G, dt = shape
    dev = upload(make_case(B, N, H, d, G, dtype=dt, seed=1, backward=True))
    c = lib.Coupling(B, N, H, d, G, dev["x_mid"].dtype, backward=True, dot=dot)
    a = [dev[k] for k in ("x_mid", "fx", "W_slice", "bias", "tau", "M")]
    c.forward(*a)
    c.backward(*a, dev["dout"])
    c.backward(*a, dev["dout"], fused=False)
    torch.cuda.synchronize()
    assert _nodes(lambda: c.forward(*a)) == lib.forward_launch_count(c.shape)
    lse = c.lse
    for given in (True, False):
        c.lse = lse if given else None
        assert _nodes(lambda: c.backward(*a, dev["dout"])) == lib.coupling_bwd_launch_count(c.shape, given)
        assert _nodes(lambda: c.backward(*a, dev["dout"], fused=False)) == lib.backward_launch_count(c.shape, given)
