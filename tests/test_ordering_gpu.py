"""Kernels that may start under the ones before them (programmatic dependence): calls right behind
one another on one coupling, behind and before other kernels on their inputs, on two streams at
once, and from a captured graph give the bits that calls with a synchronisation between them give.
"""
import pytest
import torch

from paper_2609_32525_gb300.workloads import make_case

from _parity import upload

pytestmark = pytest.mark.gpu

SHAPES = [(1, 20011, 4, 32, 100, "bf16"), (2, 3000, 2, 32, 600, "bf16"), (1, 4096, 4, 32, 32, "f32"),
          (1, 65536, 4, 32, 64, "f32"), (1, 2000, 2, 64, 64, "bf16")]
ids = [("B{}N{}H{}d{}G{}{}").format(*s) for s in SHAPES]
KEYS = ("x_mid", "fx", "W_slice", "bias", "tau", "M", "dout")


def _coupling(lib, shape):
    B, N, H, d, G, dt = shape
    return lib.Coupling(B, N, H, d, G, torch.bfloat16 if dt == "bf16" else torch.float32, backward=True)


def _inputs(shape, seed):
    return upload(make_case(*shape[:5], dtype=shape[5], seed=seed, backward=True))


def _step(c, v):
    """One training step's outputs, copied on the stream that it ran on."""
    a = [v[k] for k in KEYS[:-1]]
    out = {"out": c.forward(*a), **c.backward(*a, v["dout"])}
    return {k: t.clone() for k, t in out.items()}


def _expected(lib, shape, seeds):
    r = []
    for s in seeds:
        c = _coupling(lib, shape)
        v = _inputs(shape, s)
        torch.cuda.synchronize()
        r.append(_step(c, v))
        torch.cuda.synchronize()
        assert c.device_status() == lib.FS_OK
    return r


def _same(got, want):
    for g, w in zip(got, want):
        for k in w:
            assert torch.equal(g[k], w[k]), k


@pytest.mark.parametrize("shape", SHAPES, ids=ids)
def test_back_to_back(lib, shape):
    want = _expected(lib, shape, (1, 2, 3))
    c, vs = _coupling(lib, shape), [_inputs(shape, s) for s in (1, 2, 3)]
    torch.cuda.synchronize()
    got = [_step(c, v) for _ in range(3) for v in vs]
    torch.cuda.synchronize()
    _same(got, want * 3)


@pytest.mark.parametrize("shape", SHAPES, ids=ids)
def test_between_other_kernels(lib, shape):
    """Inputs written by the kernel before the call and overwritten by the one after it."""
    want = _expected(lib, shape, (1, 2))
    c, vs = _coupling(lib, shape), [_inputs(shape, s) for s in (1, 2)]
    buf = {k: torch.zeros_like(vs[0][k]) for k in KEYS}
    torch.cuda.synchronize()
    got = []
    for v in vs * 3:
        for k in reversed(KEYS):
            buf[k].copy_(v[k])
        got.append(_step(c, buf))
        for k in KEYS:
            buf[k].fill_(float("nan"))
    torch.cuda.synchronize()
    _same(got, want * 3)


def test_two_streams(lib):
    pairs = [(SHAPES[0], SHAPES[1]), (SHAPES[0], SHAPES[2])]
    for pair in pairs:
        want = [_expected(lib, s, (1, 2)) for s in pair]
        cs, vs = [_coupling(lib, s) for s in pair], [[_inputs(s, i) for i in (1, 2)] for s in pair]
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        torch.cuda.synchronize()
        got = [[], []]
        for i in range(6):
            for k in range(2):
                with torch.cuda.stream(streams[k]):
                    got[k].append(_step(cs[k], vs[k][i % 2]))
        torch.cuda.synchronize()
        for k in range(2):
            assert cs[k].device_status() == lib.FS_OK
            _same(got[k], want[k] * 3)


@pytest.mark.parametrize("shape", SHAPES, ids=ids)
def test_captured_graph(lib, shape):
    want = _expected(lib, shape, (1, 2))
    c, vs = _coupling(lib, shape), [_inputs(shape, s) for s in (1, 2)]
    buf = {k: vs[0][k].clone() for k in KEYS}
    a = [buf[k] for k in KEYS[:-1]]
    _step(c, buf)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        c.forward(*a)
        c.backward(*a, buf["dout"])
    got = []
    for v in vs * 3:
        for k in KEYS:
            buf[k].copy_(v[k])
        graph.replay()
        got.append({"out": c.out.clone(), **{k: getattr(c, k).clone() for k in want[0] if k != "out"}})
    torch.cuda.synchronize()
    _same(got, want * 3)
