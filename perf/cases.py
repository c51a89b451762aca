"""The work that users of this library have it do, as cases that can be timed and compared.

Every case is one call sequence of one coupling (slice -> token mix -> deslice) through
the public entry points of `paper_2609_32525_gb300.flashslice`:

  forward  Coupling.forward: inference of one layer
  train    Coupling.forward and Coupling.backward: one layer of a training step
  frozen   a FrozenSlice layer: fs_slice_fwd_lse with the first layer's statistics,
           fs_mix, fs_deslice_fwd
  untied   a layer whose deslice has its own projection and temperature: fs_slice_fwd,
           fs_mix, fs_deslice_fwd with lse = None

Inputs follow the repository's workloads (x_mid standard normal or a 16-component
mixture, W ~ N(0, 1/d), temperatures 0.5 or U[0.3, 1], M close to the identity or
N(0, 1/G)).  In a layer x_mid, fx and the gradient of the output all come from the same
point's hidden features, so fx and dout are a per-head linear map of x_mid plus noise.
"""
from __future__ import annotations

import math

import torch

from paper_2609_32525_gb300 import flashslice as fs

KINDS = ("forward", "train", "frozen", "untied")
MIXTURE = 16  # components of the point mixture


def listed():
    def case(name, kind, B, N, H, d, G, dtype, mixture=False, tau="half", mixer="identity"):
        return {"name": name, "kind": kind, "B": B, "N": N, "H": H, "d": d, "G": G, "dtype": dtype,
                "mixture": mixture, "tau": tau, "mixer": mixer}

    return [
        # A small 2-D problem (a few thousand points, 32 slices) in fp32: the smallest call,
        # launches and latency.
        case("tiny_f32", "forward", 1, 4096, 8, 32, 32, "f32"),
        # A surface mesh with the usual 64 slices, inference.
        case("surface_bf16", "forward", 1, 32768, 8, 32, 64, "bf16", tau="drawn", mixer="dense"),
        # Three meshes of an odd number of points and a slice count that is no power of two.
        case("ragged_bf16", "forward", 3, 20011, 8, 32, 100, "bf16", tau="drawn"),
        # A batch of volume samples at a moderate slice count.
        case("batched_bf16", "forward", 4, 262144, 8, 32, 256, "bf16", mixture=True),
        # A million-point mesh at the largest slice count: the headline inference workload.
        case("large_g_bf16", "forward", 1, 1048576, 8, 32, 1024, "bf16"),
        # fp32 inference of a volume sample.
        case("volume_f32", "forward", 1, 262144, 8, 32, 512, "f32"),
        # A later layer that reuses the first layer's weights and statistics.
        case("frozen_bf16", "frozen", 1, 262144, 8, 32, 1024, "bf16"),
        # A layer whose deslice has its own projection.
        case("untied_bf16", "untied", 2, 65536, 8, 32, 256, "bf16", mixture=True, tau="drawn"),
        # One layer of a training step on a surface mesh: the usual training call.
        case("train_surface_bf16", "train", 1, 32768, 8, 32, 64, "bf16", tau="drawn"),
        # One layer of the large training step.
        case("train_bf16", "train", 2, 524288, 8, 32, 512, "bf16", mixture=True),
        # The same in fp32 on a smaller sample.
        case("train_f32", "train", 2, 65536, 8, 32, 256, "f32", mixture=True),
        # A layer with wide heads (4 x 64 channels), training.
        case("train_wide_bf16", "train", 1, 16384, 4, 64, 64, "bf16", tau="drawn"),
    ]


def _pairs(c):
    """(point, head, slot) triples: what the time of a case grows with."""
    return c["B"] * c["N"] * c["H"] * c["G"]


# Upper limits of _pairs for drawn cases, by kind of arithmetic: the listed cases' costs.
_MOST = {"bf16": 1 << 33, "bf16 train": 1 << 32, "f32": 1 << 31, "f32 train": 1 << 28, "other": 1 << 27}


def draw(rng):
    """A case of the same ranges: 1,000 to a million points, 16 to 1024 slices, odd and
    ragged sizes among them."""
    kind = rng.choices(KINDS, (5, 4, 1, 1))[0]
    dtype = rng.choices(("bf16", "f32"), (3, 1))[0]
    d = rng.choices((32, 16, 64), (8, 1, 1))[0]
    H = {32: 8, 16: 8, 64: 4}[d]
    if d != 32:
        most = _MOST["other"]
    else:
        most = _MOST[dtype + (" train" if kind == "train" else "")]
    while True:
        B = rng.choice((1, 1, 2, 3, 4))
        N = int(round(math.exp(rng.uniform(math.log(1000), math.log(1 << 20)))))
        if rng.random() < 0.5:  # half of the samples are padded to whole blocks of 128 points
            N = max(1024, N // 128 * 128)
        G = int(round(math.exp(rng.uniform(math.log(16), math.log(1024)))))
        if rng.random() < 0.6:  # the usual slice counts
            G = 1 << max(4, min(10, round(math.log2(G))))
        c = {"kind": kind, "B": B, "N": N, "H": H, "d": d, "G": G, "dtype": dtype,
             "mixture": rng.random() < 0.4, "tau": rng.choice(("half", "drawn")),
             "mixer": rng.choice(("identity", "identity", "dense"))}
        if _pairs(c) <= most and c["B"] * c["N"] <= 1 << 20:
            return c


# ---- inputs ------------------------------------------------------------------------------


def _weights(c, g):
    H, d, G = c["H"], c["d"], c["G"]
    W = torch.randn(H, d, G, generator=g, device="cuda") / math.sqrt(d)
    bias = torch.randn(H, G, generator=g, device="cuda") * 0.1
    if c["tau"] == "half":
        tau = torch.full((H,), 0.5, device="cuda")
    else:
        tau = 0.3 + 0.7 * torch.rand(H, generator=g, device="cuda")
    return W, bias, tau


def _related(x, g):
    """Unit-variance features from a per-head linear map of x and as much noise."""
    B, N, H, d = x.shape
    A = torch.randn(H, d, d, generator=g, device="cuda") / math.sqrt(d)
    A = A / x[0, :4096].float().std()
    y = torch.randn(B, N, H, d, generator=g, device="cuda", dtype=x.dtype)
    for h in range(H):
        y[:, :, h] += x[:, :, h] @ A[h].to(x.dtype)
    return y.mul_(math.sqrt(0.5))


def _inputs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    B, N, H, d, G = c["B"], c["N"], c["H"], c["d"], c["G"]
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    x = torch.randn(B, N, H, d, generator=g, device="cuda", dtype=dt)
    if c["mixture"]:
        means = 2.0 * torch.randn(MIXTURE, H, d, generator=g, device="cuda")
        comp = torch.randint(0, MIXTURE, (B, N), generator=g, device="cuda")
        x = means.to(dt)[comp] + 0.5 * x
    v = {"x": x, "fx": _related(x, g)}
    v["W"], v["bias"], v["tau"] = _weights(c, g)
    if c["mixer"] == "identity":
        v["M"] = torch.eye(G, device="cuda") + 0.1 * torch.randn(H, G, G, generator=g, device="cuda")
    else:
        v["M"] = torch.randn(H, G, G, generator=g, device="cuda") / math.sqrt(G)
    if c["kind"] == "train":
        v["dout"] = _related(x, g)
    if c["kind"] == "untied":
        v["W2"], v["bias2"], v["tau2"] = _weights(c, g)
    return v


def prepare(case, seed):
    c = case
    v = _inputs(c, seed)
    train = c["kind"] == "train"
    s = {"kind": c["kind"], "in": v,
         "layer": fs.Coupling(c["B"], c["N"], c["H"], c["d"], c["G"], v["x"].dtype, backward=train)}
    if c["kind"] == "frozen":  # the first layer's statistics
        l = s["layer"]
        s["lse"] = torch.empty(c["B"], c["H"], c["N"], device="cuda")
        fs.fs_stats(l.shape, v["x"], v["W"], v["bias"], v["tau"], s["lse"], fs.workspace(l.shape, fs.FS_OP_STATS))
    return s


def run(state):
    l, v = state["layer"], state["in"]
    x, fx, W, bias, tau, M = v["x"], v["fx"], v["W"], v["bias"], v["tau"], v["M"]
    kind = state["kind"]
    if kind == "forward":
        return {"out": l.forward(x, fx, W, bias, tau, M)}
    if kind == "train":
        out = l.forward(x, fx, W, bias, tau, M)
        return {"out": out, **l.backward(x, fx, W, bias, tau, M, v["dout"])}
    if kind == "frozen":
        fs.fs_slice_fwd_lse(l.shape, x, fx, W, bias, tau, state["lse"], l.tokens, l.wsum, True, l.ws_slice)
        fs.fs_mix(l.shape, M, l.tokens, l.tokens_mixed)
        fs.fs_deslice_fwd(l.shape, x, W, bias, tau, l.tokens_mixed, state["lse"], l.out, l.ws_deslice)
        return {"out": l.out}
    fs.fs_slice_fwd(l.shape, x, fx, W, bias, tau, l.tokens, l.wsum, l.lse, True, l.ws_slice)
    fs.fs_mix(l.shape, M, l.tokens, l.tokens_mixed)
    fs.fs_deslice_fwd(l.shape, x, v["W2"], v["bias2"], v["tau2"], l.tokens_mixed, None, l.out, l.ws_deslice)
    return {"out": l.out}


def work(case):
    """Bytes: the point tensors read and written once, and the weights.  flops: one product
    of [points x d] by [d x slots] (2 C G per point) for each of the logits, the slice and
    the deslice; the untied deslice's own logits; in training d z', dfx, dx, dW and the two
    parts of dw; and the mix."""
    c = case
    pts, C, G, H, d = c["B"] * c["N"], c["H"] * c["d"], c["G"], c["H"], c["d"]
    e = 2 if c["dtype"] == "bf16" else 4
    train = c["kind"] == "train"
    tensors = 6 if train else 3  # x, fx, out; dout, dx, dfx
    weights = 4 * (H * d * G + H * G + H + H * G * G)
    n = {"forward": 3, "frozen": 3, "untied": 4, "train": 9}[c["kind"]]
    mix = 2 * c["B"] * H * G * G * d
    nbytes = tensors * pts * C * e + weights * (2 if train else 1)
    if c["kind"] == "frozen":
        nbytes += 4 * pts * H
    return {"bytes": nbytes, "flops": n * 2 * C * G * pts + mix * (3 if train else 1)}


# ---- the same in 64 bits -------------------------------------------------------------------


def exact(case, seed):
    """Plain torch in 64 bits, head by head over ranges of points; None where that takes long."""
    c = case
    train = c["kind"] == "train"
    # At the card's 64-bit rates the largest listed cases take 12 to 18 seconds.
    if _pairs(c) * c["d"] > 1 << 38:
        return None
    v = _inputs(c, seed)
    B, N, H, d, G = c["B"], c["N"], c["H"], c["d"], c["G"]
    eps = 1e-5
    x, fx, M = v["x"], v["fx"], v["M"].double()
    step = max(1, (1 << 26) // G)

    def parts():
        for n0 in range(0, N, step):
            yield slice(n0, min(N, n0 + step))

    def softmax(b, h, r, W, bias, tau):
        a = torch.addmm(bias[h].double(), x[b, r, h].double(), W[h].double()).div_(tau[h].double())
        return torch.softmax(a, dim=1), a

    out = torch.empty(B, N, H, d, dtype=torch.float64, device="cuda")
    res = {"out": out}
    if train:
        dout = v["dout"]
        dx, dfx = torch.empty_like(out), torch.empty_like(out)
        dW = torch.zeros(H, d, G, dtype=torch.float64, device="cuda")
        db = torch.zeros(H, G, dtype=torch.float64, device="cuda")
        dt = torch.zeros(H, dtype=torch.float64, device="cuda")
        dM = torch.zeros(H, G, G, dtype=torch.float64, device="cuda")
        res.update(dx_mid=dx, dfx=dfx, dW=dW, dbias=db, dtau=dt, dM=dM)
    W2, b2, t2 = (v["W2"], v["bias2"], v["tau2"]) if c["kind"] == "untied" else (v["W"], v["bias"], v["tau"])
    for b in range(B):
        for h in range(H):
            U = torch.zeros(G, d, dtype=torch.float64, device="cuda")
            S = torch.zeros(G, dtype=torch.float64, device="cuda")
            for r in parts():
                w, _ = softmax(b, h, r, v["W"], v["bias"], v["tau"])
                U += w.T @ fx[b, r, h].double()
                S += w.sum(0)
            z = U / (S + eps)[:, None]
            zm = M[h] @ z
            dzm = torch.zeros_like(zm)
            for r in parts():
                w, _ = softmax(b, h, r, W2, b2, t2)
                out[b, r, h] = w @ zm
                if train:
                    dzm += w.T @ dout[b, r, h].double()
            if not train:
                continue
            dz = M[h].T @ dzm
            dM[h] += dzm @ z.T
            dU = dz / (S + eps)[:, None]
            dS = -(dz * z).sum(1) / (S + eps)
            t = v["tau"][h].double()
            for r in parts():
                w, a = softmax(b, h, r, v["W"], v["bias"], v["tau"])
                f, o, xr = fx[b, r, h].double(), dout[b, r, h].double(), x[b, r, h].double()
                dfx[b, r, h] = w @ dU
                dw = (o @ zm.T).addmm_(f, dU.T).add_(dS)
                dw -= (w * dw).sum(1, keepdim=True)
                da = dw.mul_(w)
                dx[b, r, h] = (da @ v["W"][h].double().T) / t
                dW[h] += (xr.T @ da) / t
                db[h] += da.sum(0) / t
                a -= torch.logsumexp(a, dim=1, keepdim=True)
                dt[h] -= (da * a).sum() / t
    return res
