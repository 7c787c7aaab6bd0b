"""What the time of this library is measured on: the calls a program makes that serves a model with
moderately sparse weights, over the sizes it makes them at.

A case is one call, or the calls of one step, through the public binding (``tl3.Matrix``):

  spmm     Y = W X, activations [hidden, batch]        (decode and, from N = 65 on, prefill)
  nt       Yt = act(Xt W^T + b), activations [batch, hidden], with the fused bias and activation
  block    the six linear layers of one decoder block, each fed by the one before it
  host     Y = W X with X and Y in pinned host memory, the blocking call
  convert  dense W on the GPU -> packed weights in the model's arena on the GPU, nothing kept on the host
  save     dense W on the GPU -> the bytes of the container, in the buffer that goes to disk
  load     the bytes of a container from disk -> packed weights in the model's arena on the GPU

Shapes, sparsities and batch widths are those of the workload configurations and of the benchmark's
sweeps, and ragged neighbours of them.  Weights are N(0, 0.02) in fp16, pruned per row by magnitude, by
a calibrated score (|w| times the norm of the input channel) or at random; activations are N(0, 1).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_08786_b200 import tl3


def _case(op, M, K, N=0, sparsity=0.5, mask="magnitude", bias=False, act="none", name=None):
    c = {"op": op, "M": M, "K": K, "N": N, "sparsity": sparsity, "mask": mask, "bias": bias, "act": act}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest call: a head-sized projection at a batch of eight.  Latency.
        _case("spmm", 1024, 1024, 8, mask="random", name="decode_1024_n8"),
        # One sequence being generated, activations as the rest of the stack holds them.
        _case("nt", 4096, 4096, 1, mask="scored", bias=True, name="decode_nt_4096_n1"),
        # The ordinary product: an attention projection at hidden size 5120, batch 16.
        _case("spmm", 5120, 5120, 16, name="decode_5120_n16"),
        # One decoder block at hidden size 5120, batch 32: q, k, v, o, fc1 (ReLU), fc2, all with bias.
        _case("block", 5120, 20480, 32, bias=True, act="relu", name="block_5120_n32"),
        # Below 50 % sparsity a sixth of the weights is in the Residual layer; a gate projection with SiLU.
        _case("nt", 11008, 4096, 24, sparsity=0.4, act="silu", name="decode_nt_11008x4096_s40_n24"),
        # The largest decode product: up-projection at hidden size 9216, batch 64.
        _case("spmm", 36864, 9216, 64, name="decode_36864x9216_n64"),
        # Host buffers in and out, a sparser matrix, and no size a multiple of anything.
        _case("host", 5001, 3003, 5, sparsity=0.7, name="host_5001x3003_s70_n5"),
        # Prefill of 512 tokens through fc1 at hidden size 5120.
        _case("nt", 20480, 5120, 512, bias=True, act="relu", name="prefill_nt_20480x5120_n512"),
        # A short prompt or a wide batch, ragged in all three sizes.
        _case("spmm", 7001, 9003, 200, sparsity=0.6, name="prefill_7001x9003_s60_n200"),
        # Weights loaded dense (a checkpoint just read to the GPU) and packed there.
        _case("convert", 5120, 5120, name="convert_5120"),
        # A pruned layer written to disk in the three-layer container.
        _case("save", 4096, 11008, sparsity=0.6, mask="scored", name="save_4096x11008_s60"),
        # A container read from disk and packed on the GPU.
        _case("load", 20480, 5120, name="load_20480x5120"),
    ]


def _size(rng, lo, hi):
    """A size of the range, spread over its logarithm: as often ragged as a multiple of 128."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(128, (v + 64) // 128 * 128) if rng.random() < 0.5 else v


def draw(rng):
    op = rng.choice(["spmm", "spmm", "nt", "nt", "block", "host", "wide", "wide", "convert", "save", "load"])
    sparsity = rng.choice([0.4, 0.5, 0.5, 0.5, 0.6, 0.7])
    mask = rng.choice(["magnitude", "magnitude", "scored", "random"])
    bias, act = rng.random() < 0.5, rng.choice(["none", "none", "relu", "silu", "gelu_tanh"])
    narrow = int(round(math.exp(rng.uniform(0.0, math.log(64)))))           # 1 .. 64
    wide = int(round(math.exp(rng.uniform(math.log(65), math.log(512)))))   # 65 .. 512
    if op == "block":
        hidden = _size(rng, 1024, 4608)
        return _case("block", hidden, 4 * hidden, narrow, sparsity, mask, bias, act)
    M, K = _size(rng, 700, 24000), _size(rng, 700, 24000)
    most = {"spmm": 105e6, "nt": 105e6, "wide": 80e6}.get(op, 60e6)
    while M * K > most:
        M, K = max(700, M * 3 // 4), max(700, K * 3 // 4)
    if op == "wide":
        op = rng.choice(["spmm", "nt"])
        return _case(op, M, K, wide, sparsity, mask, bias and op == "nt", act if op == "nt" else "none")
    if op == "nt":
        return _case("nt", M, K, narrow, sparsity, mask, bias, act)
    if op in ("spmm", "host"):
        return _case(op, M, K, narrow, sparsity, mask)
    return _case(op, M, K, 0, sparsity, mask)


# ---- inputs -------------------------------------------------------------------------------------
def _weights(g, M, K, sparsity, mask):
    """Pruned fp16 weights on the GPU (pruned entries are +0.0)."""
    W = torch.empty((M, K), dtype=torch.float16, device="cuda")
    keep = K - int(round(sparsity * K))
    scale = None
    if mask == "scored":
        scale = torch.exp(0.5 * torch.randn(K, generator=g, device="cuda"))     # outlier input channels
    for r in range(0, M, 4096):
        w = torch.randn((min(4096, M - r), K), generator=g, device="cuda").mul_(0.02).half()
        if mask == "random":
            kept = torch.rand(w.shape, generator=g, device="cuda") >= sparsity
        else:
            score = w.abs().float()
            if scale is not None:
                score *= scale
            best = torch.sort(score, dim=1, descending=True, stable=True).indices[:, :keep]
            kept = torch.zeros(w.shape, dtype=torch.bool, device="cuda").scatter_(1, best, True)
        W[r:r + 4096] = torch.where(kept, w, torch.zeros_like(w))
    return W


def _packed(g, M, K, case):
    """A handle with its weights on the GPU, as a program keeps it for the life of the model."""
    m = tl3.Matrix.encode_on_device(_weights(g, M, K, case["sparsity"], case["mask"]), device_only=True)
    m.upload_packed_on_device()
    return m


def _activations(g, rows, cols):
    """rows x cols on the GPU, the pitch a multiple of eight elements."""
    buf = torch.empty((rows, (cols + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    return buf.normal_(generator=g)[:, :cols]


def _bias(g, case, M):
    return torch.randn(M, generator=g, device="cuda").mul_(0.1).half() if case["bias"] else None


def _room(M, K):
    """Bytes that hold the packed weights or the container of a layer at 40 % sparsity or more."""
    return 2 * ((M + 127) // 128 * 128) * ((K + 127) // 128 * 128) + (1 << 20)


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    op, M, K, N = case["op"], case["M"], case["K"], case["N"]
    s = {"op": op, "act": None if case["act"] == "none" else case["act"], "N": N}
    if op in ("spmm", "nt"):
        s["m"] = _packed(g, M, K, case)
        s["X"] = _activations(g, K, N) if op == "spmm" else _activations(g, N, K)
        s["bias"] = _bias(g, case, M)
        # a decode step writes into buffers that it keeps, a prefill of any length makes its output
        s["Y"] = None if N > 64 else torch.empty((M, N) if op == "spmm" else (N, M), dtype=torch.float16, device="cuda")
    elif op == "block":
        shapes = [(M, M)] * 4 + [(K, M), (M, K)]                    # q, k, v, o, fc1, fc2
        s["layers"] = [(_packed(g, r, c, case), _bias(g, case, r), _activations(g, N, r)) for r, c in shapes]
        s["X"] = _activations(g, N, M)
    elif op == "host":
        s["m"] = _packed(g, M, K, case)
        s["X"] = torch.empty((K, N), dtype=torch.float16, pin_memory=True)
        s["X"].copy_(torch.randn((K, N), generator=g, device="cuda").half())
        s["Y"] = torch.empty((M, N), dtype=torch.float16, pin_memory=True)
        s["dX"] = torch.empty(K * ((N + 7) // 8 * 8), dtype=torch.float16, device="cuda")
        s["dY"] = torch.empty(M * N, dtype=torch.float16, device="cuda")
        s["ws"] = s["m"].new_workspace(N)
        s["Xn"], s["Yn"] = s["X"].numpy(), s["Y"].numpy()
    elif op in ("convert", "save"):
        s["W"] = _weights(g, M, K, case["sparsity"], case["mask"])
        if op == "convert":
            s["arena"] = torch.zeros(_room(M, K), dtype=torch.uint8, device="cuda")
        else:
            s["file"] = np.zeros(_room(M, K), dtype=np.uint8)
    else:
        m = tl3.Matrix.encode_on_device(_weights(g, M, K, case["sparsity"], case["mask"]))
        s["file"] = m.serialize()
        s["arena"] = torch.zeros(_room(M, K), dtype=torch.uint8, device="cuda")
        m.close()
    return s


# ---- one pass -----------------------------------------------------------------------------------
def run(s):
    op = s["op"]
    if op == "spmm":
        return s["m"].spmm(s["X"], s["Y"])
    if op == "nt":
        return s["m"].spmm_nt(s["X"], s["Y"], bias=s["bias"], activation=s["act"])
    if op == "block":
        (q, bq, yq), (k, bk, yk), (v, bv, yv), (o, bo, yo), (f1, b1, y1), (f2, b2, y2) = s["layers"]
        q.spmm_nt(s["X"], yq, bias=bq)
        k.spmm_nt(s["X"], yk, bias=bk)
        v.spmm_nt(s["X"], yv, bias=bv)
        o.spmm_nt(yv, yo, bias=bo)                  # (attention itself is not this library's: v stands for its result)
        f1.spmm_nt(yo, y1, bias=b1, activation=s["act"])
        f2.spmm_nt(y1, y2, bias=b2)
        return [yq, yk, yv, yo, y1, y2]
    if op == "host":
        s["m"].spmm_host(s["Xn"], s["Yn"], s["dX"], s["dY"], s["ws"])
        return s["Yn"]
    if op == "save":
        m = tl3.Matrix.encode_on_device(s["W"])
        data = m.serialize()
        s["file"][:len(data)] = np.frombuffer(data, dtype=np.uint8)
        return s["file"]
    if op == "convert":
        m = tl3.Matrix.encode_on_device(s["W"], device_only=True)
    else:
        m = tl3.Matrix.deserialize(s["file"])
    blob = m.upload_packed_on_device()
    s["arena"][:blob.numel()].copy_(blob)
    m.bind(s["arena"])
    return s["arena"]


# ---- what a pass cannot do without, and how closely results agree ---------------------------------
def _weight_bytes(case, M, K):
    """Kept values at two bytes, positions at one bit per weight."""
    return M * K * (2.0 * (1.0 - case["sparsity"]) + 0.125)


def work(case):
    op, M, K, N = case["op"], case["M"], case["K"], case["N"]
    keep = 1.0 - case["sparsity"]
    if op == "block":
        shapes = [(M, M)] * 4 + [(K, M), (M, K)]
        return {"bytes": sum(_weight_bytes(case, r, c) + 2.0 * N * (r + c) for r, c in shapes),
                "flops": sum(2.0 * r * c * keep * N for r, c in shapes)}
    if op in ("spmm", "nt", "host"):
        return {"bytes": _weight_bytes(case, M, K) + 2.0 * N * (M + K), "flops": 2.0 * M * K * keep * N}
    if op in ("convert", "save"):
        return {"bytes": 2.0 * M * K + _weight_bytes(case, M, K), "flops": 0}
    return {"bytes": 2.0 * _weight_bytes(case, M, K), "flops": 0}


def tolerance(case):
    if case["op"] in ("convert", "save", "load"):
        return "exact"
    # fp32 sums and one rounding to fp16 differ from the same product in 64 bits by 2.1e-4 (largest
    # element: 4.9e-4) whatever the size; three roundings in a row by 4.2e-4 (2.0e-3).  Four times that.
    return {"rel": 1.7e-3, "max": 8e-3} if case["op"] == "block" else {"rel": 8e-4, "max": 2e-3}


# ---- the same results in 64 bits -------------------------------------------------------------------
def _linear(W, Xt, bias, act):
    """act(Xt W^T + b) in 64 bits."""
    y = Xt @ W.double().T
    if bias is not None:
        y += bias.double()
    if act == "relu":
        return y.relu_()
    if act == "silu":
        return y / (1.0 + torch.exp(-y))
    if act == "gelu_tanh":
        return 0.5 * y * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (y + 0.044715 * y ** 3)))
    return y


def exact(case, seed):
    """What run() returns for these inputs, from the dense weights (the draws are those of prepare())."""
    op, M, K, N = case["op"], case["M"], case["K"], case["N"]
    if op in ("convert", "save", "load"):
        return None                                                 # bytes
    g = torch.Generator(device="cuda").manual_seed(seed)
    if op == "block":
        layers = []
        for r, c in [(M, M)] * 4 + [(K, M), (M, K)]:
            W, b = _weights(g, r, c, case["sparsity"], case["mask"]), _bias(g, case, r)
            _activations(g, N, r)                                   # the output buffer's first contents
            layers.append((W, b))
        x = _activations(g, N, M).double()
        (q, bq), (k, bk), (v, bv), (o, bo), (f1, b1), (f2, b2) = layers
        yq, yk, yv = _linear(q, x, bq, "none"), _linear(k, x, bk, "none"), _linear(v, x, bv, "none")
        yo = _linear(o, yv, bo, "none")
        y1 = _linear(f1, yo, b1, case["act"])
        return [yq, yk, yv, yo, y1, _linear(f2, y1, b2, "none")]
    W = _weights(g, M, K, case["sparsity"], case["mask"])
    if op == "nt":
        X = _activations(g, N, K).double()
        return _linear(W, X, _bias(g, case, M), case["act"])
    X = _activations(g, K, N) if op == "spmm" else torch.randn((K, N), generator=g, device="cuda").half()
    y = W.double() @ X.double()
    return y if op == "spmm" else y.cpu().numpy()
