"""Performance cases: the work a user of the library has it do, through its public entry points.

A case is a dict of plain values.  Its "op" says which entry point runs it:

* "gemm": ``kselect.gemm`` with a shipped deployment, C = op(A) op(B) + beta C, batched;
* "grouped": ``kselect.gemm_grouped``, an uneven group of GEMMs in one call;
* "vgg16": ``vgg.VGG16.forward``, a whole network's inference, returning its logits;
* "mlp": ``kselect.mlp_loss_grad``, one training pass of the learned selector.

Sizes come from the tuning grid (M, N, K log-uniform in [16, 4096], batch in
{1, 2, 4, 8, 16}, either storage order of A and B), the single 256-cubed GEMM, the
large cubes that the benchmark times, VGG16's layers, the uneven groups (32 to 4096)
and the selector's training set.  Operand values are those of the repository's
recipes: uniform in [-1, 1); He-normal weights and non-negative images for VGG16.
"""
import json
import math
import os

import numpy as np
import torch

from paper_2008_13145_gb300 import kselect as ks
from paper_2008_13145_gb300 import vgg

DEPLOY = os.path.join(os.path.dirname(os.path.abspath(vgg.__file__)), "deploy")

# FP32 requests of more work than this take longer than any listed case.
F32_FLOPS_MOST = 2 * 4096 ** 3
TC_FLOPS_MOST = 2 * 8192 ** 3


def gemm(name, deploy, M, N, K, batch=1, ta="N", tb="N", pad=1, beta=0.0):
    """pad: leading dimensions are rounded up to this many elements (1: rows packed as they are)."""
    return {"name": name, "op": "gemm", "deploy": deploy, "M": M, "N": N, "K": K, "batch": batch, "ta": ta, "tb": tb,
            "pad": pad, "beta": beta}


def listed():
    return [
        # One small FP32 product: the latency of a call (the paper's smallest complete example).
        gemm("f32 256", "f32", 256, 256, 256),
        # Few output tiles and a long K, batched and ragged, A stored transposed: work has to be found along K.
        gemm("f32 ragged long-K", "f32", 323, 312, 3945, 8, "T", "N"),
        # The top of the tuning grid: a large square FP32 product.
        gemm("f32 4096", "f32", 4096, 4096, 4096),
        # An ordinary FP32 product for the deployment that may also use tensor cores, accumulated into C.
        gemm("f32mix 1733x912x1408", "f32mix", 1733, 912, 1408, 2, "N", "T", 4, 0.5),
        # FP32 storage at split-BF16 accuracy: an ordinary batched size of the grid.
        gemm("x3 1024x768x640 b4", "f32x3", 1024, 768, 640, 4, "N", "N", 4),
        # TF32 with a large output for its K: writing C is most of it.
        gemm("tf32 3634x1714x406 b8", "tf32", 3634, 1714, 406, 8, "T", "T", 4),
        # The largest product that the benchmark times: the tensor cores' sustained rate.
        gemm("bf16 8192", "bf16", 8192, 8192, 8192, 1, "N", "T", 8),
        # A ragged batch of small BF16 products whose rows are not 16-byte aligned.
        gemm("bf16 ragged 2185x637x95 b16", "bf16", 2185, 637, 95, 16, "N", "N", 1),
        # An uneven group of 256 problems in one call (a mixture of layers or experts), BF16.
        {"name": "grouped bf16 256", "op": "grouped", "family": "bf16", "count": 256, "lo": 32, "hi": 4096,
         "draw": 3},
        # A smaller group with FP32 operands at FP32-level accuracy.
        {"name": "grouped f32 48", "op": "grouped", "family": "f32x3", "count": 48, "lo": 64, "hi": 2048, "draw": 5},
        # Whole-network inference: 13 convolutions and 3 fully connected layers, FP32, 16 images.
        {"name": "vgg16 f32 b16", "op": "vgg16", "deploy": "f32", "batch": 16, "layout": "nhwc", "hw": 224},
        # Forward and backward of the learned selector over its training set.
        {"name": "mlp loss+grad 2000", "op": "mlp", "n": 2000, "masked": True},
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(["f32", "f32mix", "f32x3", "tf32", "bf16", "grouped", "vgg16", "mlp"],
                       [5, 2, 2, 2, 3, 2, 1, 1])[0]
    if kind == "grouped":
        return {"op": "grouped", "family": rng.choice(["bf16", "tf32", "f32x3"]), "count": _log_int(rng, 16, 256),
                "lo": rng.choice([32, 64, 128]), "hi": rng.choice([1024, 2048, 3000]), "draw": rng.randrange(1 << 20)}
    if kind == "vgg16":
        layout = rng.choice(["nhwc", "batched"])
        return {"op": "vgg16", "deploy": rng.choice(["f32", "f32mix"]),
                "batch": rng.randint(1, 15 if layout == "nhwc" else 8), "layout": layout,
                "hw": rng.choice([64, 96, 160, 224])}
    if kind == "mlp":
        return {"op": "mlp", "n": _log_int(rng, 100, 20000), "masked": rng.random() < 0.5}
    tc = kind in ("tf32", "bf16")
    hi, most = (8192, TC_FLOPS_MOST) if tc else (4096, F32_FLOPS_MOST)
    while True:
        c = gemm("", kind, _log_int(rng, 16, hi), _log_int(rng, 16, hi), _log_int(rng, 16, hi),
                 rng.choice([1, 2, 4, 8, 16]), rng.choice("NT"), rng.choice("NT"),
                 rng.choice([1, 8 if kind == "bf16" else 4]), rng.choice([0.0, 0.0, 0.0, 0.5]))
        elements = c["batch"] * (c["M"] * c["K"] + c["K"] * c["N"] + c["M"] * c["N"])
        if 2 * c["M"] * c["N"] * c["K"] * c["batch"] <= most and elements <= 200e6:
            del c["name"]
            return c


# ---------------------------------------------------------------- inputs
def _generator(seed, stream):
    return torch.Generator("cuda").manual_seed((seed * 1000003 + stream) & 0x7FFFFFFFFFFF)


def _uniform(shape, seed, stream):
    return torch.rand(shape, generator=_generator(seed, stream), device="cuda") * 2 - 1


def _up(x, m):
    return (x + m - 1) // m * m


def _operand(batch, rows, cols, pad, seed, stream, dtype):
    """(batch, rows, cols) uniform values inside rows of _up(cols, pad) elements."""
    t = torch.zeros((batch, rows, _up(cols, pad)), device="cuda", dtype=dtype)
    t[:, :, :cols] = _uniform((batch, rows, cols), seed, stream).to(dtype)
    return t


def _gemm_inputs(c, seed):
    M, N, K, b, pad = c["M"], c["N"], c["K"], c["batch"], c["pad"]
    dtype = torch.bfloat16 if c["deploy"] == "bf16" else torch.float32
    A = _operand(b, *((M, K) if c["ta"] == "N" else (K, M)), pad, seed, 1, dtype)
    B = _operand(b, *((K, N) if c["tb"] == "N" else (N, K)), pad, seed, 2, dtype)
    C = _operand(b, M, N, pad, seed, 3, torch.float32)
    return A, B, C


def _group_shapes(c):
    rng = np.random.Generator(np.random.Philox(key=[c["draw"], 0]))
    return np.clip(np.rint(np.exp(rng.uniform(math.log(c["lo"]), math.log(c["hi"]), (3, c["count"])))).astype(np.int64),
                   c["lo"], c["hi"]).T.tolist()


def _group_inputs(c, seed):
    """Per problem (M, N, K, A, B, C): A is M x K, B is N x K, rows 16-byte aligned; the C's are parts of one buffer."""
    dtype = torch.bfloat16 if c["family"] == "bf16" else torch.float32
    shapes = _group_shapes(c)
    out = torch.zeros(sum(M * _up(N, 8) for M, N, _ in shapes), device="cuda")
    at, probs = 0, []
    for i, (M, N, K) in enumerate(shapes):
        A = _operand(1, M, K, 8, seed, 2 * i, dtype)[0]
        B = _operand(1, N, K, 8, seed, 2 * i + 1, dtype)[0]
        n = M * _up(N, 8)
        probs.append((M, N, K, A, B, out[at:at + n].view(M, _up(N, 8))))
        at += n
    return probs, out


def _images(c, seed):
    """Non-negative images, NHWC or NCHW as the layout wants them."""
    x = torch.randn((c["batch"], c["hw"], c["hw"], 3), generator=_generator(seed, 9), device="cuda").abs()
    return x if c["layout"] == "nhwc" else x.permute(0, 3, 1, 2).contiguous()


def _mlp_inputs(c, seed):
    n = c["n"]
    params = 0.2 * torch.randn(ks.MLP_PARAMS, generator=_generator(seed, 1), device="cuda")
    X = torch.rand((n, 7), generator=_generator(seed, 2), device="cuda")
    T = -3 * torch.rand((n, 8), generator=_generator(seed, 3), device="cuda")
    mask = (torch.rand((n, 8), generator=_generator(seed, 4), device="cuda") > 0.1).float() if c["masked"] else None
    return params, X, T, mask


def _deployment(name):
    with open(os.path.join(DEPLOY, name + ".json")) as f:
        return json.load(f)


def prepare(case, seed):
    c = case
    if c["op"] == "gemm":
        A, B, C = _gemm_inputs(c, seed)
        return {"c": c, "h": ks.Handle(_deployment(c["deploy"])), "A": A, "B": B, "C": C}
    if c["op"] == "grouped":
        probs, out = _group_inputs(c, seed)
        problems = [dict(M=M, N=N, K=K, transA="N", transB="T", alpha=1.0, beta=0.0, A=A, lda=A.shape[1], B=B,
                         ldb=B.shape[1], C=C, ldc=C.shape[1]) for M, N, K, A, B, C in probs]
        return {"c": c, "h": ks.Handle(_deployment("grouped")[c["family"]]["selector"]), "problems": problems,
                "out": out, "precision": ks.PRECISIONS[c["family"]]}
    if c["op"] == "vgg16":
        net = vgg.VGG16(ks.Handle(_deployment(c["deploy"])), c["batch"], hw=c["hw"], seed=seed, layout=c["layout"])
        return {"c": c, "net": net, "x": _images(c, seed)}
    params, X, T, mask = _mlp_inputs(c, seed)
    return {"c": c, "params": params, "X": X, "T": T, "mask": mask, "grad": torch.empty_like(params),
            "loss": torch.empty(1, device="cuda")}


def run(state):
    c = state["c"]
    if c["op"] == "gemm":
        A, B, C = state["A"], state["B"], state["C"]
        ks.gemm(state["h"], c["ta"], c["tb"], c["M"], c["N"], c["K"], 1.0, A, A.shape[2], B, B.shape[2], c["beta"], C,
                C.shape[2], c["batch"])
        return C[:, :, :c["N"]]
    if c["op"] == "grouped":
        ks.gemm_grouped(state["h"], state["problems"], state["precision"])
        return state["out"]
    if c["op"] == "vgg16":
        return state["net"].forward(state["x"])
    ks.mlp_loss_grad(state["params"], state["X"], state["T"], state["mask"], state["grad"], state["loss"])
    return {"grad": state["grad"], "loss": state["loss"]}


# ---------------------------------------------------------------- what a pass cannot do without
def _vgg_layers(hw):
    """[("conv", side, Cin, Cout) | ("pool",) | ("fc", Kin, Nout)] of VGG16 for hw x hw images."""
    out, cin, side = [], 3, hw
    for v in (64, 64, 0, 128, 128, 0, 256, 256, 256, 0, 512, 512, 512, 0, 512, 512, 512, 0):
        if v == 0:
            out.append(("pool",))
            side //= 2
        else:
            out.append(("conv", side, cin, v))
            cin = v
    kin = side * side * cin
    for n in (4096, 4096, 1000):
        out.append(("fc", kin, n))
        kin = n
    return out


def work(case):
    c = case
    if c["op"] == "gemm":
        M, N, K, b = c["M"], c["N"], c["K"], c["batch"]
        elem = 2 if c["deploy"] == "bf16" else 4
        return {"bytes": b * (elem * (M * K + K * N) + 4 * M * N * (2 if c["beta"] else 1)), "flops": 2 * M * N * K * b}
    if c["op"] == "grouped":
        elem = 2 if c["family"] == "bf16" else 4
        return {"bytes": sum(elem * (M * K + K * N) + 4 * M * N for M, N, K in _group_shapes(c)),
                "flops": sum(2 * M * N * K for M, N, K in _group_shapes(c))}
    if c["op"] == "vgg16":
        n, flops, weights = c["batch"], 0, 0
        for layer in _vgg_layers(c["hw"]):
            if layer[0] == "conv":
                _, side, ci, co = layer
                flops += 2 * n * side * side * 9 * ci * co
                weights += 9 * ci * co + co
            elif layer[0] == "fc":
                _, kin, nout = layer
                flops += 2 * n * kin * nout
                weights += kin * nout + nout
        return {"bytes": 4 * (weights + n * (c["hw"] * c["hw"] * 3 + 1000)), "flops": flops}
    # Forward, then the gradients of the activations (all layers but the first) and of the weights.
    n, w = c["n"], (7 * 64, 64 * 64, 64 * 8)
    return {"bytes": 4 * (2 * ks.MLP_PARAMS + n * (7 + 8 + (8 if c["masked"] else 0)) + 1),
            "flops": 2 * n * (2 * sum(w) + w[1] + w[2])}


# ---------------------------------------------------------------- the same results in 64 bits
def _exact_vgg(c, seed):
    """The network with the weights VGG16 draws from its seed, written out with torch in 64 bits."""
    def normal(stream, rows, cols, std):
        rng = np.random.Generator(np.random.Philox(key=[seed, stream]))
        w = rng.normal(0.0, std, size=(1, rows, cols)).astype(np.float32)[0]
        return torch.from_numpy(w).cuda().double()

    x = _images(c, seed).double()
    if c["layout"] == "nhwc":
        x = x.permute(0, 3, 1, 2).contiguous()
    layers = _vgg_layers(c["hw"])
    for i, layer in enumerate(layers):
        if layer[0] == "pool":
            x = torch.nn.functional.max_pool2d(x, 2)
        elif layer[0] == "conv":
            _, side, ci, co = layer
            W = normal(2 * i, co, 9 * ci, float(np.sqrt(2.0 / (9 * ci)))).view(co, 3, 3, ci)  # column (kh, kw, c)
            bias = normal(2 * i + 1, 1, co, 0.05)[0]
            p = torch.nn.functional.pad(x, (1, 1, 1, 1))
            y = torch.zeros((co, x.shape[0] * side * side), device="cuda", dtype=torch.float64)
            for kh in range(3):
                for kw in range(3):
                    part = p[:, :, kh:kh + side, kw:kw + side].transpose(0, 1).reshape(ci, -1)
                    y.addmm_(W[:, kh, kw], part)
            x = torch.relu(y + bias[:, None]).view(co, -1, side, side).transpose(0, 1).contiguous()
        else:
            _, kin, nout = layer
            if x.dim() == 4:
                x = x.permute(0, 2, 3, 1).reshape(x.shape[0], -1)  # the fully connected weights read (h, w, c)
            x = x @ normal(2 * i, nout, kin, float(np.sqrt(2.0 / kin))).t() + normal(2 * i + 1, 1, nout, 0.05)[0]
            if i + 1 < len(layers):
                x = torch.relu(x)
    return x


def exact(case, seed):
    c = case
    if c["op"] == "gemm":
        A, B, C = _gemm_inputs(c, seed)
        M, N, K = c["M"], c["N"], c["K"]
        out = torch.empty((c["batch"], M, N), device="cuda", dtype=torch.float64)
        for i in range(c["batch"]):
            a = A[i, :, :K].double() if c["ta"] == "N" else A[i, :, :M].double().t()
            b = B[i, :, :N].double() if c["tb"] == "N" else B[i, :, :K].double().t()
            out[i] = a @ b
            if c["beta"]:
                out[i] += c["beta"] * C[i, :, :N].double()
        return out
    if c["op"] == "grouped":
        probs, out = _group_inputs(c, seed)
        out = out.double()
        at = 0
        for M, N, K, A, B, C in probs:
            out[at:at + C.numel()].view(M, -1)[:, :N] = A[:, :K].double() @ B[:, :K].double().t()
            at += C.numel()
        return out
    if c["op"] == "vgg16":
        return _exact_vgg(c, seed)
    params, X, T, mask = _mlp_inputs(c, seed)
    p = params.double().requires_grad_()
    w1, b1, w2, b2, w3, b3 = torch.split(p, [448, 64, 4096, 64, 512, 8])
    h = torch.relu(X.double() @ w1.view(7, 64) + b1)
    h = torch.relu(h @ w2.view(64, 64) + b2)
    r = (h @ w3.view(64, 8) + b3 - T.double()) * (1.0 if mask is None else mask.double())
    loss = (r * r).sum() / (T.numel() if mask is None else mask.double().sum())
    loss.backward()
    return {"grad": p.grad, "loss": loss.detach().view(1)}
