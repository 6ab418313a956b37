"""Timed cases of the Monarch multiply library: what its users run, through the public binding.

A case is a dict of plain values.  ``kind`` names the use, the other keys its sizes:

  fwd        y = M x                                          (inference through one layer)
  train      y = M x, then dx, dL, dR reusing u of the forward  (one layer of a training step)
  mlp        y = M2 GELU(M1 x + b1) + b2                      (inference through the feed-forward block)
  mlp_train  the block forward, then its seven gradients      (the block in a training step)
  rect_train general class, few large blocks: forward, then dx, dL, dR
  cplx       z = M^H (M x) with complex factors               (one MM* product)
  project    dense matrix -> nearest Monarch matrix, materialised  (dense-to-sparse initialisation)

Tensors have the distributions of ``paper_2204_00595_b200.inputs``: unit-variance activations and gradients,
weights of variance 1 / fan-in, biases of variance 0.02.
"""
import math

import torch

import paper_2204_00595_b200 as P

DTYPES = {"bf16": (torch.bfloat16, P.BF16, 2), "f32": (torch.float32, P.F32, 4)}


def listed():
    return [
        # One small fp32 layer on one small batch: the latency of a single call.
        {"name": "fwd_f32_m16_t64", "kind": "fwd", "dtype": "f32", "m": 16, "tokens": 64},
        # Decoding: a feed-forward block on one token of each of a few concurrent sequences.
        {"name": "mlp_bf16_m64_t16", "kind": "mlp", "dtype": "bf16", "m": 64, "tokens": 16},
        # Prefill / batch inference through a narrow layer: 16 sequences of 1024 tokens.
        {"name": "fwd_bf16_m32_t16384", "kind": "fwd", "dtype": "bf16", "m": 32, "tokens": 16384},
        # Training a narrow layer on packed sequences of uneven length, one of several accumulated micro-batches.
        {"name": "train_bf16_m32_t4999_acc", "kind": "train", "dtype": "bf16", "m": 32, "tokens": 4999,
         "accumulate": True},
        # Training an ordinary layer.
        {"name": "train_bf16_m64_t8192", "kind": "train", "dtype": "bf16", "m": 64, "tokens": 8192},
        # Training the widest layer.
        {"name": "train_bf16_m128_t4096", "kind": "train", "dtype": "bf16", "m": 128, "tokens": 4096},
        # Training in single precision (scientific models, numerically delicate layers).
        {"name": "train_f32_m64_t2048", "kind": "train", "dtype": "f32", "m": 64, "tokens": 2048},
        # Prefill / batch inference through a feed-forward block, the largest batch.
        {"name": "mlp_bf16_m64_t32768", "kind": "mlp", "dtype": "bf16", "m": 64, "tokens": 32768},
        # A feed-forward block in a training step.
        {"name": "mlp_train_bf16_m64_t4096", "kind": "mlp_train", "dtype": "bf16", "m": 64, "tokens": 4096},
        # Training with the four large blocks that the paper's language and vision models use.
        {"name": "rect_train_bf16_4x1024_t8192", "kind": "rect_train", "dtype": "bf16", "q": 4, "b1": 1024,
         "b": 1024, "r": 4, "tokens": 8192},
        # A transform with complex factors and its conjugate transpose (the MM* class: DFT-like operators).
        {"name": "cplx_bf16_m64_t2048", "kind": "cplx", "dtype": "bf16", "m": 64, "tokens": 2048},
        # Converting a pretrained 4096 x 4096 weight matrix.
        {"name": "project_f32_m64", "kind": "project", "dtype": "f32", "m": 64, "noise": 2.0},
    ]


def draw(rng):
    kind = rng.choice(["fwd", "fwd", "train", "train", "mlp", "mlp_train", "rect_train", "cplx", "project"])
    case = {"kind": kind, "dtype": rng.choice(["bf16", "bf16", "bf16", "f32"])}
    if kind == "project":
        case["m"] = rng.choice([16, 32, 64])
        case["noise"] = round(rng.uniform(0.5, 3.0), 3)
        return case
    if kind == "rect_train":
        # slices of 192 .. 1024: a quarter of the usual hidden sizes 768 .. 4096, square and expanding layers
        case.update(dtype="bf16", q=4, b1=rng.choice([192, 256, 384, 512, 768, 1024]),
                    b=rng.choice([192, 256, 384, 512, 768, 1024]), r=rng.choice([2, 4]))
        case["tokens"] = log_int(rng, 64, 8192)
        return case
    m = case["m"] = rng.choice([16, 32, 64, 64, 128, 128])
    # elements of one token tensor: at most those of the largest listed batches; fewer in fp32 and where a pass is
    # several multiplies
    most = {"fwd": 1 << 26, "train": 1 << 26, "mlp": 1 << 26, "mlp_train": 1 << 25, "cplx": 1 << 25}[kind]
    if case["dtype"] == "f32":
        most >>= 3
    case["tokens"] = log_int(rng, 1, min(32768, most // (m * m)))
    if kind == "train":
        case["accumulate"] = rng.random() < 0.3
    return case


def log_int(rng, low, high):
    return max(low, min(high, round(math.exp(rng.uniform(math.log(low), math.log(high))))))


def prepare(case, seed):
    kind, (dt, code, _) = case["kind"], DTYPES[case["dtype"]]
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape, std=1.0):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).mul_(std).to(dt)

    def zeros(*shape):
        return torch.zeros(shape, device="cuda", dtype=torch.float32)

    s = {"kind": kind, "accumulate": int(case.get("accumulate", False))}
    if kind == "rect_train":
        q, b1, b, r, t = (case[k] for k in ("q", "b1", "b", "r", "tokens"))
        s.update(sizes=(t, q, b1, b, r), x=normal(t, q * b1), R=normal(q, b, b1, std=b1 ** -0.5),
                 L=normal(b, r, q, std=q ** -0.5), dy=normal(t, r * b))
        s.update(y=torch.empty_like(s["dy"]), dx=torch.empty_like(s["x"]), dL=zeros(b, r, q), dR=zeros(q, b, b1),
                 ws=P.Workspace(P.monarch_rect_workspace_bytes(t, q, b1, b, r, code)),
                 ws_bwd=P.Workspace(P.monarch_rect_bwd_workspace_bytes(t, q, b1, b, r, code)))
        return s
    m = case["m"]
    n, std = m * m, m ** -0.5
    if kind == "project":
        # a Monarch matrix under dense noise of `noise` times its entries' deviation
        L, R = normal(m, m, m, std=std), normal(m, m, m, std=std)
        A = torch.empty(n, n, device="cuda", dtype=dt)
        P.monarch_dense(L, R, A, n, m)
        A.add_(normal(n, n, std=case["noise"] / m))
        s.update(sizes=(n, m), A=A, L=torch.empty_like(L), R=torch.empty_like(R), M=torch.empty_like(A))
        return s
    t = case["tokens"]
    s["sizes"] = (t, n, m)
    planes = (2,) if kind == "cplx" else ()
    s["x"] = normal(*planes, t, n)
    s["y"] = torch.empty_like(s["x"])

    def workspace(op):
        return P.Workspace.for_op(op, t, m, code)

    if kind == "cplx":
        s.update(L=normal(2, m, m, m, std=std * 0.5 ** 0.5), R=normal(2, m, m, m, std=std * 0.5 ** 0.5),
                 z=torch.empty_like(s["x"]), ws=workspace(P.OP_CPLX))
        return s
    if kind in ("fwd", "train"):
        s.update(L=normal(m, m, m, std=std), R=normal(m, m, m, std=std), ws=workspace(P.OP_FWD))
    else:
        s.update(L1=normal(m, m, m, std=std), R1=normal(m, m, m, std=std), b1=normal(n, std=0.02 ** 0.5),
                 L2=normal(m, m, m, std=std), R2=normal(m, m, m, std=std), b2=normal(n, std=0.02 ** 0.5),
                 ws=workspace(P.OP_MLP_FWD))
    if kind in ("train", "mlp_train"):
        s.update(dy=normal(t, n), dx=torch.empty_like(s["x"]),
                 ws_bwd=workspace(P.OP_BWD if kind == "train" else P.OP_MLP_BWD))
    if kind == "train":
        s.update(dL=zeros(m, m, m), dR=zeros(m, m, m))
    if kind == "mlp_train":
        s["grads"] = [zeros(m, m, m), zeros(m, m, m), zeros(n), zeros(m, m, m), zeros(m, m, m), zeros(n)]
    return s


def run(s):
    kind = s["kind"]
    if kind == "fwd":
        P.monarch_fwd(s["x"], s["L"], s["R"], s["y"], *s["sizes"], s["ws"])
        return s["y"]
    if kind == "train":
        P.monarch_fwd(s["x"], s["L"], s["R"], s["y"], *s["sizes"], s["ws"])
        P.monarch_bwd(s["x"], s["dy"], s["L"], s["R"], s["dx"], s["dL"], s["dR"], s["accumulate"], *s["sizes"],
                      s["ws_bwd"], fwd_workspace=s["ws"])
        return s["y"], s["dx"], s["dL"], s["dR"]
    if kind in ("mlp", "mlp_train"):
        P.monarch_mlp_fwd(s["x"], s["L1"], s["R1"], s["b1"], s["L2"], s["R2"], s["b2"], s["y"], *s["sizes"], s["ws"])
        if kind == "mlp":
            return s["y"]
        P.monarch_mlp_bwd(s["x"], s["dy"], s["L1"], s["R1"], s["b1"], s["L2"], s["R2"], s["dx"], *s["grads"],
                          s["accumulate"], *s["sizes"], s["ws_bwd"])
        return s["y"], s["dx"], s["grads"]
    if kind == "rect_train":
        P.monarch_rect_fwd(s["x"], s["L"], s["R"], s["y"], *s["sizes"], s["ws"])
        P.monarch_rect_bwd(s["x"], s["dy"], s["L"], s["R"], s["dx"], s["dL"], s["dR"], s["accumulate"], *s["sizes"],
                           s["ws_bwd"], fwd_workspace=s["ws"])
        return s["y"], s["dx"], s["dL"], s["dR"]
    if kind == "cplx":
        P.monarch_cplx_fwd(s["x"], s["L"], s["R"], s["y"], 0, *s["sizes"], s["ws"])
        P.monarch_cplx_fwd(s["y"], s["L"], s["R"], s["z"], 1, *s["sizes"], s["ws"])
        return s["y"], s["z"]
    # The factors are unique only up to the sign of each rank-1 pair; the matrix that they stand for is unique.
    P.monarch_project(s["A"], s["L"], s["R"], *s["sizes"])
    P.monarch_dense(s["L"], s["R"], s["M"], *s["sizes"])
    return s["M"]


def work(case):
    kind, e = case["kind"], DTYPES[case["dtype"]][2]
    if kind == "rect_train":
        q, b1, b, r, t = (case[k] for k in ("q", "b1", "b", "r", "tokens"))
        weights = q * b * b1 + b * r * q
        return {"bytes": e * (2 * t * (q * b1 + r * b) + weights) + 4 * weights, "flops": 6 * t * weights}
    m = case["m"]
    n, w = m * m, 2 * m ** 3
    if kind == "project":
        # leading singular pair of m * m slices: no fewer than one pass over a slice for u and one for v
        return {"bytes": e * (2 * n * n + 2 * w), "flops": 4 * n * n}
    t = case["tokens"]
    act, flops = e * t * n, 2 * t * w
    grads = w * (8 if case.get("accumulate") else 4)
    if kind == "fwd":
        return {"bytes": 2 * act + e * w, "flops": flops}
    if kind == "train":
        return {"bytes": 4 * act + e * w + grads, "flops": 3 * flops}
    if kind == "mlp":
        return {"bytes": 2 * act + e * (2 * w + 2 * n), "flops": 2 * flops}
    if kind == "mlp_train":
        return {"bytes": 4 * act + e * (2 * w + 2 * n) + 8 * w + 8 * n, "flops": 6 * flops}
    return {"bytes": 6 * act + 2 * e * w, "flops": 8 * flops}


def tolerance(case):
    """bf16: inputs, intermediates and outputs are rounded to 8 bits once each.  fp32: sums of 32-bit products; the
    projection stops at a cosine of 2e-6 between the columns of a slice."""
    if case["dtype"] == "bf16":
        return {"rel": 1e-2}
    return {"rel": 5e-5} if case["kind"] == "project" else {"rel": 1e-5}
