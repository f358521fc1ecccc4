"""The products this framework is used for, as cases that can be timed and compared.

A case is one call (or one training step) through the public entry points, on a
plan that the program made once and keeps:

  plan    ``Plan.run``: C = op(A) op(B), both operands new on every call
  reuse   ``Plan.quantize_pack(A)`` + ``Plan.gemm``: a fixed right operand packed
          once (inference with fixed weights), a new left operand on every call
  layer   ``tdg_matmul`` forward and both adjoints of one layer
  mlp     one training step of a 128-1024-1024-10 tanh MLP (loss and gradients)

Sizes, block lengths, packings, targets and input families are those of the
repository's benchmark, tests and application studies.  ``draw`` spreads the same
kinds over their whole range of sizes, odd ones among them.
"""
from __future__ import annotations

import math

import torch

from paper_1110_5765_gb300 import Plan
from paper_1110_5765_gb300.autograd import tdg_matmul

MLP_DIMS = (128, 1024, 1024, 10)


def _plan(name, M, N, K, form, *, W=1, dtype="f32", L=128, bits=0, target=0.0, transA="N",
          transB="N", source="uniform", kind="plan"):
    case = {"kind": kind, "M": M, "N": N, "K": K, "form": form, "W": W, "dtype": dtype, "L": L,
            "bits": bits, "target": target, "transA": transA, "transB": transB,
            "source": source}
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the single small product: 64-blocks, 8-bit companders; latency and launches
        _plan("single_256_f64", 256, 256, 256, "sym", W=2, dtype="f64", L=64, bits=8,
              source="gaussian"),
        # an ordinary ragged call, rows of C and B that are no multiple of 16 bytes
        _plan("ragged_f32_asym", 1000, 777, 1531, "asym", W=2, target=20.0),
        # the distortion sweep's fp32 point (the benchmark's workload) ...
        _plan("sweep_4096_f32_sym", 4096, 4096, 4096, "sym", W=2, target=20.0),
        # ... and its fp64 point
        _plan("sweep_4096_f64_sym", 4096, 4096, 4096, "sym", W=3, dtype="f64", target=40.0),
        # eigenface study: X^T X of 10304 pixels x 4096 images, then the images on 400 columns
        _plan("eigen_cov_tc_int", 4096, 4096, 10304, "tc_int", target=30.0, transA="T",
              source="pixels"),
        _plan("eigen_proj_f64_sym", 4096, 400, 10304, "sym", W=3, dtype="f64", target=30.0,
              transA="T", source="pixels"),
        # 2DPCA study: few output tiles over many slabs
        _plan("pca2d_cov_f32_sym", 288, 288, 21600, "sym", W=2, target=20.0, transB="T",
              source="pixels"),
        # inference with fixed weights: the left operand alone is packed per call
        _plan("infer_4096_tc_fp8", 4096, 1024, 1024, "tc_fp8", source="gaussian", kind="reuse"),
        # training: one layer's product with both adjoints, and a whole step
        _plan("layer_4096x1024_f32", 4096, 1024, 1024, "sym", W=2, target=20.0,
              source="gaussian", kind="layer"),
        {"name": "mlp_step_4096", "kind": "mlp", "M": 4096, "target": 20.0},
        # the precision form: the largest products, on tensor cores
        _plan("precision_8192_tc_int", 8192, 8192, 8192, "tc_int", target=40.0,
              source="laplace"),
        _plan("precision_8192_tc_fp8", 8192, 8192, 8192, "tc_fp8", source="laplace"),
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi]; about half of them odd."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.5:
        v = v // 16 * 16
    return max(lo, min(hi, v))


def draw(rng):
    what = rng.choice(("f32", "f32", "f64", "tc_int", "tc_fp8", "reuse", "layer", "mlp"))
    source = rng.choice(("uniform", "gaussian", "laplace"))
    tA, tB = rng.choice("NNT"), rng.choice("NNT")
    if what == "mlp":
        return {"kind": "mlp", "M": _size(rng, 256, 4096), "target": 20.0}
    if what == "layer":
        return _plan(None, _size(rng, 256, 4096), _size(rng, 128, 2048), _size(rng, 128, 2048),
                     "sym", W=2, target=20.0, source="gaussian", kind="layer")
    if what == "reuse":
        form, W, bits = rng.choice((("tc_fp8", 1, 0), ("tc_int", 1, 8), ("sym", 2, 6)))
        return _plan(None, _size(rng, 128, 4096), _size(rng, 128, 4096), _size(rng, 128, 4096),
                     form, W=W, bits=bits, source="gaussian", kind="reuse")
    if what == "f64":
        W = rng.choice((2, 3))
        bits = rng.choice((0, 8))
        return _plan(None, _size(rng, 64, 2048), _size(rng, 64, 2048), _size(rng, 64, 4096),
                     rng.choice(("sym", "sym", "asym")), W=W if not bits else 2, dtype="f64",
                     L=rng.choice((64, 128)), bits=bits, target=0.0 if bits else 40.0,
                     transA=tA, transB=tB, source=source)
    if what == "f32":
        return _plan(None, _size(rng, 64, 4096), _size(rng, 64, 4096), _size(rng, 64, 8192),
                     rng.choice(("sym", "sym", "asym")), W=2, target=20.0, transA=tA, transB=tB,
                     source=rng.choice(("uniform", "pixels")))
    bits = rng.choice((0, 8)) if what == "tc_int" else 0
    return _plan(None, _size(rng, 128, 8192), _size(rng, 128, 8192), _size(rng, 128, 8192), what,
                 bits=bits, target=30.0 if what == "tc_int" and not bits else 0.0, transA=tA,
                 transB=tB, source=source)


# ------------------------------------------------------------------ inputs
def _matrix(rows, cols, source, dtype, gen):
    if source == "gaussian":
        x = torch.randn(rows, cols, generator=gen, device="cuda")
    elif source == "pixels":     # integers 0..255 with each row's mean removed
        x = torch.randint(0, 256, (rows, cols), generator=gen, device="cuda").float()
        x -= x.mean(dim=1, keepdim=True)
    else:
        x = torch.rand(rows, cols, generator=gen, device="cuda") * 2 - 1
        if source == "laplace":  # scale 1, by the inverse of its distribution function
            x = -torch.sign(x) * torch.log1p(-x.abs().clamp(max=1 - 2.0 ** -24))
    return x.to(torch.float64) if dtype == "f64" else x


def _operands(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    M, N, K = case["M"], case["N"], case["K"]
    A = _matrix(*((M, K) if case["transA"] == "N" else (K, M)), case["source"], case["dtype"], gen)
    B = _matrix(*((K, N) if case["transB"] == "N" else (N, K)), case["source"], case["dtype"], gen)
    return A, B, gen


def _mlp_inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(case["M"], MLP_DIMS[0], generator=gen, device="cuda")
    labels = torch.randint(0, MLP_DIMS[-1], (case["M"],), generator=gen, device="cuda")
    weights = [torch.randn(i, o, generator=gen, device="cuda") / math.sqrt(i)
               for i, o in zip(MLP_DIMS[:-1], MLP_DIMS[1:])]
    return X, labels, weights


def prepare(case, seed):
    state = {"kind": case["kind"]}
    if case["kind"] == "mlp":
        X, labels, weights = _mlp_inputs(case, seed)
        state.update(X=X, labels=labels, weights=[w.requires_grad_() for w in weights],
                     opts=dict(L=128, W=2, form="sym", target_snr_db=case["target"]))
        return state
    A, B, gen = _operands(case, seed)
    if case["kind"] == "layer":
        G = torch.randn(case["M"], case["N"], generator=gen, device="cuda")
        state.update(A=A.requires_grad_(), B=B.requires_grad_(), G=G,
                     opts=dict(L=case["L"], W=case["W"], form=case["form"],
                               target_snr_db=case["target"]))
        return state
    goal = dict(bits=case["bits"]) if case["bits"] else {}
    if case["target"]:
        goal = dict(target_snr_db=case["target"])
    plan = Plan(case["M"], case["N"], case["K"], L=case["L"], W=case["W"], dtype=case["dtype"],
                form=case["form"], transA=case["transA"], transB=case["transB"], **goal)
    C = torch.empty(case["M"], case["N"], dtype=A.dtype, device="cuda")
    if case["kind"] == "reuse":
        plan.quantize_pack(A, B)      # the weights are packed once
        A = _matrix(*A.shape, case["source"], case["dtype"], gen)
    state.update(plan=plan, A=A, B=B, C=C)
    return state


# ------------------------------------------------------------------ one pass
def run(state):
    kind = state["kind"]
    if kind == "plan":
        return state["plan"].run(state["A"], state["B"], state["C"])
    if kind == "reuse":
        state["plan"].quantize_pack(state["A"])
        return state["plan"].gemm(state["C"])
    if kind == "layer":
        C = tdg_matmul(state["A"], state["B"], **state["opts"])
        dA, dB = torch.autograd.grad(C, (state["A"], state["B"]), state["G"])
        return {"C": C.detach(), "dA": dA, "dB": dB}
    logits = _mlp(state["X"], state["weights"], lambda a, b: tdg_matmul(a, b, **state["opts"]))
    loss = torch.nn.functional.cross_entropy(logits, state["labels"])
    grads = torch.autograd.grad(loss, state["weights"])
    return {"logits": logits.detach(), "grads": list(grads)}


def _mlp(X, weights, matmul):
    h = X
    for k, w in enumerate(weights):
        h = matmul(h, w)
        if k + 1 < len(weights):
            h = torch.tanh(h)
    return h


# ------------------------------------------------------------------ what it takes, and how exact it is
def work(case):
    if case["kind"] == "mlp":
        n, flops, values = case["M"], 0, case["M"] * (MLP_DIMS[0] + MLP_DIMS[-1])
        for k, (i, o) in enumerate(zip(MLP_DIMS[:-1], MLP_DIMS[1:])):
            flops += 2 * n * i * o * (3 if k else 2)     # forward, dW and, but for X, dX
            values += 2 * i * o                          # weights in, gradients out
        return {"bytes": 4 * values, "flops": flops}
    M, N, K = case["M"], case["N"], case["K"]
    size = 8 if case["dtype"] == "f64" else 4
    if case["kind"] == "layer":
        return {"bytes": 2 * size * (M * K + K * N + M * N), "flops": 6 * M * N * K}
    right = 0 if case["kind"] == "reuse" else K * N      # the kept operand is not read again
    return {"bytes": size * (M * K + right + M * N), "flops": 2 * M * N * K}


def tolerance(case):
    """Of the result that the same companders and packing give.  The running sums over
    the slabs taken in another order differ by up to 3.0e-7 (fp32, 169 slabs) and 3.9e-16
    (fp64), at most 1.7e-6 and 2.4e-15 of a value; four times that.  The training step:
    inputs moved by 1e-7 move the gradients by up to 3.0e-3, since a value that rounds to
    another integer changes the packed sums of its row."""
    if case["kind"] == "mlp":
        return {"rel": 1.2e-2, "max": 0.15}
    if case["dtype"] == "f64":
        return {"rel": 2e-15, "max": 1e-14}
    return {"rel": 1.2e-6, "max": 8e-6}


def exact(case, seed):
    if case["kind"] == "mlp":
        # companding noise of up to five products in a row (20 dB targets): about a
        # tenth of the gradients, so 64 bits say nothing of the step's arithmetic;
        # the layer cases hold its products one by one
        return None
    A, B, gen = _operands(case, seed)
    if case["kind"] == "layer":
        G = torch.randn(case["M"], case["N"], generator=gen, device="cuda").double()
        A, B = A.double(), B.double()
        return {"C": A @ B, "dA": G @ B.t(), "dB": A.t() @ G}
    if case["kind"] == "reuse":
        A = _matrix(*A.shape, case["source"], case["dtype"], gen)
    a = A.double() if case["transA"] == "N" else A.double().t()
    b = B.double() if case["transB"] == "N" else B.double().t()
    return a @ b
