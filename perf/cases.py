"""The work that programs built on this library have it do, as cases that can be timed and compared.

A case is one pass through the public Python entry points at one size.  What a pass is, by its "op":

    quant           rotate activation rows and quantize each to low-bit codes (Plan.forward_quant): the online step of
                    a low-bit model, one call for each linear layer's input
    inverse         x = Q^T y (Plan.inverse): rotated rows back in the original basis
    linear          a quantized linear layer from end to end: rotate (and quantize) the token rows, then the product with
                    the folded weight's codes (Plan.forward or forward_quant, then dequant_gemm)
    learn           one step of learning the angles: new angles, rotated rows, dL/dx and dL/dtheta
                    (Plan.set_angles, forward, backward)
    fold            one weight matrix through newly set angles: W Q^T as codes (Plan.set_angles, fold_weights)
    composite       activation rows whose length n1 * n2 is no power of two, to codes (Plan.composite_forward_quant)
    composite_learn one learning step of both factors of such a rotation (cayley, composite_forward, composite_backward)
    calibrate       one step of layer-wise calibration: loss, gradient and update (LayerCalibrator)

Rows and tokens go from a single decoded token to the batches of a calibration run.  Rows that start in host memory are
bound by the link to the host and are not timed here.
"""
from __future__ import annotations

import math

import torch

from paper_2509_09679_b200 import GemmOperand, Plan, synth
from paper_2509_09679_b200.calibrate import LayerCalibrator
from paper_2509_09679_b200.composite import composite_backward

DEVICE = "cuda"


def listed():
    return [
        # the smallest call: the tiny fp32 configuration, where launching is most of the time
        dict(name="quant_n256_f32_tiny", op="quant", n=256, rows=1024, dtype="f32", bits=4),
        # one decoded token through a weight-only 2-bit layer
        dict(name="linear_decode_w2a16", op="linear", n=4096, out=4096, rows=1, wbits=2, abits=0),
        # an uneven prefill batch through the widest 2-bit layer of the 8192-wide shape
        dict(name="linear_prefill_w2a16_n8192", op="linear", n=8192, out=28672, rows=1000, wbits=2, abits=0),
        # prefill activations of the 4096-wide shape to INT4 (16 x 2048 tokens)
        dict(name="quant_n4096_prefill_int4", op="quant", n=4096, rows=32768, dtype="bf16", bits=4),
        # prefill activations of the 8192-wide shape to INT2
        dict(name="quant_n8192_prefill_int2", op="quant", n=8192, rows=65536, dtype="bf16", bits=2),
        # rotated rows of a narrower layer back to the original basis, an odd number of them
        dict(name="inverse_n2048_odd_rows", op="inverse", n=2048, rows=20011, dtype="bf16"),
        # the largest: an angle-learning step on 128 sequences x 2048 tokens
        dict(name="learn_n4096_full", op="learn", n=4096, rows=262144, dtype="bf16"),
        # the same step for a small fp32 layer, odd rows
        dict(name="learn_n1024_f32_odd_rows", op="learn", n=1024, rows=9973, dtype="f32"),
        # a 28672 x 8192 weight folded to 2 bits after the angles changed
        dict(name="fold_n8192_int2", op="fold", n=8192, rows=28672, dtype="bf16", bits=2, keep=False),
        # 5120-wide activations (40 x 128) to INT4
        dict(name="composite_d5120_int4", op="composite", n1=40, n=128, rows=32768, dtype="bf16", bits=4),
        # one learning step of both factors of the 40 x 128 rotation on one 2048-token sequence
        dict(name="composite_learn_d5120", op="composite_learn", n1=40, n=128, rows=2048, dtype="bf16"),
        # one calibration step of a square W4A4 layer on 2048 tokens
        dict(name="calibrate_n4096_w4a4", op="calibrate", n=4096, out=4096, rows=2048, dtype="bf16", wbits=4, abits=4),
    ]


def _log_int(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# rows * n of the largest batch each op is given at one call: as in the largest listed case of that op
_MOST = dict(quant=1 << 27, inverse=1 << 27, learn=1 << 26, fold=1 << 27, composite=1 << 27, composite_learn=1 << 24)


def draw(rng):
    op = rng.choice(["quant", "quant", "linear", "linear", "inverse", "learn", "fold", "composite", "composite_learn", "calibrate"])
    dtype = rng.choice(["bf16", "bf16", "f32"])
    bits = rng.choice([2, 4, 8])
    if op in ("quant", "inverse", "learn", "fold"):
        n = rng.choice([128, 256, 512, 1024, 2048, 4096, 4096, 8192])
        case = dict(op=op, n=n, rows=_log_int(rng, 64 if op in ("learn", "fold") else 1, _MOST[op] // n), dtype=dtype)
        if op in ("quant", "fold"):
            case["bits"] = bits
        if op == "fold":
            case["keep"] = rng.random() < 0.25
        return case
    if op == "linear":
        n = rng.choice([1024, 2048, 4096, 8192])
        out = 4 * _log_int(rng, 128, 4096)
        return dict(op=op, n=n, out=out, rows=_log_int(rng, 1, 4096), wbits=bits, abits=rng.choice([0, 4, 8]))
    if op == "calibrate":  # the dense products take K blocks of 64; angles are learned where codes are few
        n = rng.choice([512, 1024, 2048, 4096])
        return dict(op=op, n=n, out=64 * _log_int(rng, 4, 64), rows=64 * _log_int(rng, 2, 32), dtype=dtype, wbits=min(bits, 4),
                    abits=rng.choice([0, 4, 8]))
    n1, n2 = rng.choice([(40, 128), (40, 128), (12, 256), (7, 1024)])
    case = dict(op=op, n1=n1, n=n2, rows=_log_int(rng, 1 if op == "composite" else 64, _MOST[op] // (n1 * n2)), dtype=dtype)
    if op == "composite":
        case["bits"] = bits
    return case


def _dtype(case):
    return torch.float32 if case.get("dtype", "bf16") == "f32" else torch.bfloat16


def _activations(rows, n, seed, dtype):
    """Heavy-tailed rows with a few outlier channels."""
    return synth.rows(rows, n, "student_t3", seed, outliers=8, outlier_scale=50.0, dtype=dtype, device=DEVICE)


def _weights(rows, n, seed, dtype):
    return synth.rows(rows, n, "normal", seed, scale=0.02, dtype=dtype, device=DEVICE)


def prepare(case, seed):
    op, n, rows, dtype = case["op"], case["n"], case["rows"], _dtype(case)
    seed = 16 * int(seed)
    theta = synth.angles(n, "normal", seed, DEVICE)
    s = dict(case=case, theta=theta)
    if op == "calibrate":
        s["cal"] = LayerCalibrator(_weights(case["out"], n, seed + 1, dtype), case["wbits"], case["abits"] or None, theta)
        s["x"] = _activations(rows, n, seed + 2, dtype)
        return s
    s["plan"] = Plan(n, DEVICE)
    s["plan"].set_angles(theta)
    if op == "linear":
        codes, scales, _ = s["plan"].fold_weights(_weights(case["out"], n, seed + 1, torch.bfloat16), case["wbits"])
        s["weight"] = GemmOperand(codes, scales, case["wbits"])
        s["x"] = _activations(rows, n, seed + 2, torch.bfloat16)
    elif op == "fold":
        s["x"] = _weights(rows, n, seed + 1, dtype)
    elif op in ("composite", "composite_learn"):
        s["params"] = synth.cayley_params(case["n1"], seed + 1, device=DEVICE)
        s["q1"] = s["plan"].cayley(s["params"], case["n1"])
        s["x"] = _activations(rows, case["n1"] * n, seed + 2, dtype)
        if op == "composite_learn":
            s["g"] = synth.rows(rows, case["n1"] * n, "normal", seed + 3, dtype=dtype, device=DEVICE)
    else:
        s["x"] = _activations(rows, n, seed + 2, dtype)
        if op == "learn":
            s["g"] = synth.rows(rows, n, "normal", seed + 3, dtype=dtype, device=DEVICE)
    return s


def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "calibrate":
        cal = state["cal"]
        loss, grad = cal.loss_and_grad(state["x"])
        cal.step(grad, 0.0)  # the end of the cosine schedule: the update runs and leaves the angles where they are
        return loss, grad, cal.theta
    plan, x = state["plan"], state["x"]
    if op == "quant":
        return plan.forward_quant(x, case["bits"])
    if op == "inverse":
        return plan.inverse(x)
    if op == "linear":
        if case["abits"] == 0:
            return plan.dequant_gemm(GemmOperand(plan.forward(x)), state["weight"])
        codes, scales = plan.forward_quant(x, case["abits"])
        return plan.dequant_gemm(GemmOperand(codes, scales, case["abits"]), state["weight"])
    if op == "learn":
        plan.set_angles(state["theta"])
        y = plan.forward(x)
        return y, *plan.backward(x, state["g"])
    if op == "fold":
        plan.set_angles(state["theta"])
        return plan.fold_weights(x, case["bits"], want_rotated=case["keep"])
    if op == "composite":
        return plan.composite_forward_quant(state["q1"], x, case["bits"])
    plan.set_angles(state["theta"])
    q1 = plan.cayley(state["params"], case["n1"])
    y = plan.composite_forward(q1, x)
    return y, *composite_backward(plan, q1, state["params"], x, state["g"])


def work(case):
    op, n, rows = case["op"], case["n"], case["rows"]
    size = 4 if case.get("dtype", "bf16") == "f32" else 2
    levels = n.bit_length() - 1
    rotation = 3 * n * levels  # flops of one row through Q: 3 n log2 n
    angles = 4 * levels * n // 2
    if op == "quant":
        return dict(bytes=rows * (n * size + n * case["bits"] / 8 + 2) + angles, flops=rows * rotation)
    if op == "inverse":
        return dict(bytes=rows * 2 * n * size + angles, flops=rows * rotation)
    if op == "linear":
        out = case["out"]
        return dict(bytes=rows * n * 2 + out * (n * case["wbits"] / 8 + 2) + rows * out * 4 + angles,
                    flops=rows * rotation + 2 * rows * n * out)
    if op == "learn":  # x and g read, y and dx written; y, both walks down and one product pair for each angle
        return dict(bytes=rows * 4 * n * size + 2 * angles, flops=rows * (3 * rotation + 2 * n * levels))
    if op == "fold":
        return dict(bytes=rows * (n * size + n * case["bits"] / 8 + 2 + (n * size if case["keep"] else 0)) + angles,
                    flops=rows * rotation)
    if op == "calibrate":  # the target, the quantized product, two gradient products; rotations and gradients of x and W
        out = case["out"]
        return dict(bytes=(rows + out) * n * size + 2 * angles + 4,
                    flops=8 * rows * n * out + (rows + out) * (3 * rotation + 2 * n * levels))
    n1 = case["n1"]
    d, dense = n1 * n, 2 * n1 * n1 * n
    if op == "composite":
        return dict(bytes=rows * (d * size + d * case["bits"] / 8 + 2) + angles + 4 * n1 * n1,
                    flops=rows * (n1 * rotation + dense))
    return dict(bytes=rows * 4 * d * size + 2 * angles + 4 * n1 * n1,
                flops=rows * (n1 * (3 * rotation + 2 * n * levels) + 3 * dense))


def tolerance(case):
    """From each op against the same op in float64, over the listed cases and sixty drawn ones: about four times the
    largest error seen."""
    op, bf16 = case["op"], case.get("dtype", "bf16") == "bf16"
    if op in ("quant", "fold"):  # fp32 sums: an fp16 scale may round the other way (one part in 1024), a code in 1e6 too
        if case.get("keep") and bf16:
            return {"rel": 7e-3, "max": 2e-2, "differ": 2e-4}
        return {"rel": 1e-3, "max": 2e-3, "differ": 2e-4}
    if op == "linear":  # rows rounded to bf16 before the product: 1.7e-3; a scale that rounds the other way: 8e-5, max 7e-3
        return {"rel": 1e-3, "max": 3e-2} if case["abits"] else {"rel": 7e-3, "max": 1.2e-1}
    if op in ("inverse", "learn"):  # one rounding of the results to bf16: 1.7e-3; fp32 throughout: 2.7e-7
        return {"rel": 7e-3, "max": 2e-2} if bf16 else {"rel": 1.2e-6, "max": 1.4e-5}
    if op == "calibrate":  # gradients rounded to bf16 and summed with much cancellation: 1.3e-2; in fp32 only codes that
        return {"rel": 3e-2, "max": 6e-1} if bf16 else {"rel": 2.5e-2, "max": 5e-1}  # round the other way: 7e-3
    if op == "composite":
        if bf16 and case["n1"] == 40:  # tensor-core factors, bf16 and tf32 terms: codes shift by the error over their step
            return {"rel": 2e-3, "max": 7e-3, "differ": {2: 2e-4, 4: 3.5e-3, 8: 1e-2}[case["bits"]]}
        return {"rel": 1e-3, "max": 2e-3, "differ": 2e-4}
    return {"rel": 9e-3, "max": 4e-2} if bf16 else {"rel": 7e-6, "max": 2.2e-5}


# ---- the same passes in 64 bits, in plain torch ----------------------------------------------------------------------
_CHUNK = 1 << 26  # elements of the rows that are worked on at a time


def _stages(theta):
    """(cos, sin) of each stage's pairs."""
    t = theta.double()
    return list(zip(torch.cos(t), torch.sin(t)))


def _turn(x, stage, s, back=False):
    """Stage s (pairs at distance 2^s) on the last axis of x, or its transpose."""
    d = 1 << s
    c, sn = (v.view(-1, d) for v in stage)
    if back:
        sn = -sn
    v = x.reshape(*x.shape[:-1], -1, 2, d)
    lo, hi = v[..., 0, :], v[..., 1, :]
    return torch.stack((c * lo - sn * hi, sn * lo + c * hi), dim=-2).reshape(x.shape)


def _rotate(theta, x, back=False):
    stages = _stages(theta)
    x = x.double()
    for s in (range(len(stages) - 1, -1, -1) if back else range(len(stages))):
        x = _turn(x, stages[s], s, back)
    return x


def _gradients(theta, x, g):
    """(y, dx, dtheta): y = Q x, and the gradients of <g, y>."""
    stages = _stages(theta)
    y, g, dth = _rotate(theta, x), g.double(), []
    z = y
    for s in range(len(stages) - 1, -1, -1):
        u, w = (t.reshape(t.shape[0], -1, 2, 1 << s) for t in (z, g))
        dth.append((w[:, :, 1] * u[:, :, 0] - w[:, :, 0] * u[:, :, 1]).sum(0).reshape(-1))
        z, g = _turn(z, stages[s], s, True), _turn(g, stages[s], s, True)
    return y, g, torch.stack(dth[::-1])


def _chunks(rows, width):
    step = max(1, _CHUNK // width)
    return [slice(r, min(rows, r + step)) for r in range(0, rows, step)]


def _scales(y, bits):
    return y.abs().amax(dim=1) / (2 ** (bits - 1) - 1)


def _quantized(y, bits):
    """Rows through codes and 16-bit scales and back."""
    s = _scales(y, bits).half().double().unsqueeze(1)
    q = torch.where(s > 0, y / s, torch.zeros_like(y)).round().clamp(-(2 ** (bits - 1)), 2 ** (bits - 1) - 1)
    return q * s


def _cayley(params, n1):
    i, j = torch.triu_indices(n1, n1, 1, device=params.device)
    a = torch.zeros((n1, n1), dtype=torch.float64, device=params.device)
    a[i, j] = params.double()
    a = a - a.t()
    eye = torch.eye(n1, dtype=torch.float64, device=params.device)
    inv = torch.linalg.inv(eye + a)
    return (eye - a) @ inv, inv


def exact(case, seed):
    """What run() returns, in 64 bits: scales before their rounding to 16, None in the place of codes."""
    op, n, rows, dtype = case["op"], case["n"], case["rows"], _dtype(case)
    seed = 16 * int(seed)
    theta = synth.angles(n, "normal", seed, DEVICE)
    if op in ("quant", "inverse"):
        x = _activations(rows, n, seed + 2, dtype)
        if op == "quant":
            return None, torch.cat([_scales(_rotate(theta, x[c]), case["bits"]) for c in _chunks(rows, n)])
        return torch.cat([_rotate(theta, x[c], back=True) for c in _chunks(rows, n)])
    if op == "fold":
        w = _weights(rows, n, seed + 1, dtype)
        parts = [_rotate(theta, w[c]) for c in _chunks(rows, n)]
        return None, torch.cat([_scales(y, case["bits"]) for y in parts]), torch.cat(parts) if case["keep"] else None
    if op == "learn":
        x, g = _activations(rows, n, seed + 2, dtype), synth.rows(rows, n, "normal", seed + 3, dtype=dtype, device=DEVICE)
        y, dx = (torch.empty((rows, n), dtype=torch.float64, device=DEVICE) for _ in range(2))
        dth = 0
        for c in _chunks(rows, n):
            y[c], dx[c], part = _gradients(theta, x[c], g[c])
            dth = dth + part
        return y, dx, dth
    if op == "linear":
        w = _quantized(_rotate(theta, _weights(case["out"], n, seed + 1, torch.bfloat16)), case["wbits"])
        y = _rotate(theta, _activations(rows, n, seed + 2, torch.bfloat16))
        return (_quantized(y, case["abits"]) if case["abits"] else y) @ w.t()
    if op == "calibrate":
        w, x = _weights(case["out"], n, seed + 1, dtype).double(), _activations(rows, n, seed + 2, dtype).double()
        wq, y = _quantized(_rotate(theta, w), case["wbits"]), _rotate(theta, x)
        yq = _quantized(y, case["abits"]) if case["abits"] else y
        err = yq @ wq.t() - x @ w.t()
        e = err * (2.0 / err.numel())
        return (err * err).mean(), _gradients(theta, x, e @ wq)[2] + _gradients(theta, w, e.t() @ yq)[2], theta.double()
    n1 = case["n1"]
    params = synth.cayley_params(n1, seed + 1, device=DEVICE)
    q1, inv = _cayley(params, n1)
    x = _activations(rows, n1 * n, seed + 2, dtype)
    if op == "composite":
        return None, torch.cat([_scales(torch.einsum("ik,rkj->rij", q1, _rotate(theta, x[c].reshape(-1, n1, n))).flatten(1),
                                        case["bits"]) for c in _chunks(rows, n1 * n)])
    g = synth.rows(rows, n1 * n, "normal", seed + 3, dtype=dtype, device=DEVICE).double().reshape(rows, n1, n)
    gp = torch.einsum("ki,rkj->rij", q1, g)
    xp, dx, dth = _gradients(theta, x.reshape(-1, n), gp.reshape(-1, n))
    xp = xp.reshape(rows, n1, n)
    dq1 = torch.einsum("rij,rkj->ik", g, xp)
    da = -(torch.eye(n1, dtype=torch.float64, device=DEVICE) + q1).t() @ dq1 @ inv.t()
    i, j = torch.triu_indices(n1, n1, 1, device=DEVICE)
    return torch.einsum("ik,rkj->rij", q1, xp).flatten(1), dx.reshape(rows, -1), dth, dq1, (da - da.t())[i, j]
