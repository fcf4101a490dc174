"""Workloads of the library's public entry points, for timing one revision against another.

A training step with this library is: the INT8 linear layers forward and backward (App. A), the optimizer step of
every weight matrix (Sec. 3.5), and, every interval of steps, the subspace refresh of the matrices that are due
(Sec. 3.2, 3.3, 3.5).  Around it stand the quantizer calls that bring weights and projections in and out.  The cases
below take those calls over the layer shapes of the LLaMA stacks of ``synth.STACKS`` and over generic sizes between
them; gradients are the rank-32 signal plus Gaussian noise of ``synth.GradientModel``, drawn on the device.

    listed()          the named cases
    draw(rng)         one more case of the same ranges
    prepare(case, s)  what a training program holds before the call, made from the seed s
    run(state)        one pass; returns everything the path writes
    work(case)        bytes and flops one pass cannot do without
    tolerance(case)   how far another correct implementation's outputs may be off
"""
import math

import torch

from paper_2407_08296_b200 import binding as B
from paper_2407_08296_b200 import synth

REFRESH_ITERS = 12          # the refresh's documented setting: 12 iterations, a block of 2 r columns
LATE_LR = 4e-4              # a tenth of the default: where a decaying schedule is when refreshes have become rare
START_STEP = 1000           # optimizer steps already taken: bias corrections and moments as in mid-training


def listed():
    return [
        # One matrix of the LLaMA-60M MLP stepped by a call of its own, as a fused backward hook does: the smallest call,
        # where launches and host work are what there is.
        {"name": "step_60m_mlp", "kind": "step", "m": 512, "n": 1376, "r": 128, "moments": 32, "side": "left"},
        # One LLaMA-1B MLP matrix the same way: taller than wide, projected on its shorter (right-hand) side.
        {"name": "step_1b_down", "kind": "step", "m": 5461, "n": 2048, "r": 512, "moments": 32, "side": "right"},
        # The whole LLaMA-130M stack as a plan: an ordinary step of a small model, a quarter of a millisecond.
        {"name": "plan_130m", "kind": "plan", "hidden": 768, "mlp": 2048, "layers": 12, "r": 256, "moments": 32, "side": "left"},
        # LLaMA-350M with 8-bit moments, every matrix projected on its shorter side (GaLore's rule): the memory-saving setting.
        {"name": "plan_350m_8bit", "kind": "plan", "hidden": 1024, "mlp": 2736, "layers": 24, "r": 256, "moments": 8, "side": "short"},
        # The whole LLaMA-1B stack, the library's headline step: ragged 5461-wide rows, 10 GB moved.
        {"name": "plan_1b", "kind": "plan", "hidden": 2048, "mlp": 5461, "layers": 24, "r": 512, "moments": 32, "side": "left"},
        # Four LLaMA-7B layers, one GPU's share of the stack when its matrices are spread over eight: rank 1024.
        {"name": "plan_7b_4layers", "kind": "plan", "hidden": 4096, "mlp": 11008, "layers": 4, "r": 1024, "moments": 32, "side": "left"},
        # One LLaMA-130M matrix whose interval has run out under the adaptive schedule (refresh, similarity for the gate, step
        # on the new projection): bound by latency.
        {"name": "refresh_130m_1", "kind": "refresh", "m": 768, "n": 2048, "r": 256, "count": 1, "side": "left"},
        # Eight LLaMA-1B MLP matrices due in the same step, refreshed and stepped in one batched call each.
        {"name": "refresh_1b_8", "kind": "refresh", "m": 2048, "n": 5461, "r": 512, "count": 8, "side": "left"},
        # A training batch through one LLaMA-1B down projection (K = 5461 is ragged).
        {"name": "forward_1b_8192", "kind": "forward", "tokens": 8192, "m": 2048, "n": 5461},
        # A few tokens through a LLaMA-7B MLP weight: sampling from the model being trained.  Bound by the weight's bytes.
        {"name": "forward_7b_8", "kind": "forward", "tokens": 8, "m": 11008, "n": 4096},
        # Both gradients of a LLaMA-7B MLP matrix for an odd number of tokens (packed sequences).
        {"name": "backward_7b_3001", "kind": "backward", "tokens": 3001, "m": 11008, "n": 4096},
        # A weight brought in (Quant_8) and read back in fp32, as loading and exporting a checkpoint do.
        {"name": "quantize_7b", "kind": "quantize", "bits": 8, "m": 4096, "n": 11008},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds of ``listed``, sizes over their whole range (log-uniform, odd ones included)."""
    kind = rng.choice(["step", "plan", "refresh", "forward", "backward", "quantize"])
    if kind == "step":
        m, n = _log_int(rng, 256, 11008), _log_int(rng, 256, 11008)
        side = rng.choice(["left", "left", "right"])
        return {"kind": kind, "m": m, "n": n, "r": _rank(rng, n if side == "right" else m, min(m, n)), "moments": rng.choice([32, 32, 8]), "side": side}
    if kind == "plan":
        hidden = _log_int(rng, 256, 4096)
        mlp = hidden * 8 // 3 + rng.randint(-5, 5)
        per_layer = 4 * hidden * hidden + 3 * hidden * mlp
        most = min(32, max(1, 800_000_000 // per_layer))         # no more elements than the listed stacks hold
        return {"kind": kind, "hidden": hidden, "mlp": mlp, "layers": _log_int(rng, 1, most), "r": _rank(rng, hidden, hidden),
                "moments": rng.choice([32, 32, 8]), "side": rng.choice(["left", "short"])}
    if kind == "refresh":
        short = _log_int(rng, 256, 4096)
        long = min(11008, int(short * rng.choice([1.0, rng.uniform(1.0, 2.7), 8 / 3])))
        m, n = (short, long) if rng.random() < 0.6 else (long, short)
        case = {"kind": kind, "m": m, "n": n, "r": _rank(rng, short, short), "count": rng.choice([1, 1, 2, 4, 8]),
                "side": "right" if m > n and rng.random() < 0.5 else "left"}
        while case["count"] > 1 and work(case)["flops"] > 5e12:
            case["count"] //= 2
        return case
    if kind in ("forward", "backward"):
        m, n = _log_int(rng, 512, 11008), _log_int(rng, 512, 11008)
        most = min(16384, int(1.0e12 / (2.0 * m * n)))
        return {"kind": kind, "tokens": _log_int(rng, 1 if kind == "forward" else 256, max(512, most)), "m": m, "n": n}
    return {"kind": kind, "bits": rng.choice([8, 8, 4]), "m": _log_int(rng, 256, 11008), "n": _log_int(rng, 256, 11008)}


def _rank(rng, rows, short):
    """A multiple of 32 near a quarter of the short side (the rank rule of the stacks), or an eighth."""
    r = short // rng.choice([4, 4, 8]) // 32 * 32
    return max(32, min(r, 1024, rows // 32 * 32))


# ---------------------------------------------------------------------------------------------- inputs
def _gradient(m, n, gen, scale_u=None):
    """bf16 gradient: U diag(1/k) V^T with 32 nearly orthonormal Gaussian columns, plus 1e-3 Gaussian noise."""
    k = min(synth.SIGNAL_RANK, m, n)
    u = torch.randn(m, k, device="cuda", generator=gen) / math.sqrt(m)
    v = torch.randn(n, k, device="cuda", generator=gen) / math.sqrt(n)
    u /= torch.arange(1, k + 1, device="cuda", dtype=torch.float32)
    noise = torch.randn(m, n, device="cuda", generator=gen)
    g = B.zeros_matrix(m, n, torch.bfloat16)
    g.copy_(torch.addmm(noise, u, v.T, beta=synth.NOISE_STD))
    return g


def _gaussian(m, n, std, gen):
    x = B.zeros_matrix(m, n, torch.float32)
    x.copy_(torch.randn(m, n, device="cuda", generator=gen))
    return x.mul_(std)


class _Flat:
    """One allocation per kind of optimizer state, cut into the matrices' pieces (so that it is saved as a whole)."""

    def __init__(self):
        self.wanted = []

    def ask(self, rows, pitch, dtype):
        self.wanted.append((rows, pitch, dtype))
        return len(self.wanted) - 1

    def make(self):
        self.whole, self.parts, used = {}, [], {}
        for rows, pitch, dtype in self.wanted:
            used[dtype] = used.get(dtype, 0) + rows * pitch + (-(rows * pitch)) % 64
        for dtype, count in used.items():
            self.whole[dtype] = torch.zeros(count, dtype=dtype, device="cuda")
        at = {dtype: 0 for dtype in used}
        for rows, pitch, dtype in self.wanted:
            self.parts.append(self.whole[dtype][at[dtype]:at[dtype] + rows * pitch].view(rows, pitch))
            at[dtype] += rows * pitch + (-(rows * pitch)) % 64
        return self


def _items(shapes, r, moments, side, seed, gen):
    """The optimizer state of a list of matrices: gradients, INT8 weights, INT4 projections, moments; with it the whole
    buffers that a step writes, by name."""
    flats = {k: _Flat() for k in ("codes", "scales", "zeros", "M", "V", "M_scale", "V_scale")}
    plan = []
    for m, n in shapes:
        right = side == "right" or (side == "short" and m > n)
        cols = m if right else n
        groups, pitch = (n + B.GROUP - 1) // B.GROUP, B.round_up(cols, 64)
        asked = {"codes": flats["codes"].ask(m, B.round_up(n, 64), torch.int8),
                 "scales": flats["scales"].ask(m, groups, torch.float32), "zeros": flats["zeros"].ask(m, groups, torch.float32)}
        if moments == 8:
            asked["M"] = flats["M"].ask(r, pitch, torch.int8)
            asked["V"] = flats["V"].ask(r, pitch, torch.uint8)
            for k in ("M_scale", "V_scale"):
                asked[k] = flats[k].ask(r, (cols + 31) // 32, torch.float32)
        else:
            asked["M"] = flats["M"].ask(r, pitch, torch.float32)
            asked["V"] = flats["V"].ask(r, pitch, torch.float32)
        plan.append((m, n, right, cols, asked))
    flats = {k: f.make() for k, f in flats.items() if f.wanted}
    items = []
    for i, (m, n, right, cols, asked) in enumerate(plan):
        part = {k: flats[k].parts[v] for k, v in asked.items()}
        w = B.QTensor(part["codes"], part["scales"], part["zeros"], m, n, B.round_up(n, 64), 8)
        B.quantize_int8(_gaussian(m, n, synth.WEIGHT_STD, gen), w)
        # a projection has orthonormal columns; Gaussian ones of the same length have the same entries, at no cost
        rows = n if right else m
        p = B.quantize_int4(_gaussian(rows, r, 1.0 / math.sqrt(rows), gen))
        M, V = part["M"][:, :cols], part["V"][:, :cols]
        # moments of a projected gradient whose noise has standard deviation 1e-3, START_STEP steps into training
        if moments == 8:
            M.copy_(torch.randint(-127, 128, M.shape, device="cuda", generator=gen))
            V.copy_(torch.randint(200, 256, V.shape, device="cuda", generator=gen))
            part["M_scale"].fill_(7e-4)
            part["V_scale"].fill_(1e-6)
        else:
            M.copy_(torch.randn(M.shape, device="cuda", generator=gen)).mul_(2.3e-4)
            V.copy_(torch.rand(V.shape, device="cuda", generator=gen)).mul_(2e-7).add_(5e-7)
        items.append({"G": _gradient(m, n, gen), "P": p, "W": w, "M": M, "V": V, "seed": synth.matrix_seed(seed, i),
                      "side": "right" if right else "left", **{k: part[k] for k in ("M_scale", "V_scale") if k in part}})
    outputs = {"%s.%s" % (k, str(d).rsplit(".", 1)[-1]): t for k, f in flats.items() for d, t in f.whole.items()}
    return items, outputs


def _stack_shapes(case):
    h, f = case["hidden"], case["mlp"]
    return [s for _ in range(case["layers"]) for s in [(h, h)] * 4 + [(h, f)] * 2 + [(f, h)]]


def _block(r, m, n):
    return min((2 * r + 63) // 64 * 64, min(m, n) // 64 * 64)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    st = {"kind": kind, "status": torch.zeros(1, dtype=torch.int32, device="cuda"), "t": START_STEP}
    if kind in ("step", "plan"):
        shapes = [(case["m"], case["n"])] if kind == "step" else _stack_shapes(case)
        items, st["outputs"] = _items(shapes, case["r"], case["moments"], case["side"], seed, gen)
        if kind == "plan":
            st["plan"] = B.StepPlan(items)
        else:
            st["item"] = items[0]
            st["workspace"] = torch.empty(B.workspace_bytes(B.QG_OP_PROJECT_STEP, case["m"], case["n"], case["r"]),
                                          dtype=torch.uint8, device="cuda")
    elif kind == "refresh":
        m, n, r = case["m"], case["n"], case["r"]
        st["r"], st["side"] = r, case["side"]
        pm, pn = (n, m) if case["side"] == "right" else (m, n)
        items, st["outputs"] = _items([(m, n)] * case["count"], r, 32, case["side"], seed, gen)
        st["outputs"].pop("M.float32").zero_()
        st["outputs"]["sim"] = torch.zeros(case["count"], device="cuda")
        for i, it in enumerate(items):
            prev = _gaussian(pm, r, 1.0 / math.sqrt(pm), gen)
            it.update(P=B.dense_projection(pm, r), P_prev=B.quantize_int4(prev, B.dense_projection(pm, r)), sim=st["outputs"]["sim"][i:i + 1])
            it["P_new"] = it["P"]
        st["items"], st["batch"] = items, B.StepBatch(items)
        each = B.workspace_bytes(B.QG_OP_REFRESH, pm, pn, _block(r, m, n))
        st["workspace"] = torch.empty(each * case["count"], dtype=torch.uint8, device="cuda")
    elif kind in ("forward", "backward"):
        t, m, n = case["tokens"], case["m"], case["n"]
        st["W"] = B.quantize_int8(_gaussian(m, n, synth.WEIGHT_STD, gen))
        st["X"] = B.zeros_matrix(t, n, torch.bfloat16)
        st["X"].copy_(torch.randn(t, n, device="cuda", generator=gen))
        if kind == "backward":
            st["dY"] = B.zeros_matrix(t, m, torch.bfloat16)
            st["dY"].copy_(torch.randn(t, m, device="cuda", generator=gen).mul_(1e-3))
    else:
        st["bits"], st["x"] = case["bits"], _gaussian(case["m"], case["n"], synth.WEIGHT_STD, gen)
    return st


def run(st):
    kind = st["kind"]
    if kind in ("step", "plan"):
        st["t"] += 1
        hyper = B.Hyper(step=st["t"])
        if kind == "plan":
            st["plan"].step(hyper)
        else:
            B.project_step_item(st["item"], hyper, workspace=st["workspace"], status=st["status"])
        return st["outputs"]
    if kind == "refresh":
        # A column of a projection is a singular vector: its sign is a tie between its two largest entries, and with it the
        # sign of a row of M.  What is fixed, and comes back, is what the step makes of the new projection: W, V, similarity.
        B.refresh_subspace_batched(st["items"], st["r"], iters=REFRESH_ITERS, workspace=st["workspace"], status=st["status"],
                                   side=st["side"])
        st["t"] += 1
        st["batch"].step(B.Hyper(lr=LATE_LR, step=st["t"]))
        return st["outputs"]
    if kind == "forward":
        return B.int8_linear_forward(st["X"], st["W"], status=st["status"])
    if kind == "backward":
        return (B.int8_linear_backward_input(st["dY"], st["W"], status=st["status"]),
                B.int8_linear_backward_weight(st["dY"], st["X"], status=st["status"]))
    q = B.quantize_int8(st["x"]) if st["bits"] == 8 else B.quantize_int4(st["x"])
    return q.codes, q.scales, q.zeros, B.dequantize(q)


# ---------------------------------------------------------------------------------------------- units
def work(case):
    kind = case["kind"]
    if kind in ("step", "plan"):
        shapes = [(case["m"], case["n"])] if kind == "step" else _stack_shapes(case)
        r, bytes_, flops = case["r"], 0, 0
        for m, n in shapes:
            right = case["side"] == "right" or (case["side"] == "short" and m > n)
            cols, rows = (m, n) if right else (n, m)
            # gradient, codes in and out, scales and zeros in and out, projection, moments in and out
            state = 4 * r * cols + 16 * r * ((cols + 31) // 32) if case["moments"] == 8 else 16 * r * cols
            bytes_ += 4 * m * n + 16 * m * ((n + 255) // 256) + rows * r // 2 + 8 * rows * ((r + 255) // 256) + state
            flops += 4 * m * n * r
        return {"bytes": bytes_, "flops": flops}
    m, n = case["m"], case["n"]
    groups = 8 * m * ((n + 255) // 256)
    if kind == "refresh":
        r, b = case["r"], _block(case["r"], m, n)
        rows = n if case["side"] == "right" else m
        # per iteration two products with the gradient and an orthonormalisation (Gram matrix and its application); then the
        # projected matrix, its eigenvectors (about 9 b^3) and the rotation of the block onto them
        step = work({**case, "kind": "step", "moments": 32})
        flops = step["flops"] + REFRESH_ITERS * (4 * m * n * b + 2 * rows * b * b) + 2 * m * n * b + (m + n - rows) * b * b + 9 * b ** 3 + 2 * rows * b * r
        # the step reads the gradient and the new projection; the refresh writes the one and compares it with the old
        return {"bytes": case["count"] * (step["bytes"] + 2 * (rows * r // 2 + 8 * rows * ((r + 255) // 256))), "flops": case["count"] * flops}
    if kind == "forward":
        t = case["tokens"]
        return {"bytes": m * n + groups + 2 * t * (m + n), "flops": 2 * t * m * n}
    if kind == "backward":
        t = case["tokens"]
        return {"bytes": m * n + groups + 2 * t * (m + n) + 2 * t * n + 2 * m * n, "flops": 4 * t * m * n}
    code = 1.0 if case["bits"] == 8 else 0.5
    return {"bytes": (4 + 4 + 2 * code) * m * n + 2 * groups, "flops": 4 * m * n}


def tolerance(case):
    kind = case["kind"]
    if kind == "quantize":
        return "exact"                     # defined to the bit
    if kind in ("forward", "backward"):
        # fp32 sums in another order, rounded once to bfloat16: 2.5e-4 and one unit in the last place (2^-7) were seen against
        # torch's fp32 product of the same operands
        return {"rel": 1e-3, "max": 0.02}
    if kind == "refresh":
        # Products on the CUDA cores instead of the tensor cores, or the eigen-iteration in another order: 1.7e-3 of the codes
        # one level apart, V 3e-4 (the largest 2e-2), similarity 2.5e-3, 6e-4 of the zero points one apart.
        return {"rel": 1e-2, "max": 0.3, "differ": 7e-3}
    # Against the CUDA-core kernels: M, V 1e-6, scales 2e-5 (the largest 4e-3, where an approximated root meets a small
    # denominator), 2e-5 of the codes one level apart.  A group whose minimum lies at a tie of the zero point's rounding may
    # take its zero point, and with it all its codes, one apart: one such group in 3072 is what the zeros' bound allows for.
    # 8-bit moments add codes that lie within the fp32 error of a rounding boundary.
    return {"rel": 3e-3, "max": 0.3, "differ": 2e-3 if case["moments"] == 8 else 1e-3}
