"""The calls whose speed matters to a user of this package, as cases that can be prepared and run.

A case is a dict of plain values.  ``op`` says which calls it makes:

    quantize        bof4_quantize of one tensor (with ``dq`` also bof4_scales_compress of its constants)
    dequantize      bof4_dequantize of one tensor (with ``dq`` after bof4_scales_expand of its constants)
    quantize_batch, dequantize_batch    the same over the list of tensors of a model or of some layers
    opq_quantize    bof4_quantize_opq and the read-back of its count (bof4_outlier_count)
    opq_dequantize  bof4_dequantize with the outlier list written back
    fit             bof4_fit_codebook over a list of tensors
    gemv            bof4_gemv through a list of matrices (one token)
    gemm            bof4_gemm_tc through a list of matrices (several tokens in flight)

``sizes`` lists the element counts of the tensors, ``shapes`` the rows x cols of the matrices.
Weights are near-Gaussian with a standard deviation of 0.01 to 0.04, as the weights of language
models are, with rare large outliers where outliers are what the call is for.
"""
import numpy as np
import torch

import paper_2505_06653_b200 as bof4

# Printed MSE codebooks for block size 64 (Tab. 6), signed and absolute normalisation.
LEVELS = {
    "signed": [-0.8568463921546936, -0.6692874431610107, -0.5235266089439392, -0.4004882574081421, -0.2910638153553009,
               -0.1900092959403992, -0.0938529595732689, 0.0, 0.0887671709060669, 0.1794802695512772, 0.2743096053600311,
               0.3760197460651398, 0.4886530041694641, 0.6188603639602661, 0.7791395783424377, 1.0],
    "abs": [-1.0, -0.7535245418548584, -0.579203724861145, -0.4385998845100403, -0.3167679905891418, -0.2059924453496933,
            -0.1015387624502182, 0.0, 0.0887245312333107, 0.1793769598007202, 0.2741499841213226, 0.3758211433887482,
            0.4884937703609467, 0.6187058687210083, 0.7790452241897583, 1.0],
}
DTYPE = {"bf16": torch.bfloat16, "f32": torch.float32}
CODE = {"bf16": bof4.BF16, "f32": bof4.F32}
NORM = {"abs": bof4.NORM_ABS, "signed": bof4.NORM_SIGNED}
METRIC = {"mse": bof4.METRIC_MSE, "mae": bof4.METRIC_MAE}
BYTES = {"bf16": 2, "f32": 4}
DEVICE = "cuda"

# One layer of the three model shapes that the workloads of this repository use.
LAYER_7B = [(4096, 4096)] * 4 + [(4096, 11008)] * 3
LAYER_8B = [(4096, 4096), (1024, 4096), (1024, 4096), (4096, 4096), (14336, 4096), (14336, 4096), (4096, 14336)]
MLP_70B = (28672, 8192)


def _sizes(shapes):
    return ",".join(str(r * c) for r, c in shapes)


def _shapes(shapes):
    return ",".join("%dx%d" % s for s in shapes)


def listed():
    return [
        # A small fp32 tensor (an adapter, a bias-like remainder, a test set) whose length is no multiple of anything: one call.
        {"name": "quantize_f32_1m_ragged", "op": "quantize", "sizes": str((1 << 20) + 37), "dtype": "f32", "scales": "f32",
         "block": 64, "norm": "abs", "dq": False},
        # One attention projection of a 7B-shaped model quantised by itself, its constants stored in 8 bits.
        {"name": "quantize_bf16_16m_dq", "op": "quantize", "sizes": str(4096 * 4096), "dtype": "bf16", "scales": "bf16",
         "block": 128, "norm": "signed", "dq": True},
        # A model converted several layers per call: the throughput workload of the benchmark, four of its layers.
        {"name": "quantize_batch_8b_4_layers", "op": "quantize_batch", "sizes": _sizes(LAYER_8B * 4), "dtype": "bf16", "scales": "bf16",
         "block": 64, "norm": "signed"},
        # A key or value projection decoded before use, the smallest matrix of the 8B shape.
        {"name": "dequantize_bf16_4m_dq", "op": "dequantize", "sizes": str(1024 * 4096), "dtype": "bf16", "scales": "bf16",
         "block": 64, "norm": "signed", "dq": True},
        # The same four layers decoded in one call.
        {"name": "dequantize_batch_8b_4_layers", "op": "dequantize_batch", "sizes": _sizes(LAYER_8B * 4), "dtype": "bf16", "scales": "bf16",
         "block": 64, "norm": "signed"},
        # An MLP matrix of the 70B shape with its outliers preserved; the count is read back, as a converter must before it stores the list.
        {"name": "opq_quantize_70b_mlp", "op": "opq_quantize", "sizes": str(MLP_70B[0] * MLP_70B[1]), "dtype": "bf16", "scales": "bf16",
         "block": 64, "norm": "signed", "q": 0.95},
        # ... and decoded with the outliers written back.
        {"name": "opq_dequantize_70b_mlp", "op": "opq_dequantize", "sizes": str(MLP_70B[0] * MLP_70B[1]), "dtype": "bf16", "scales": "bf16",
         "block": 64, "norm": "signed", "q": 0.95},
        # The first configuration of the workloads: 2^20 fp32 weights, 50 iterations; short passes in a long chain.
        {"name": "fit_mse_f32_1m", "op": "fit", "sizes": str(1 << 20), "dtype": "f32", "block": 64, "norm": "abs", "metric": "mse", "iters": 50},
        # The second one: 2^26 bf16 weights with heavy tails, 100 iterations, signed normalisation.
        {"name": "fit_mse_bf16_64m", "op": "fit", "sizes": str(1 << 26), "dtype": "bf16", "block": 64, "norm": "signed", "metric": "mse",
         "iters": 100},
        # The third one, the fitting sweep over a 7B-shaped model (a quarter of its layers), weighted medians: the largest.
        {"name": "fit_mae_bf16_7b_8_layers", "op": "fit", "sizes": _sizes(LAYER_7B * 8), "dtype": "bf16", "block": 64, "norm": "signed",
         "metric": "mae", "iters": 30},
        # One token through the seven projections of an 8B-shaped layer.
        {"name": "gemv_8b_layer", "op": "gemv", "shapes": _shapes(LAYER_8B), "dtype": "bf16", "scales": "bf16", "block": 64, "norm": "signed",
         "q": 0.0},
        # 32 sequences in flight through the same layer, with preserved outliers.
        {"name": "gemm_8b_layer_32_opq", "op": "gemm", "shapes": _shapes(LAYER_8B), "dtype": "bf16", "scales": "bf16", "block": 64,
         "norm": "signed", "q": 0.95, "rhs": 32},
    ]


# ----------------------------------------------------------------------------- drawn cases

OPS = ["quantize", "dequantize", "quantize_batch", "dequantize_batch", "opq_quantize", "opq_dequantize", "fit", "fit", "gemv", "gemm"]


def _log(rng, lo, hi):
    """An integer from lo to hi, even over the logarithm."""
    return int(round(lo * (hi / lo) ** rng.random()))


def _count(rng, lo, hi, block):
    """A tensor length: whole blocks as most tensors have, or any length."""
    n = _log(rng, lo, hi)
    return n if rng.random() < 0.4 else max(block, n // block * block)


def draw(rng):
    op = rng.choice(OPS)
    block = rng.choice([32, 64, 64, 64, 128, 256, 1024])
    c = {"op": op, "block": block, "norm": rng.choice(["signed", "abs"]), "dtype": rng.choice(["bf16", "bf16", "f32"])}
    if op == "fit":
        c["metric"] = rng.choice(["mse", "mae"])
        total = _log(rng, 1 << 16, 1 << (28 if c["dtype"] == "bf16" else 24))
        c["iters"] = _log(rng, 10, 60)
        k = rng.choice([1, 1, 2, 7, 14])
        cuts = [rng.uniform(0.2, 1.0) for _ in range(k)]
        c["sizes"] = ",".join(str(_count(rng, m, m + m // 8, block)) for m in (max(block, int(total * x / sum(cuts) * 0.9)) for x in cuts))
        return c
    c["scales"] = "f32" if c["dtype"] == "f32" or rng.random() < 0.25 else "bf16"
    if op in ("gemv", "gemm"):
        c["q"] = rng.choice([0.0, 0.95])
        unit = max(block, 64)
        out = []
        for _ in range(rng.choice([1, 1, 2, 4])):
            rows = _log(rng, 512, 28672)
            cols = _log(rng, 1024, 16384) // unit * unit
            if op == "gemm":
                rows = max(128, rows // 128 * 128)
            out.append((rows, max(unit, cols)))
        c["shapes"] = _shapes(out)
        if op == "gemm":
            c["rhs"] = rng.choice([16, 32, 48, 64])
            c["dtype"] = "bf16"
        return c
    if op in ("quantize_batch", "dequantize_batch"):
        k = rng.choice([2, 5, 7, 14, 28])
        c["sizes"] = ",".join(str(_count(rng, 1 << 14, 1 << 25, block)) for _ in range(k))
        return c
    c["sizes"] = str(_count(rng, 1 << 13, 1 << (27 if c["dtype"] == "bf16" else 26), block))
    if op in ("quantize", "dequantize"):
        c["dq"] = rng.random() < 0.3
    else:
        c["q"] = rng.choice([0.9, 0.95, 0.97, 0.99])
    return c


# ----------------------------------------------------------------------------- inputs


def _weights(n, dtype, gen, heavy=False, outliers=False):
    """n weights N(0, s^2), s from 0.01 to 0.04; `heavy`: 1 % of them Student-t with 4 degrees of freedom; `outliers`: 0.01 % of
    them replaced by 10 to 40 standard deviations."""
    s = 0.01 + 0.03 * torch.rand(1, generator=gen, device=DEVICE)
    w = torch.randn(n, generator=gen, device=DEVICE)
    if heavy or outliers:
        every = 100 if heavy else 10000
        k = n // every      # one at a random place of every 100 or 10000 weights: no place twice
        at = torch.arange(k, device=DEVICE) * every + torch.randint(0, every, (k,), generator=gen, device=DEVICE)
        if heavy:
            chi2 = torch.randn(4, k, generator=gen, device=DEVICE).square_().sum(0)
            w[at] = torch.randn(k, generator=gen, device=DEVICE) / (chi2 / 4).sqrt()
        else:
            sign = torch.randint(0, 2, (k,), generator=gen, device=DEVICE) * 2 - 1
            w[at] = (10 + 30 * torch.rand(k, generator=gen, device=DEVICE)) * sign
    return w.mul_(s).to(DTYPE[dtype])


def _matrices(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split(",")]


def _counts(case):
    if "shapes" in case:
        return [r * c for r, c in _matrices(case)]
    return [int(v) for v in case["sizes"].split(",")]


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed))
    op, block, norm = case["op"], case["block"], NORM[case["norm"]]
    st = {"case": case, "block": block, "norm": norm}
    if op == "fit":
        st["w"] = [_weights(n, case["dtype"], gen, heavy=case["metric"] == "mse") for n in _counts(case)]
        st["levels"], st["mask"] = bof4.bof4_default_init(norm)
        return st
    q = case.get("q", 0.0)
    st["levels"] = torch.tensor(np.array(LEVELS[case["norm"]], np.float32), device=DEVICE)
    st["scales"] = CODE[case["scales"]]
    st["out_dtype"] = CODE[case["dtype"]]
    if q:
        st["tau"] = float(np.float32(bof4.bof4_opq_threshold(q, block)))
    w = [_weights(n, case["dtype"], gen, outliers=q > 0) for n in _counts(case)]
    if op in ("quantize", "quantize_batch", "opq_quantize"):
        st["w"] = w
        if op == "opq_quantize":
            # A converter goes through the layers with one set of buffers.
            n, cap = w[0].numel(), w[0].numel() // 64 + 1024
            new = lambda m, t: torch.zeros(m, dtype=t, device=DEVICE)  # noqa: E731
            st["capacity"] = cap
            st["out"] = (new((n + 1) // 2, torch.uint8), new(-(-n // block), DTYPE[case["scales"]]), new(cap, torch.int32),
                         new(cap, torch.bfloat16), new(1, torch.int64))
            st["workspace"] = new(bof4.bof4_workspace_bytes(bof4.OP_OPQ, n, block), torch.uint8)
        return st
    # What a program that decodes has in hand: codes, constants and outlier lists, as the quantiser wrote them.
    st["n"] = [t.numel() for t in w]
    st["codes"], st["consts"], st["outliers"] = [], [], []
    for t in w:
        if q:
            codes, consts, idx, val, cnt = bof4.bof4_quantize_opq(t, block, norm, st["levels"], st["tau"], t.numel() // 64 + 1024,
                                                                  st["scales"])
            k = bof4.bof4_outlier_count(cnt, idx.numel())
            st["outliers"].append((idx[:k].clone(), val[:k].clone(), cnt))
        else:
            codes, consts = bof4.bof4_quantize(t, block, norm, st["levels"], st["scales"])
            st["outliers"].append(None)
        st["codes"].append(codes)
        st["consts"].append(consts)
    if case.get("dq"):
        st["packed"] = bof4.bof4_scales_compress(st["consts"][0], norm)
        del st["consts"]
    if op in ("gemv", "gemm"):
        x = [torch.randn(case.get("rhs", 1) * c, generator=gen, device=DEVICE).to(DTYPE[case["dtype"]]) for _, c in _matrices(case)]
        st["shapes"] = _matrices(case)
        st["x"] = [t.view(case["rhs"], -1) if op == "gemm" else t for t in x]
    return st


# ----------------------------------------------------------------------------- one pass


def run(st):
    op, block = st["case"]["op"], st["block"]
    if op == "quantize":
        codes, consts = bof4.bof4_quantize(st["w"][0], block, st["norm"], st["levels"], st["scales"])
        if st["case"]["dq"]:
            return [codes, *bof4.bof4_scales_compress(consts, st["norm"])]
        return [codes, consts]
    if op == "dequantize":
        consts = bof4.bof4_scales_expand(*st["packed"]) if st["case"]["dq"] else st["consts"][0]
        return bof4.bof4_dequantize(st["codes"][0], consts, block, st["levels"], st["out_dtype"], n=st["n"][0])
    if op == "quantize_batch":
        return bof4.bof4_quantize_batch(st["w"], block, st["norm"], st["levels"], st["scales"])
    if op == "dequantize_batch":
        return bof4.bof4_dequantize_batch(st["codes"], st["consts"], st["n"], block, st["levels"], st["out_dtype"])
    if op == "opq_quantize":
        out = bof4.bof4_quantize_opq(st["w"][0], block, st["norm"], st["levels"], st["tau"], st["capacity"], st["scales"],
                                     workspace=st["workspace"], out=st["out"])
        return [*out[:4], bof4.bof4_outlier_count(out[4], st["capacity"])]
    if op == "opq_dequantize":
        return bof4.bof4_dequantize(st["codes"][0], st["consts"][0], block, st["levels"], st["out_dtype"], st["outliers"][0], n=st["n"][0])
    if op == "fit":
        levels, log = bof4.bof4_fit_codebook(st["w"], block, st["norm"], METRIC[st["case"]["metric"]], st["levels"], st["mask"],
                                             st["case"]["iters"])
        return [levels, log]
    if op == "gemv":
        return [bof4.bof4_gemv(codes, consts, r, c, block, st["levels"], x, outliers)
                for (r, c), codes, consts, x, outliers in zip(st["shapes"], st["codes"], st["consts"], st["x"], st["outliers"])]
    return [bof4.bof4_gemm_tc(codes, consts, r, c, block, st["levels"], x, outliers=outliers)
            for (r, c), codes, consts, x, outliers in zip(st["shapes"], st["codes"], st["consts"], st["x"], st["outliers"])]


# ----------------------------------------------------------------------------- what a pass needs


def work(case):
    """Bytes: the weights (or codes and constants) read once and the results written once; a fit reads its weights once per iteration,
    since the levels of an iteration depend on all the weights seen in the one before.  Operations: the multiplications and
    additions of the products; elsewhere the division of a weight by its constant (two in an MSE fit for the sums)."""
    ns, op = _counts(case), case["op"]
    n = sum(ns)
    if op == "fit":
        passes = n * case["iters"]
        return {"bytes": passes * BYTES[case["dtype"]] + 64 + 8 * case["iters"], "flops": 3 * passes}
    blocks = sum(-(-m // case["block"]) for m in ns)
    packed = n / 2 + blocks * (BYTES[case["scales"]] if not case.get("dq") else 1 + 4 / 256 + (1 / 8 if case["norm"] == "signed" else 0))
    if case.get("q"):
        packed += 6 * n * (1e-4 + 1 - case["q"] ** (1 / case["block"]))     # index and value of the outliers
    if op in ("gemv", "gemm"):
        rhs = case.get("rhs", 1)
        xy = sum(rhs * (c * BYTES[case["dtype"]] + r * 4) for r, c in _matrices(case))
        return {"bytes": packed + xy, "flops": 2 * n * rhs}
    return {"bytes": packed + n * BYTES[case["dtype"]], "flops": n}


def tolerance(case):
    """Codes, constants, outlier lists and decoded weights are exact by definition.  A fit's sums, levels and errors and the fp32
    products depend on the order of summation."""
    return {"rel": 1e-5} if case["op"] in ("fit", "gemv", "gemm") else "exact"
