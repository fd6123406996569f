"""What a user of this library has it do, as cases that can be timed: each is ONE pass through the public binding.

A case is a dict of plain values; ``kind`` names the path and the rest its sizes and options:

* ``token``    hierarchical activation quantization: tensor abs-max -> g on the device -> quantize (no block SSE)
* ``prefill``  the same with the block SSE, followed by the de-quantization of the result
* ``weight``   quantize + tensor MSE in one call
* ``layer``    a list of weight matrices in one multi-tensor launch
* ``fake``     fused fake-quantize (x -> x_hat)
* ``study``    the scoring pass of the numerical study: quantize, segment MSE, clipping-only SSE and its segment MSE,
               histograms of codes and scales
* ``search``   brute-force scale search + tensor MSE, as the full sweep (default) or with the pruned-sweep option

Inputs are those of ``paper_2605_08565_b200/inputs.py``; shapes are the benchmark configurations' own, parts of them, or
ragged ones of the same size.
"""
import torch

from paper_2605_08565_b200 import binding as mxq
from paper_2605_08565_b200 import inputs

FMT = {"ue8m0": mxq.MXQ_SF_UE8M0, "ue4m3": mxq.MXQ_SF_UE4M3, "ue5m3": mxq.MXQ_SF_UE5M3}
CODES = {"ue8m0": 255, "ue4m3": 127, "ue5m3": 255}
RECIPE = {"absmax": mxq.MXQ_ABSMAX, "absmax_pz": mxq.MXQ_ABSMAX_PZ, "4o6": mxq.MXQ_4O6, "4o6_pz": mxq.MXQ_4O6_PZ,
          "brute": mxq.MXQ_BRUTE, "brute_pz": mxq.MXQ_BRUTE_PZ, "ocp": mxq.MXQ_ABSMAX_OCP, "clip7": mxq.MXQ_ABSMAX_CLIP7}
DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}
BYTES = {"f32": 4, "bf16": 2}
SEGMENTS = 151   # standard deviations of the numerical study


def _case(kind, rows, cols, dtype, B, fmt, recipe, **more):
    return dict({"kind": kind, "rows": rows, "cols": cols, "dtype": dtype, "B": B, "fmt": fmt, "recipe": recipe}, **more)


def listed():
    def named(name, c):
        return dict(c, name=name)
    return [
        # decoding: the activations of a few tokens are quantized before every linear layer; latency and launches
        named("decode_4_tokens", _case("token", 4, 4096, "bf16", 16, "ue4m3", "4o6")),
        # a layer's activations for a long prompt, quantized and read back (simulated FP4 activations)
        named("prefill_8192x4096", _case("prefill", 8192, 4096, "bf16", 16, "ue4m3", "4o6", out="bf16")),
        # an MLP weight matrix, the common recipe of the experiments
        named("weight_14336x4096", _case("weight", 14336, 4096, "bf16", 16, "ue4m3", "absmax_pz")),
        # the finest block size of the sweep over block sizes
        named("weight_finest_blocks", _case("weight", 4096, 4096, "bf16", 2, "ue4m3", "absmax")),
        # an odd-sized matrix whose blocks do not fill the last chunk
        named("weight_ragged", _case("weight", 1001, 1000, "bf16", 8, "ue5m3", "4o6_pz")),
        # one decoder layer of the weight set (seven matrices) in one launch
        named("layer_one_launch", _case("layer", 4096, 4096, "bf16", 8, "ue4m3", "4o6", divide=1)),
        # simulated MX format inside a training or evaluation step
        named("fake_quant_mx", _case("fake", 8192, 4096, "bf16", 32, "ue8m0", "ocp", out="bf16")),
        # the numerical study's scoring of one recipe at one block size (50,000 blocks per standard deviation)
        named("study_scoring", _case("study", SEGMENTS, 400000, "f32", 8, "ue4m3", "4o6_pz")),
        # the search on a small tensor: 1024 x 1024, N(0, 1), under a tensor scale
        named("search_1024x1024", _case("search", 1024, 1024, "f32", 16, "ue4m3", "brute", data="normal", scaled=True, prune=False)),
        # bulk search, every code of the larger FP8 scale format on every block
        named("search_bulk", _case("search", 4096, 4096, "f32", 8, "ue5m3", "brute", data="laplace", scaled=True, prune=False)),
        # bulk search with small blocks through the pruned sweep
        named("search_pruned_bulk", _case("search", 8192, 8192, "f32", 4, "ue4m3", "brute", data="laplace", scaled=True, prune=True)),
        # weight matrix searched through the pruned sweep, no tensor scale
        named("search_pruned_weight", _case("search", 4096, 14336, "bf16", 16, "ue5m3", "brute_pz", data="student_t", scaled=False, prune=True)),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _size(rng, lo, hi, step):
    """rows x cols with a product between lo and hi, cols a multiple of step; odd row counts are as likely as even ones."""
    n = _log_int(rng, lo, hi)
    cols = step * _log_int(rng, 1, max(1, min(n, 16384) // step))
    return max(1, n // cols), cols


def draw(rng):
    kind = rng.choice(["token", "prefill", "weight", "weight", "layer", "fake", "study", "search", "search", "search"])
    fp8 = rng.choice(["ue4m3", "ue5m3"])
    fmt = rng.choice(["ue4m3", "ue5m3", "ue4m3", "ue5m3", "ue8m0"])
    one_pass = rng.choice(["absmax", "absmax_pz", "4o6", "4o6_pz"])
    B = rng.choice([2, 4, 8, 16, 32, 64])
    dtype = rng.choice(["bf16", "bf16", "f32"])
    out = rng.choice(["bf16", "f32"])
    if kind == "token":
        return _case(kind, _log_int(rng, 1, 64), rng.choice([1024, 4096, 14336]), "bf16", rng.choice([16, 32]), fp8, rng.choice(["absmax", "4o6"]))
    if kind == "prefill":
        return _case(kind, _log_int(rng, 65, 8192), rng.choice([1024, 4096, 4096]), "bf16", rng.choice([16, 32]), fp8, rng.choice(["absmax", "4o6"]), out=out)
    if kind == "layer":
        return _case(kind, 4096, 4096, "bf16", rng.choice([8, 16, 32]), fp8, one_pass, divide=rng.choice([1, 2, 4, 8]))
    if kind == "study":
        B = rng.choice([4, 8, 16, 32])
        return _case(kind, SEGMENTS, B * _log_int(rng, 100, 400000 // B), "f32", B, "ue4m3", one_pass)
    if kind == "weight":
        rows, cols = _size(rng, 1 << 14, 14336 * 4096, B)
        return _case(kind, rows, cols, dtype, B, fmt, one_pass)
    if kind == "fake":
        rows, cols = _size(rng, 1 << 14, 8192 * 4096, B)
        return _case(kind, rows, cols, dtype, B, fmt, rng.choice(["absmax", "4o6", "ocp", "clip7"]) if fmt == "ue8m0" else one_pass, out=out)
    prune = rng.random() < 0.5
    rows, cols = _size(rng, 1 << 16, 4096 * (14336 if prune else 4096), B)
    data = rng.choice(["normal", "laplace", "student_t"])
    return _case(kind, rows, cols, "bf16" if data == "student_t" else "f32", B, fmt, rng.choice(["brute", "brute_pz"]), data=data,
                 scaled=rng.random() < 0.5, prune=prune)


def _shapes(case):
    """The seven matrices of a decoder layer, every side divided by `divide`."""
    d = case["divide"]
    return [(r // d, c // d) for _, r, c in inputs.LLAMA8B_LAYER_SHAPES]


def _values(case, seed):
    kind, rows, cols, dt = case["kind"], case["rows"], case["cols"], DTYPE[case["dtype"]]
    if kind in ("token", "prefill", "fake"):
        return inputs.outlier_columns(rows, cols, seed, dtype=dt, device="cuda")
    if kind == "study":
        return inputs.sigma_sweep(cols, seed, rows, dtype=dt, device="cuda")
    data = case.get("data", "student_t")
    if data == "normal":
        return inputs.normal(rows * cols, seed, 1.0, dt, "cuda")
    if data == "laplace":
        return inputs.laplace(rows * cols, seed, dt, "cuda")
    return inputs.student_t(rows * cols, 4, cols ** -0.5, seed, dt, "cuda")


def _tensor_scale(x):
    amax = torch.empty(1, dtype=torch.float32, device=x.device)
    g = torch.empty(1, dtype=torch.float32, device=x.device)
    mxq.mxq_tensor_amax(x, x.numel(), amax, g)
    return amax, g


def prepare(case, seed):
    kind, B = case["kind"], case["B"]
    s = {"case": case}
    if kind == "layer":
        xs = [inputs.student_t(r * c, 4, c ** -0.5, seed * 7 + i, DTYPE[case["dtype"]], "cuda") for i, (r, c) in enumerate(_shapes(case))]
        outs = [mxq.alloc_outputs(x.numel(), B, x.device) for x in xs]
        s["x"], s["outs"] = xs, outs
        s["h"], s["d"] = mxq.make_tensor_descs([(x, *o) for x, o in zip(xs, outs)])
        return s
    x = s["x"] = _values(case, seed)
    dev, n = x.device, x.numel()
    if kind == "fake":
        s["xhat"] = torch.empty(n, dtype=DTYPE[case["out"]], device=dev)
        return s
    s["codes"], s["scales"], s["sse"] = mxq.alloc_outputs(n, B, dev, with_sse=kind != "token")
    if kind in ("token", "prefill"):
        s["amax"] = torch.empty(1, dtype=torch.float32, device=dev)
        s["g"] = torch.empty(1, dtype=torch.float32, device=dev)
    if kind == "prefill":
        s["xhat"] = torch.empty(n, dtype=DTYPE[case["out"]], device=dev)
    if kind in ("weight", "search"):
        s["mse"] = torch.empty(1, dtype=torch.float64, device=dev)
        s["ws"] = torch.empty(mxq.mxq_tensor_mse_workspace_bytes(n // B) // 8, dtype=torch.float64, device=dev)
        s["g"] = _tensor_scale(x)[1] if case.get("scaled") else None   # a search runs many times under one tensor scale
    if kind == "study":
        s["clip"] = torch.empty(n // B, dtype=torch.float32, device=dev)
        s["mse"] = torch.empty(case["rows"], dtype=torch.float64, device=dev)
        s["cmse"] = torch.empty(case["rows"], dtype=torch.float64, device=dev)
        s["code_hist"] = torch.zeros(16, dtype=torch.int64, device=dev)
        s["scale_hist"] = torch.zeros(256, dtype=torch.int64, device=dev)
    return s


def run(s):
    case = s["case"]
    kind, B, fmt, recipe = case["kind"], case["B"], FMT[case["fmt"]], RECIPE[case["recipe"]]
    if kind == "layer":
        mxq.mxq_quantize_batch(s["h"], s["d"], len(s["x"]), mxq.MXQ_BF16, B, fmt, recipe)
        return s["outs"]
    x = s["x"]
    n = x.numel()
    if kind == "fake":
        mxq.mxq_fake_quantize(x, n, B, fmt, recipe, 1.0, None, s["xhat"])
        return s["xhat"]
    codes, scales, sse = s["codes"], s["scales"], s["sse"]
    if kind == "token":
        mxq.mxq_tensor_amax(x, n, s["amax"], s["g"])
        mxq.mxq_quantize_ex(x, n, B, fmt, recipe, 1.0, s["g"], codes, scales, None)
        return s["amax"], s["g"], codes, scales
    if kind == "prefill":
        mxq.mxq_tensor_amax(x, n, s["amax"], s["g"])
        mxq.mxq_quantize_ex(x, n, B, fmt, recipe, 1.0, s["g"], codes, scales, sse)
        mxq.mxq_dequantize_ex(codes, scales, n, B, fmt, 1.0, s["g"], s["xhat"])
        return s["amax"], s["g"], codes, scales, sse, s["xhat"]
    if kind == "weight":
        mxq.mxq_quantize_mse(x, n, B, fmt, recipe, 1.0, None, codes, scales, sse, s["mse"], s["ws"])
        return codes, scales, sse, s["mse"]
    if kind == "study":
        blocks = case["cols"] // B
        mxq.mxq_quantize_ex(x, n, B, fmt, recipe, 1.0, None, codes, scales, sse)
        mxq.mxq_segment_mse(sse, n // B, blocks, case["cols"], s["mse"])
        mxq.mxq_block_clip_sse(x, n, B, fmt, 1.0, None, scales, s["clip"])
        mxq.mxq_segment_mse(s["clip"], n // B, blocks, case["cols"], s["cmse"])
        s["code_hist"].zero_()
        s["scale_hist"].zero_()
        mxq.mxq_histograms(codes, scales, n, B, s["code_hist"], s["scale_hist"])
        return codes, scales, sse, s["mse"], s["clip"], s["cmse"], s["code_hist"], s["scale_hist"]
    if case["prune"]:
        mxq.mxq_set_option(mxq.MXQ_OPT_BRUTE_PRUNE, 1)
    mxq.mxq_quantize_mse(x, n, B, fmt, recipe, 1.0, s["g"], codes, scales, sse, s["mse"], s["ws"])
    if case["prune"]:
        mxq.mxq_set_option(mxq.MXQ_OPT_BRUTE_PRUNE, 0)
    return codes, scales, sse, s["mse"]


def work(case):
    kind, B = case["kind"], case["B"]
    n = sum(r * c for r, c in _shapes(case)) if kind == "layer" else case["rows"] * case["cols"]
    b_in = BYTES[case["dtype"]]
    # multiply by the scale's reciprocal, round, residual (2), square-accumulate (2)
    per_candidate = 6
    candidates = 2 if case["recipe"].startswith("4o6") else 1
    if kind == "search" and not case["prune"]:
        candidates = CODES[case["fmt"]]       # every code on every block is what was asked for
    if kind == "token":
        per_elem = b_in + 0.5 + 1.0 / B
    elif kind == "prefill":
        per_elem = b_in + 0.5 + 5.0 / B + BYTES[case["out"]]
    elif kind == "fake":
        per_elem = b_in + BYTES[case["out"]]
    elif kind == "study":
        per_elem = b_in + 0.5 + 9.0 / B
    else:
        per_elem = b_in + 0.5 + 5.0 / B
    return {"bytes": n * per_elem, "flops": float(n) * per_candidate * candidates}


def tolerance(case):
    # Codes, scale bytes and counts are whole numbers and equal; block SSEs and de-quantized values are defined to the last bit
    # (binary32, fixed order).  Only the order of the binary64 sums behind an MSE is free: two trees over the same block
    # SSEs differ by up to 4e-16 relative.
    return {"rel": 2e-15, "max": 2e-15, "differ": 0.0}
