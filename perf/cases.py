"""Workloads of the HARP library, as calls of its public entry points.

A processor is built once per layer and kept (`prepare`); a pass (`run`) is one call on data
that is already on the GPU.  Four uses are covered:

* rows of activations through a processor while a model runs (`harp.apply_`): batches from a
  single token to a long prefill, forward before a layer and transposed after it;
* rows in fp32, as a fitting loop keeps them;
* a weight matrix, or a layer's curvature proxy, processed on both sides (`harp.two_sided_`) in
  bf16 or fp32;
* the gradient with respect to the block kernels (`harp.harp_grad_blocks`), which fitting takes
  once per batch of calibration rows.

Dimensions and schedules are those of the five benchmark configurations and of the greedy
Mixed-Radix schedule for d = 4096 and 5120.
"""
import math

import torch

import paper_2605_29843_b200 as harp
from paper_2605_29843_b200 import workloads as wl

# schedule name -> (radices, block kind, permutation)
PLANS = {
    "d2048": ((2,) * 11, "givens_h2", "identity"),
    "d4096": ((4,) * 6, "expm_h", "digit_reversal"),
    "d4096_greedy": ((8, 8, 8, 8), "expm_h", "identity"),
    "d5120_greedy": ((8, 8, 8, 5, 2), "expm_h", "identity"),
    "d8192": ((8, 8, 8, 8, 2), "qr", "identity"),
    "d11008": ((2,) * 8 + (43,), "givens_h2", "identity"),
    "d14336": ((16, 16, 8, 7), "qr", "identity"),
    "d14336_permuted": ((16, 16, 8, 7), "qr", "random"),
    "d28672": ((8, 8, 8, 8, 7), "qr", "identity"),
}
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
CODES = {"bf16": harp.HARP_BF16, "f32": harp.HARP_F32}
MAX_BF16 = 65536 * 28672         # elements of the largest bf16 batch
MAX_F32 = 4096 * 11008           # elements of the largest fp32 matrix
MAX_GRAD = 16384 * 4096          # elements of the largest fitting batch


def dim(plan):
    return math.prod(PLANS[plan][0])


def apply_case(plan, rows, dtype, transpose, name=None):
    case = {"op": "apply", "plan": plan, "rows": rows, "dtype": dtype, "transpose": transpose}
    return {"name": name, **case} if name else case


def two_sided_case(out, inn, dtype, name=None):
    case = {"op": "two_sided", "plan_out": out, "plan_in": inn, "dtype": dtype}
    return {"name": name, **case} if name else case


def grad_case(plan, rows, dtype, name=None):
    case = {"op": "grad", "plan": plan, "rows": rows, "dtype": dtype}
    return {"name": name, **case} if name else case


def listed():
    return [
        # one token of a decode step in front of a wide layer: launches and latency
        apply_case("d14336", 1, "bf16", False, "decode 1 row d14336"),
        # a decode batch of sixteen sequences, back on the output side of a layer
        apply_case("d4096", 16, "bf16", True, "decode 16 rows d4096 T"),
        # calibration rows in fp32 through an all-radix-2 processor
        apply_case("d2048", 4096, "f32", False, "fp32 rows d2048"),
        # a prefill batch, permutation and signs included
        apply_case("d4096", 16384, "bf16", False, "prefill d4096"),
        # an ordinary batch of a ragged number of tokens, output side
        apply_case("d4096", 2051, "bf16", True, "ragged batch d4096 T"),
        # mixed-radix width with a large odd radix, output side
        apply_case("d11008", 8192, "bf16", True, "prefill d11008 T"),
        # wide mixed-radix layer, long prefill
        apply_case("d14336", 32768, "bf16", False, "prefill d14336"),
        # the same width behind an arbitrary permutation, ragged batch, output side
        apply_case("d14336_permuted", 4099, "bf16", True, "permuted ragged d14336 T"),
        # the widest rows, the largest batch
        apply_case("d28672", 65536, "bf16", False, "prefill d28672"),
        # a weight matrix processed on both sides in the dtype it is stored in
        two_sided_case("d8192", "d28672", "bf16", "weight 8192x28672"),
        # a weight matrix processed in fp32 ahead of quantisation
        two_sided_case("d4096_greedy", "d11008", "f32", "fp32 weight 4096x11008"),
        # one fitting step's gradient with respect to the block kernels
        grad_case("d4096", 16384, "bf16", "gradient d4096"),
    ]


def log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.random()
    if kind < 0.7:
        plan = rng.choice(sorted(PLANS))
        dtype = "f32" if plan == "d2048" or rng.random() < 0.2 else "bf16"
        most = (MAX_F32 if dtype == "f32" else MAX_BF16) // dim(plan)
        return apply_case(plan, log_uniform(rng, 1, min(65536, most)), dtype, rng.random() < 0.5)
    if kind < 0.85:
        dtype = "f32" if rng.random() < 0.4 else "bf16"
        while True:
            out = rng.choice(["d2048", "d4096_greedy", "d5120_greedy", "d8192"])
            inn = out if rng.random() < 0.3 else rng.choice(["d4096_greedy", "d5120_greedy", "d8192", "d11008", "d14336", "d28672"])
            if dim(out) * dim(inn) <= (MAX_F32 if dtype == "f32" else 8192 * 28672):
                return two_sided_case(out, inn, dtype)
    plan = rng.choice(["d2048", "d4096", "d8192", "d14336"])
    dtype = "f32" if plan == "d2048" or rng.random() < 0.3 else "bf16"
    return grad_case(plan, log_uniform(rng, 256, MAX_GRAD // dim(plan)), dtype)


def make_plan(name, seed):
    radices, kind, perm = PLANS[name]
    return harp.plan_from_spec(wl.make_plan(seed, dim(name), radices, kind, perm=perm))


def activations(gen, rows, d, dtype):
    """Normal rows with a fixed set of outlier channels (0.5 %, x50), drawn in slices of the batch."""
    x = torch.empty((rows, d), dtype=dtype, device="cuda")
    gain = torch.ones(d, device="cuda")
    gain[torch.randperm(d, generator=gen, device="cuda")[: max(1, d // 200)]] = 50.0
    step = max(1, (1 << 26) // d)
    for r in range(0, rows, step):
        n = min(step, rows - r)
        x[r:r + n] = torch.randn((n, d), generator=gen, device="cuda") * gain
    return x


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dtype = DTYPES[case["dtype"]]
    s = {"op": case["op"]}
    if case["op"] == "two_sided":
        s["out"] = make_plan(case["plan_out"], seed)
        # a curvature proxy is processed with the same processor on both sides
        s["in"] = s["out"] if case["plan_in"] == case["plan_out"] else make_plan(case["plan_in"], seed + 1)
        w = torch.randn((s["out"].d, s["in"].d), generator=gen, device="cuda") * 0.02
        s["w"] = (0.5 * (w + w.T) if s["in"] is s["out"] else w).to(dtype).contiguous()
        # kept by the program for all its layers, as the entry point suggests
        nbytes = harp.harp_two_sided_scratch_bytes(s["out"], s["in"], CODES[case["dtype"]])
        s["scratch"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        return s
    s["plan"] = make_plan(case["plan"], seed)
    s["x"] = activations(gen, case["rows"], s["plan"].d, dtype)
    if case["op"] == "apply":
        s["transpose"] = case["transpose"]
    else:
        s["code"] = CODES[case["dtype"]]
        s["gy"] = (torch.randn(s["x"].shape, generator=gen, device="cuda") * 1e-2).to(dtype)
        s["grad"] = torch.zeros(harp.harp_plan_n_params(s["plan"]), dtype=torch.float32, device="cuda")
    return s


def run(s):
    if s["op"] == "apply":
        return harp.apply_(s["plan"], s["x"], transpose=s["transpose"])
    if s["op"] == "two_sided":
        return harp.two_sided_(s["w"], s["out"], s["in"], s["scratch"])
    harp.harp_grad_blocks(s["plan"], s["x"].data_ptr(), s["gy"].data_ptr(), s["x"].shape[0], s["code"],
                          s["grad"].data_ptr(), False, torch.cuda.current_stream().cuda_stream)
    return s["grad"]


def work(case):
    """Rows or matrix read once and written once, block kernels read once; two operations per block
    entry and row.  The gradient reads x and dL/dy and writes one fp32 value per block entry; it takes
    the products of a forward sweep, a backward sweep and the outer products."""
    es = 2 if case["dtype"] == "bf16" else 4

    def entries(plan):
        return dim(plan) * sum(PLANS[plan][0])

    if case["op"] == "two_sided":
        d_out, d_in = dim(case["plan_out"]), dim(case["plan_in"])
        return {"bytes": 2 * d_out * d_in * es + es * (entries(case["plan_out"]) + entries(case["plan_in"])),
                "flops": 2 * (d_out * entries(case["plan_in"]) + d_in * entries(case["plan_out"]))}
    n = entries(case["plan"])
    if case["op"] == "apply":
        return {"bytes": 2 * case["rows"] * dim(case["plan"]) * es + es * n, "flops": 2 * case["rows"] * n}
    return {"bytes": 2 * case["rows"] * dim(case["plan"]) * es + 8 * n, "flops": 6 * case["rows"] * n}


def tolerance(case):
    """bf16 results carry a rounding per group of stages (2**-9 each) and bf16 block kernels; fp32
    applies and gradients (fp32 stage states, whatever the dtype of the rows) are sums in fp32."""
    if case["dtype"] == "bf16" and case["op"] != "grad":
        return {"rel": 1e-2}
    return {"rel": 1e-5}
