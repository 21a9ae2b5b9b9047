"""Workloads of the PeRQ online path, timed and compared through the package's public entry points.

`listed()` gives the fixed cases, `draw(rng)` further ones of the same ranges; `prepare` makes what a program holds
on the GPU before a call, `run` is one call, `work` what the call cannot do without, `tolerance` how far two correct
implementations may differ.  Shapes are the workload generator's (inputs.py: Llama-3 1B / 8B layers) and the layer
widths of the paper's operation-count tables (Llama-3 and Qwen3 down projections), plus ragged widths and token counts.
"""
import math

import torch

from paper_2601_22347_b200 import binding as B

# Layer widths in use: hidden sizes 2048 and 4096, down-projection inputs 6144 ... 14336 (9728 is no multiple of 1024).
WIDTHS = (2048, 3072, 4096, 6144, 8192, 9728, 12288, 14336)
MAX_TOKENS = 16384


def _rotate(name, T, d, b, fmt, group, perm, values):
    return {"name": name, "call": "rotate", "T": T, "d": d, "b": b, "fmt": fmt, "group": group, "perm": perm,
            "values": values}


def listed():
    return [
        # one token of a decode step into Llama-3-8B's down projection: latency
        _rotate("decode_1x14336_perm_g128", 1, 14336, 32, "int4", 128, "random", "gauss"),
        # a decode batch / short prompt at a small hidden size
        _rotate("hidden_256x2048_b16_token", 256, 2048, 16, "int4", 0, "none", "gauss"),
        # Llama-3-1B hidden states, permuted, full-vector rotation
        _rotate("hidden_4096x2048_full_perm_g128", 4096, 2048, 2048, "int4", 128, "random", "student"),
        # Llama-3-1B down-projection input under its MassDiff permutation
        _rotate("down_4096x8192_perm_mxfp4", 4096, 8192, 32, "mxfp4", 32, "massdiff", "swiglu"),
        # Llama-3-8B hidden states, a full prefill batch: the headline workload
        _rotate("hidden_16384x4096_b32_token", 16384, 4096, 32, "int4", 0, "none", "laplace"),
        # the same states with the full-vector rotation that block rotations are compared with
        _rotate("hidden_16384x4096_full_token", 16384, 4096, 4096, "int4", 0, "none", "laplace"),
        # Llama-3-8B down-projection input, permuted, a full prefill batch: the largest call
        _rotate("down_16384x14336_perm_g128", 16384, 14336, 128, "int4", 128, "random", "gauss"),
        # the same width with a full-vector rotation (14336 = 2^9 * 28, no power of two)
        _rotate("down_1024x14336_full_token", 1024, 14336, 14336, "int4", 0, "none", "gauss"),
        # a ragged prompt at a width that is no multiple of 1024, with the paper's asymmetric per-token quantiser
        _rotate("down_1531x9728_b128_asym", 1531, 9728, 128, "int4_asym", 0, "none", "swiglu"),
        # the gated activation of the feedforward block fused in front of the rotation
        {"name": "swiglu_4096x8192_mxfp4", "call": "swiglu", "T": 4096, "d": 8192, "b": 32, "fmt": "mxfp4", "group": 32},
        # calibration, per batch: channel, block and token statistics
        {"name": "stats_4096x8192_b32", "call": "stats", "T": 4096, "d": 8192, "b": 32, "perm": "none", "values": "swiglu"},
        # calibration, per layer: the MassDiff permutation from the accumulated channel sums
        {"name": "massdiff_8192_b32", "call": "massdiff", "d": 8192, "b": 32},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call = rng.choices(("rotate", "swiglu", "stats", "massdiff"), (16, 2, 2, 1))[0]
    if call == "massdiff":
        return {"call": call, "d": 128 * rng.randint(8, 64), "b": rng.choice((16, 32, 64, 128))}
    if call == "swiglu":
        d = rng.choice([w for w in WIDTHS if w % 1024 == 0])
        fmt, group = rng.choice((("mxfp4", 32), ("int4", 128), ("int4", 0)))
        return {"call": call, "T": _log_int(rng, 1, MAX_TOKENS // 2), "d": d, "b": rng.choice((16, 32, 64, 128)), "fmt": fmt,
                "group": group}
    values = rng.choice(("gauss", "student", "laplace", "swiglu"))
    # one width in five is ragged: any multiple of 128
    d = rng.choice(WIDTHS) if rng.random() < 0.8 else 128 * rng.randint(6, 112)
    if call == "stats":
        return {"call": call, "T": _log_int(rng, 16, MAX_TOKENS // 2), "d": d, "b": rng.choice((16, 32, 64, 128)),
                "perm": rng.choice(("none", "random")), "values": values}
    perm = rng.choice(("none", "none", "random", "massdiff"))
    fmt, group = rng.choice((("int4", 0), ("int4", 0), ("int4", 128), ("mxfp4", 32), ("mxfp4", 32), ("fp4", 0),
                             ("int4_asym", 0)))
    kind = rng.random()
    top = MAX_TOKENS * 14336
    if kind < 0.75:
        b = rng.choice((16, 32, 64, 128))
        if d % 1024:
            top = MAX_TOKENS * 2048
    elif kind < 0.85:                     # long blocks inside the row
        b = rng.choice([v for v in (128, 256, 512, 1024, 2048) if d % v == 0])
        top = MAX_TOKENS * 2048
    else:                                 # the full-vector rotation
        d = b = rng.choice(WIDTHS)
        if d & (d - 1):
            top, group = 1024 * 14336, (0 if fmt == "int4" else group)
        else:
            top = MAX_TOKENS * 4096
    T = _log_int(rng, 1, min(MAX_TOKENS, top // d))
    return {"call": call, "T": T, "d": d, "b": b, "fmt": fmt, "group": group, "perm": perm, "values": values}


def _values(kind, T, d, gen):
    """Activations [T, d] in bf16: the element distributions of the workload generator, with its outlier channels."""
    def normal():
        return torch.randn(T, d, generator=gen, device="cuda")

    if kind == "gauss":
        v, n_out, factor = normal(), max(1, d // 224), 50.0
    elif kind == "student":               # three degrees of freedom: z / sqrt(chi^2_3 / 3)
        v, n_out, factor = normal() / ((normal() ** 2 + normal() ** 2 + normal() ** 2) / 3).sqrt(), max(1, d // 128), 100.0
    elif kind == "laplace":
        u = torch.rand(T, d, generator=gen, device="cuda") - 0.5
        v, n_out, factor = -u.sign() * torch.log1p(-2 * u.abs()).clamp_min(-20.0), max(1, d // 1000), 200.0
    else:
        v, n_out, factor = torch.nn.functional.silu(normal()) * normal(), max(1, d // 256), 30.0
    ch = torch.randperm(d, generator=gen, device="cuda")[:n_out]
    v[:, ch] *= factor
    return v.to(torch.bfloat16)


def _channel_mass(x):
    return x.abs().sum(0, dtype=torch.float64).to(torch.float32)


def _permutation(kind, x, b, gen):
    if kind == "none":
        return None
    if kind == "random":
        return torch.randperm(x.shape[1], generator=gen, device="cuda").to(torch.int32)
    return torch.from_numpy(B.perq_massdiff_perm(_channel_mass(x[:2048]).cpu().numpy(), b)).cuda()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    d, b = case["d"], case["b"]
    s = {"call": case["call"], "b": b}
    if case["call"] == "massdiff":
        s["mass"] = _channel_mass(_values("swiglu", 512, d, gen))
        s["perm"] = torch.empty(d, dtype=torch.int32, device="cuda")
        s["workspace"] = torch.empty(4 * d, dtype=torch.uint8, device="cuda")
        return s
    T = case["T"]
    if case["call"] == "swiglu":
        s["gate"] = (2.0 * torch.randn(T, d, generator=gen, device="cuda")).to(torch.bfloat16)
        s["up"] = _values("gauss", T, d, gen)
    else:
        s["x"] = _values(case["values"], T, d, gen)
        s["perm"] = _permutation(case["perm"], s["x"], b, gen)
    if case["call"] == "stats":
        n = B.perq_block_l1_stats_workspace_bytes(T, d, b)
        s["workspace"] = torch.empty(max(16, n), dtype=torch.uint8, device="cuda")
        return s
    s["fmt"], s["group"] = B.FMT_BY_NAME[case["fmt"]], case["group"]
    s["codes"], s["scales"] = B.alloc_outputs(T, d, s["fmt"], s["group"], "cuda")
    return s


def run(s):
    if s["call"] == "rotate":
        return B.perq_rotate_quantize(s["x"], s["perm"], s["b"], s["fmt"], s["group"], s["codes"], s["scales"])
    if s["call"] == "swiglu":
        return B.perq_swiglu_rotate_quantize(s["gate"], s["up"], None, s["b"], s["fmt"], s["group"], s["codes"], s["scales"])
    if s["call"] == "stats":
        return B.perq_block_l1_stats(s["x"], s["perm"], s["b"], workspace=s["workspace"])
    return B.perq_massdiff_perm_device(s["mass"], s["b"], s["perm"], s["workspace"])


def _add_sub_per_row(d, b):
    """Butterfly stages, and for b = 2^k' * 4t the dense product with the 4t-dimensional base matrix."""
    base = 1
    if b & (b - 1):
        base = b
        while base % 2 == 0:
            base //= 2
        base *= 4
    return d * (math.log2(b // base) + base - 1)


def work(case):
    d, b = case["d"], case["b"]
    if case["call"] == "massdiff":        # a sort of the channels and one choice among the blocks for each
        return {"bytes": 8 * d, "flops": d * (math.log2(d) + math.log2(d // b))}
    T = case["T"]
    if case["call"] == "stats":
        perm = 4 * d if case["perm"] != "none" else 0
        return {"bytes": 2 * T * d + perm + 4 * (d + d // b + T), "flops": 2 * T * d}
    codes, scales = B.perq_out_sizes(T, d, B.FMT_BY_NAME[case["fmt"]], case["group"])
    streams = 2 if case["call"] == "swiglu" else 1
    perm = 4 * d if case.get("perm", "none") != "none" else 0
    return {"bytes": 2 * streams * T * d + perm + codes + scales, "flops": T * (_add_sub_per_row(d, b) + 2 * d * streams)}


def tolerance(case):
    if case["call"] == "massdiff":
        return "exact"
    if case["call"] == "stats":           # fp32 sums of up to 16384 magnitudes, in another order
        return {"rel": 1e-6, "max": 4e-6}
    # codes and shared exponents are exact; two fp32 roundings of the exact scale are at most 2 ulp apart
    return {"rel": 2.5e-7, "max": 5e-7}


def _base_matrix(n):
    """The +-1 base matrix of order n = 2 (q + 1), q = 1 (mod 4) a prime: Paley's second construction."""
    q = n // 2 - 1
    squares = {(a * a) % q for a in range(1, q)}
    core = torch.ones(q + 1, q + 1, dtype=torch.float64)
    for i in range(1, q + 1):
        for j in range(1, q + 1):
            core[i, j] = 0 if i == j else (1 if (i - j) % q in squares else -1)
    core[0, 0] = 0
    core[0, 1:] = core[1:, 0] = 1
    # a zero becomes [[1, -1], [-1, -1]], an entry s becomes s [[1, 1], [1, -1]]
    one = torch.tensor([[1.0, 1.0], [1.0, -1.0]], dtype=torch.float64)
    zero = torch.tensor([[1.0, -1.0], [-1.0, -1.0]], dtype=torch.float64)
    return torch.kron(core, one) + torch.kron((core == 0).to(torch.float64), zero)


def _rotated(x, b):
    """Rows of x rotated by I (x) H_b / sqrt(b), in 64 bits."""
    T, d = x.shape
    base = 1
    if b & (b - 1):
        base = b
        while base % 2 == 0:
            base //= 2
        base *= 4
    v = x.to(torch.float64).reshape(T, d // base, base)
    if base > 1:
        v = v @ _base_matrix(base).to(x.device)
    v = v.reshape(T, d)
    h = base
    while h < b:
        v = v.reshape(T, d // (2 * h), 2, h)
        v = torch.stack((v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]), 2).reshape(T, d)
        h *= 2
    return v / math.sqrt(b)


def exact(case, seed):
    """The fp32 outputs of `run` in 64 bits: scales and statistics.  Codes and shared exponents have no such value."""
    if case["call"] == "massdiff" or case.get("fmt") == "mxfp4":
        return None
    s = prepare(case, seed)
    b = case["b"]
    if case["call"] == "stats":
        x = s["x"] if s["perm"] is None else s["x"][:, s["perm"].long()]
        chan, block, token = torch.zeros(case["d"], dtype=torch.float64, device="cuda"), 0, []
        for x_raw, x_perm in zip(s["x"].split(1024), x.split(1024)):
            norms = x_perm.abs().to(torch.float64).reshape(x_perm.shape[0], -1, b).sum(2)
            chan, block = chan + x_raw.abs().to(torch.float64).sum(0), block + norms.sum(0)
            token.append(norms.max(1).values)
        return chan, block / case["T"], torch.cat(token)
    scales = []
    rows = zip(s["gate"].split(1024), s["up"].split(1024)) if case["call"] == "swiglu" else s["x"].split(1024)
    for x in rows:
        if case["call"] == "swiglu":
            g = x[0].to(torch.float64)
            x = (g / (1 + torch.exp(-g)) * x[1].to(torch.float64)).to(torch.bfloat16)
        elif s["perm"] is not None:
            x = x[:, s["perm"].long()]
        y = _rotated(x, b)
        if case["fmt"] == "int4_asym":
            lo = y.min(1).values
            step = (y.max(1).values - lo) / 15
            scales.append(torch.stack((step, torch.where(step > 0, torch.round(lo / step), torch.zeros_like(lo))), 1))
        else:
            scales.append(y.abs().reshape(y.shape[0], -1, case["group"] or case["d"]).max(2).values / 7)
    return None, torch.cat(scales)
