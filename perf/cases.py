"""The calls whose speed counts, over the range in which the library is used.

Five ways of calling the library, each with the shapes of the paper's workloads
and of this repository's configurations (synth/inputs.py, tests/, bench.py):

  layer     lbp_backward of one linear layer (Algorithm 1), outputs and workspace
            kept by the caller; `rank` = k*k is exact backpropagation
            (lbp_backward_fullrank).
  batch     lbp_backward_batch of the linear layers of one transformer block (or
            MLP), outputs and workspaces kept by the caller.
  micro     gradient accumulation over two micro-batches with lbp_backward_ex:
            (B, 1 + H*W, C) token sequences, the class token outside the grid,
            the bias gradient, g_W overwritten by the first and added to by the
            second micro-batch.
  module    forward and backward of LbpLinear with a bias: `sequence` on token
            sequences with a class token, else on a (B, H, W, C) grid with the
            projected activation saved at forward time.
  spectrum  lbp_spectrum of a gradient tensor: the profiling step of the
            low-heuristic-error selection of bases.
"""
import math

import torch

import paper_2309_15275_b200 as lbp

# --------------------------------------------------------------------- cases ----


def _layers(*pairs):
    return " ".join("%dx%d" % p for p in pairs)


def _pairs(text):
    return [tuple(int(v) for v in p.split("x")) for p in text.split()]


def listed():
    case = lambda name, call, layers, B, H, W, k, rank, dtype="bf16", x="normal", **more: dict(  # noqa: E731
        name=name, call=call, layers=layers, B=B, H=H, W=W, k=k, rank=rank, dtype=dtype, x=x, **more)
    return [
        # the smallest call: one narrow fp32 layer on two images, where the host's
        # share and the number of launches decide
        case("tiny_fp32", "layer", "64x64", 2, 16, 16, 8, 4, "fp32"),
        # fp32 training of the last linear layers of a small network on 7 x 7 maps
        # (the paper's latency table: 448 -> 1792, 49 tokens; LP_L1-4)
        case("last_linear_fp32", "layer", "448x1792", 64, 7, 7, 8, 10, "fp32"),
        # the same layers in bf16 as a module with a small batch, x_hat saved (LP_L1-2, order 4)
        case("last_linear_module", "module", "448x1792", 16, 7, 7, 4, 3, sequence=False),
        # early-stage MLP: few channels, many tokens, GELU activations
        case("early_stage_mlp", "batch", _layers((48, 192), (192, 48)), 64, 56, 56, 8, 8, x="gelu"),
        # the four linear layers of a ViT-B block: the repository's benchmark
        case("vitb_block_r8", "batch", _layers((768, 2304), (768, 768), (768, 3072), (3072, 768)),
             128, 16, 16, 8, 8),
        # the same block at twice the rank (more accuracy for more work)
        case("vitb_block_r16", "batch", _layers((768, 2304), (768, 768), (768, 3072), (3072, 768)),
             128, 16, 16, 8, 16),
        # ViT-L MLP at high resolution, heavy-tailed activations
        case("vitl_mlp_r6", "batch", _layers((1024, 4096), (4096, 1024)), 32, 32, 32, 8, 6, x="student"),
        # one wide layer on large maps at the highest rank of the paper's tables (LP_L1-8)
        case("wide_layer_r36", "layer", "768x3072", 16, 64, 64, 8, 36),
        # two accumulated micro-batches of ViT token sequences, one order-16 transform
        # over the whole 14 x 14 map (LP_L1-6)
        case("micro_batches_k16", "micro", "768x3072", 32, 14, 14, 16, 21),
        # training step of a ViT linear layer as a module: class token, bias, LP_L1-4
        case("vit_module_r10", "module", "768x3072", 64, 14, 14, 8, 10, sequence=True),
        # exact backpropagation of a ViT-B layer (what the low rank is weighed against)
        case("vitb_fc1_exact", "layer", "768x3072", 32, 16, 16, 8, 64),
        # profiling of a gradient tensor for the selection of bases
        case("spectrum_k8", "spectrum", "768x768", 128, 16, 16, 8, 64),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _channels(rng, lo, hi):
    """Mostly multiples of 64 as in real networks, some of 8 only."""
    step = 8 if rng.random() < 0.25 else 64 if hi > 64 else 16
    return max(step, int(round(_log(rng, lo, hi) / step)) * step)


def _rank(rng, k):
    """The ranks of the paper's sets (LP_L1-m: m(m+1)/2) and those in between."""
    most = min(k * k - 1, 36)
    if rng.random() < 0.5:
        return rng.choice([v for v in (1, 3, 6, 10, 15, 21, 28, 36) if v <= most])
    return max(1, min(most, int(round(_log(rng, 1, most)))))


def draw(rng):
    call = rng.choice(["layer", "layer", "layer", "batch", "batch", "micro", "module", "module",
                       "exact", "spectrum"])
    dtype = "fp32" if call in ("layer", "module", "spectrum", "exact") and rng.random() < 0.2 else "bf16"
    k = rng.choice([4, 8, 8, 16])
    case = {"call": "layer" if call == "exact" else call, "k": k, "dtype": dtype,
            "x": rng.choice(["normal", "normal", "gelu", "student"])}
    if call == "batch":
        d = _channels(rng, 48, 1024)
        if rng.random() < 0.5:
            case["layers"] = _layers((d, 4 * d), (4 * d, d))
        else:
            case["layers"] = _layers((d, 3 * d), (d, d), (d, 4 * d), (4 * d, d))
    else:
        a, b = _channels(rng, 48, 1024), rng.choice([1, 1, 3, 4])
        case["layers"] = "%dx%d" % ((a, a * b) if rng.random() < 0.6 else (a * b, a))
    side = rng.choice([7, 14, 16, 24, 28, 32, int(_log(rng, 5, 64))])
    case["H"] = side
    case["W"] = side if rng.random() < 0.7 else max(4, int(side * rng.uniform(0.6, 1.6)))
    # tokens: from a few hundred to the largest listed case, bounded by its work
    case["rank"] = k * k if call in ("exact", "spectrum") else _rank(rng, k)
    case["B"] = 1
    one = work(case)
    most_bytes, most_flops = (1.1e9, 2.0e11) if dtype == "bf16" else (2.0e8, 2.0e9)
    most = min(128.0, most_bytes / one["bytes"], most_flops / max(one["flops"], 1.0))
    case["B"] = max(1, int(_log(rng, 1.0, max(most, 1.01))))
    if call == "module":
        case["sequence"] = rng.random() < 0.5
    return case


# -------------------------------------------------------------- inputs, state ----


def _dtype(case):
    return torch.float32 if case["dtype"] == "fp32" else torch.bfloat16


def _values(gen, shape, kind, scale, dtype):
    normal = lambda: torch.randn(shape, generator=gen, device="cuda")  # noqa: E731
    if kind == "gelu":
        v = torch.nn.functional.gelu(normal())
    elif kind == "student":                  # 4 degrees of freedom
        chi2 = normal().square_()
        for _ in range(3):
            chi2 += normal().square_()
        v = normal() * torch.rsqrt(chi2 / 4.0)
    else:
        v = normal()
    return (v if scale == 1.0 else v * scale).to(dtype)


def _bases(case):
    return lbp.lbp_select_bases(case["k"], lbp.SEL_PREFIX, case["rank"])


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dt, k, rank = _dtype(case), case["k"], case["rank"]
    B, H, W = case["B"], case["H"], case["W"]
    pairs, call = _pairs(case["layers"]), case["call"]
    cin, cout = pairs[0]
    s = {"case": case, "k": k, "rank": rank, "bases": _bases(case)}
    if call in ("layer", "batch"):
        s["x"] = [_values(gen, (B, H, W, i), case["x"], 1.0, dt) for i, _ in pairs]
        s["g_y"] = [_values(gen, (B, H, W, o), "normal", 0.01, dt) for _, o in pairs]
        s["w"] = [_values(gen, (o, i), "normal", i ** -0.5, dt) for i, o in pairs]
        s["g_x"] = [torch.empty_like(x) for x in s["x"]]
        s["g_w"] = [torch.empty((o, i), dtype=torch.float32, device="cuda") for i, o in pairs]
        s["ws"] = [lbp.alloc_workspace(x, g, k, rank) for x, g in zip(s["x"], s["g_y"])]
    elif call == "micro":
        n = 1 + H * W
        s["x"] = [_values(gen, (B, n, cin), case["x"], 1.0, dt) for _ in range(2)]
        s["g_y"] = [_values(gen, (B, n, cout), "normal", 0.01, dt) for _ in range(2)]
        s["w"] = _values(gen, (cout, cin), "normal", cin ** -0.5, dt)
        s["g_x"] = [torch.empty_like(x) for x in s["x"]]
        s["g_w"] = torch.empty((cout, cin), dtype=torch.float32, device="cuda")
        s["g_b"] = torch.empty((cout,), dtype=torch.float32, device="cuda")
    elif call == "module":
        seq = case["sequence"]
        shape = (B, 1 + H * W) if seq else (B, H, W)
        s["x"] = _values(gen, shape + (cin,), case["x"], 1.0, dt).requires_grad_()
        s["g_y"] = _values(gen, shape + (cout,), "normal", 0.01, dt)
        s["module"] = lbp.LbpLinear(cin, cout, k, s["bases"], device="cuda", dtype=dt, bias=True,
                                    save_projected=not seq, grid=(H, W) if seq else None)
        with torch.no_grad():
            s["module"].weight.copy_(_values(gen, (cout, cin), "normal", cin ** -0.5, dt))
            s["module"].bias.copy_(_values(gen, (cout,), "normal", 0.1, dt))
    else:
        s["t"] = _values(gen, (B, H, W, cout), "normal", 0.01, dt)
    return s


def run(s):
    case, k, bases = s["case"], s["k"], s["bases"]
    call = case["call"]
    if call == "layer":
        x, g_y, w, g_x, g_w, ws = (s[n][0] for n in ("x", "g_y", "w", "g_x", "g_w", "ws"))
        if s["rank"] == k * k:
            return lbp.lbp_backward_fullrank(x, g_y, w, k, g_x=g_x, g_W=g_w, ws=ws)
        return lbp.lbp_backward(x, g_y, w, k, bases, g_x=g_x, g_W=g_w, ws=ws)
    if call == "batch":
        return lbp.lbp_backward_batch(s["x"], s["g_y"], s["w"], k, bases, g_xs=s["g_x"], g_Ws=s["g_w"],
                                      wss=s["ws"])
    if call == "micro":
        grid = (case["H"], case["W"])
        for i, (x, g_y, g_x) in enumerate(zip(s["x"], s["g_y"], s["g_x"])):
            lbp.lbp_backward_ex(x[:, 1:].unflatten(1, grid), g_y[:, 1:].unflatten(1, grid), s["w"], k, bases,
                                beta=0.0 if i == 0 else 1.0, g_bias=s["g_b"], x_extra=x[:, 0],
                                gy_extra=g_y[:, 0], gx_extra=g_x[:, 0], g_W=s["g_w"],
                                g_x=g_x[:, 1:].unflatten(1, grid))
        return s["g_x"], s["g_w"], s["g_b"]
    if call == "module":
        m = s["module"]
        s["x"].grad = m.weight.grad = m.bias.grad = None
        y = m(s["x"])
        y.backward(s["g_y"])
        return y, s["x"].grad, m.weight.grad, m.bias.grad
    return lbp.lbp_spectrum(s["t"], k)


# ----------------------------------------------------------- work, tolerances ----


def work(case):
    """Every input read and every output written once; multiply-adds of the two
    gradient products (and of the forward product of a module).  The transforms
    are additions and are not counted, nor is anything kept in between."""
    es = 4 if case["dtype"] == "fp32" else 2
    k, call = case["k"], case["call"]
    grid = case["B"] * case["H"] * case["W"]
    blocks = case["B"] * -(-case["H"] // k) * -(-case["W"] // k)
    rows = grid if case["rank"] == k * k else min(blocks * case["rank"], grid)
    pairs = _pairs(case["layers"])
    if call == "spectrum":
        return {"bytes": float(es * grid * pairs[0][1] + 8 * k * k), "flops": 0.0}
    extra = case["B"] if call == "micro" or case.get("sequence") else 0
    tokens = grid + extra
    nbytes = flops = 0.0
    for cin, cout in pairs:
        gw = es if call == "module" else 4
        once = es * tokens * (2 * cin + cout)
        flops_1 = 4.0 * cin * cout * (rows + extra)
        if call == "micro":
            once, flops_1 = 2 * once, 2 * flops_1
        nbytes += once + (es + gw) * cin * cout
        flops += flops_1
        if call in ("micro", "module"):
            nbytes += 4 * cout
        if call == "module":        # forward: y written, the bias read
            nbytes += es * tokens * cout + es * cout
            flops += 2.0 * tokens * cin * cout
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Errors against the same call in 64 bits, measured over the listed and some drawn
    # cases, and the bound of about four times that:
    if case["call"] == "spectrum":
        # exact responses (bf16) or 32-bit ones, squares added in 32 bits over short
        # runs and in 64 beyond: 1e-8; runs a few times longer would show 1e-7
        return {"rel": 5e-7}
    if case["dtype"] == "fp32":
        return {"rel": 4e-6}      # 32-bit sums over up to a few thousand terms: 1e-6
    # one rounding of the coefficients and one of the results: 2.9e-3
    return {"rel": 1e-2}
