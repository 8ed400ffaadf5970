"""The work a user of this library has it do, as a list of cases that can be timed and compared.

Online: ``tardis_ffn_forward`` from one token (a decoding step) to a whole prompt chunk, on the layer shapes of
``workloads.CONFIGS``, and ``tardis_stack_forward`` (a decoding step through consecutive layers).  Offline, once per
layer: the quantile calibration, Algorithm 1's range search with the neuron-level thresholds, and the building of a
layer (GPTQ predictor, constant folding).  ``listed()`` names one case for each; ``draw()`` gives others of the same
ranges.  Weights and tokens are seeded stand-ins with the structure of ``workloads/generate.py``: weights
N(0, 0.02^2), layer-normalised heavy-tailed tokens, per-neuron ranges between the q and 1 - q quantiles of
calibration pre-activations, least-squares fits, round-to-nearest predictor codes.
"""
import math
from statistics import NormalDist

import torch

import paper_2501_10054_b200 as T

ACTS = {"tanh": T.TARDIS_ACT_GELU_TANH, "erf": T.TARDIS_ACT_GELU_ERF, "relu": T.TARDIS_ACT_RELU}
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


# ---- the cases --------------------------------------------------------------------------------------------------
def _forward(d, h, n, dtype="bf16", group=128, bits=2, q=0.034, act="tanh", bias=True, outliers=False):
    """One call of tardis_ffn_forward on n tokens.  q = 0.034 flags about 10 % of the neurons with 2-bit codes."""
    return dict(kind="forward", d=d, h=h, n=n, dtype=dtype, group=group, bits=bits, q=q, act=act, bias=bias, outliers=outliers)


def _falcon(n, q):
    return _forward(4544, 18176, n, group=64, q=q, bias=False, outliers=True)


def listed():
    return [
        # the tiny fp32 layer: a call that is all latency and launches
        dict(_forward(256, 1024, 64, dtype="f32", group=64, q=0.05), name="tiny_f32_64_tokens"),
        # one decoding step of one sequence: the headline
        dict(_forward(4096, 16384, 1), name="decode_7b_1_token"),
        # decoding steps of a few, some and many sequences at once (continuous batching)
        dict(_falcon(4, 0.05), name="falcon_7b_4_tokens"),
        dict(_forward(4096, 16384, 16), name="decode_7b_16_tokens"),
        dict(_falcon(64, 0.05), name="falcon_7b_64_tokens"),
        # the same on the wide layer
        dict(_forward(8192, 32768, 1), name="large_8k_1_token"),
        dict(_forward(8192, 32768, 32), name="large_8k_32_tokens"),
        # prompts: 8 sequences of 2048 tokens through one layer
        dict(_forward(4096, 16384, 16384), name="prefill_7b_16384_tokens"),
        # a decoding step through consecutive layers with normalisation and residual stream
        dict(_forward(4096, 16384, 1), kind="stack", layers=4, name="stack_4_layers_1_token"),
        # offline, per layer: pre-activations of the calibration tokens, quantile ranges and fits
        dict(kind="calibrate", d=4096, h=16384, n=2048, q=0.05, act="tanh", bias=True, name="calibrate_7b"),
        # offline, per layer: range search at the layer's threshold, neuron-level thresholds, range search with them
        dict(kind="search", h=16384, n=2048, threshold=0.85, step=0.05, act="tanh", bias=True, name="range_search_7b"),
        # offline, per layer: the GPTQ predictor, then the fold
        dict(kind="build", d=4096, h=16384, dtype="bf16", group=128, bits=2, q=0.034, act="tanh", bias=True, name="build_7b"),
    ]


def _log_int(rng, lo, hi, multiple=1):
    """A whole number, spread evenly over the logarithm of [lo, hi], rounded to the multiple."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi, max(lo, int(round(v / multiple)) * multiple))


def draw(rng):
    kind = rng.choice(["decode"] * 6 + ["prefill", "f32", "stack", "calibrate", "search", "build"])
    act = rng.choice(["tanh", "tanh", "erf", "relu"])
    bias = rng.random() < 0.7
    q = round(rng.uniform(0.02, 0.15), 4)
    group = rng.choice([64, 128])
    ratio = rng.choice([3, 4, 4, 4, 5])
    if kind == "f32":
        d = _log_int(rng, 64, 1024, 32)
        return _forward(d, min(4096, ratio * d), _log_int(rng, 1, 256), "f32", rng.choice([16, 32]), 2, q, act, bias)
    if kind == "calibrate":
        d = _log_int(rng, 512, 4096, 8)
        return dict(kind="calibrate", d=d, h=min(16384, 4 * d), n=_log_int(rng, 200, 2048), q=q, act=act, bias=bias)
    if kind == "search":
        return dict(kind="search", h=_log_int(rng, 1024, 16384, 32), n=_log_int(rng, 200, 2048), threshold=round(rng.uniform(0.7, 0.95), 3),
                    step=round(rng.uniform(0.02, 0.1), 3), act=act, bias=bias)
    if kind == "build":
        d = _log_int(rng, 512, 4096, group)
        return dict(kind="build", d=d, h=min(16384, ratio * d), dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]) if d <= 1024 else "bf16",
                    group=group, bits=rng.choice([2, 2, 3, 4]), q=q, act=act, bias=bias)
    d = _log_int(rng, 512, 8192, group)
    h = min(32768, ratio * d)
    bits = rng.choice([2, 2, 2, 2, 2, 4])
    more = dict(group=group, bits=bits, q=q, act=act, bias=bias, outliers=rng.random() < 0.5)
    if kind == "stack":
        d = _log_int(rng, 512, 4096, group)
        more["bits"] = 2
        return dict(_forward(d, ratio * d, _log_int(rng, 1, 16), **more), kind="stack", layers=rng.randint(2, 4))
    if kind == "decode":
        return _forward(d, h, _log_int(rng, 1, 128), **more)
    most = 16384 * 4096 * 16384 // (d * h)                    # no more work than the listed prompt chunk
    return _forward(d, h, _log_int(rng, 129, min(16384, most)), **more)


# ---- inputs -----------------------------------------------------------------------------------------------------
def _tokens(n, d, dtype, gen, outliers):
    """Layer-normalised Student-t (4 degrees of freedom) tokens; with `outliers` half of them Gaussian and 1 % of the
    channels 20 times as large."""
    z = torch.randn(n, d, generator=gen, device="cuda")
    chi = torch.zeros(n, d, device="cuda")
    for _ in range(4):
        chi += torch.randn(n, d, generator=gen, device="cuda").square_()
    x = z / torch.sqrt(chi / 4)
    if outliers:
        x = torch.where(torch.rand(n, 1, generator=gen, device="cuda") < 0.5, z, x)
    x = torch.nn.functional.layer_norm(x, (d,), eps=1e-5)
    if outliers:
        x[:, torch.arange(0, d, 100, device="cuda")] *= 20.0
    return x.to(DTYPES[dtype])


def _activation(z, act):
    if act == "relu":
        return torch.relu(z)
    return torch.nn.functional.gelu(z, approximate="tanh" if act == "tanh" else "none")


def _weights(case, gen):
    d, h, dt = case["d"], case["h"], DTYPES[case.get("dtype", "bf16")]
    s = {"W1": (torch.randn(h, d, generator=gen, device="cuda") * 0.02).to(dt),
         "W2": (torch.randn(d, h, generator=gen, device="cuda") * 0.02).to(dt), "b1": None, "b2": None}
    if case["bias"]:
        s["b1"] = torch.randn(h, generator=gen, device="cuda") * 0.01
        s["b2"] = torch.randn(d, generator=gen, device="cuda") * 0.01
    return s


def _ranges_and_fits(case, s, xcal):
    """lo, hi: the q and 1 - q quantiles of every neuron's calibration pre-activations; a, c: least squares inside."""
    z = xcal.float() @ s["W1"].float().t()
    if s["b1"] is not None:
        z += s["b1"]
    zs = z.sort(dim=0).values
    k = int(case["q"] * (z.shape[0] - 1))
    lo, hi = zs[k].contiguous(), zs[z.shape[0] - 1 - k].contiguous()
    inside = ((z >= lo) & (z < hi)).float()
    cnt = inside.sum(0)
    g = _activation(z, case["act"])
    mz, mg = (inside * z).sum(0) / cnt, (inside * g).sum(0) / cnt
    dz = (z - mz) * inside
    a = (dz * (g - mg)).sum(0) / dz.square().sum(0)
    s.update(lo=lo, hi=hi, a=a, c=mg - a * mz)


def _codes(case, s):
    """Round-to-nearest codes on the grid of every neuron and group, as one bit stream per row."""
    h, d, G, bits = case["h"], case["d"], case["group"], case["bits"]
    top = (1 << bits) - 1
    w = s["W1"].float().view(h, d // G, G)
    lowest, highest = w.amin(-1).clamp(max=0.0), w.amax(-1).clamp(min=0.0)
    scale = ((highest - lowest) / top).to(s["W1"].dtype)
    zero = torch.round(-lowest / scale.float()).clamp(0, top)
    code = torch.round(w / scale.float()[..., None] + zero[..., None]).clamp(0, top).to(torch.int64)
    per = 32 // bits
    word = (code.view(h, d // per, per) << (bits * torch.arange(per, device="cuda"))).sum(-1)
    s.update(codes=torch.where(word >= 2 ** 31, word - 2 ** 32, word).to(torch.int32), scale=scale.contiguous(), zero=zero.to(torch.uint8))


class _Handle:
    """A folded layer that is given back with the state that holds it."""

    def __init__(self, case, s):
        self.value = T.tardis_fold(s["W1"], s["W2"], s["lo"], s["hi"], s["a"], s["c"], s["codes"], s["scale"], s["zero"], case["group"],
                                   b1=s["b1"], b2=s["b2"], act=ACTS[case["act"]], pred_bits=case["bits"])

    def __del__(self):
        T.tardis_destroy(self.value)


def _layer(case, gen):
    s = _weights(case, gen)
    _ranges_and_fits(case, s, _tokens(512, case["d"], case["dtype"], gen, case["outliers"]))
    _codes(case, s)
    return _Handle(case, s)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, state = case["kind"], {"case": case}
    if kind in ("forward", "stack"):
        n, d = case["n"], case["d"]
        state["handles"] = [_layer(case, gen) for _ in range(case.get("layers", 1))]
        state["x"] = _tokens(n, d, case["dtype"], gen, case["outliers"])
        state["y"] = torch.empty_like(state["x"])
        if kind == "stack":
            state["work"] = torch.empty(2, n, d, dtype=state["x"].dtype, device="cuda")
            state["gammas"] = [1.0 + 0.1 * torch.randn(d, generator=gen, device="cuda") for _ in state["handles"]]
            state["betas"] = [0.1 * torch.randn(d, generator=gen, device="cuda") for _ in state["handles"]]
    elif kind == "calibrate":
        state.update(_weights(case, gen), x=_tokens(case["n"], case["d"], "bf16", gen, False),
                     z=torch.empty(case["h"], case["n"], device="cuda"))
    elif kind == "search":
        # pre-activations as W1 of a 4096-channel layer gives them: every neuron nearly Gaussian, with a spread of its own
        h, n = case["h"], case["n"]
        spread = 1.28 * (1.0 + 0.1 * torch.randn(h, 1, generator=gen, device="cuda"))
        state["z"] = torch.randn(h, n, generator=gen, device="cuda") * spread
        state["b1"] = torch.randn(h, generator=gen, device="cuda") * 0.01 if case["bias"] else None
    else:
        d = case["d"]
        state.update(_weights(case, gen))
        x = _tokens(1024, d, case["dtype"], gen, False)
        _ranges_and_fits(case, state, x)
        H = (2.0 / x.shape[0]) * (x.double().t() @ x.double())
        H += 0.01 * H.diagonal().mean() * torch.eye(d, dtype=H.dtype, device="cuda")
        # the upper Cholesky factor of the inverse Hessian
        state["U"] = torch.linalg.cholesky(torch.cholesky_inverse(torch.linalg.cholesky(H)), upper=True).contiguous()
        state["Wf"] = torch.empty(d, d, dtype=state["W1"].dtype, device="cuda")
        state["bf"] = torch.empty(d, device="cuda")
    return state


# ---- one pass ---------------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "forward":
        return T.tardis_ffn_forward(state["handles"][0].value, state["x"], state["y"])
    if kind == "stack":
        T.tardis_stack_forward([hd.value for hd in state["handles"]], state["x"], state["y"], state["gammas"], state["betas"],
                               work=state["work"])
        return state["y"]
    act = ACTS[case["act"]]
    if kind == "calibrate":
        z = T.tardis_gemm_bf16(state["W1"], state["x"], state["z"])
        return T.tardis_calibrate(z, state["b1"], case["q"], 1.0 - case["q"], act)
    if kind == "search":
        z, b1, t, step = state["z"], state["b1"], case["threshold"], case["step"]
        lo, hi, _, _ = T.tardis_range_search(z, b1, t, step, act)
        err, thresholds = T.tardis_neuron_thresholds(z, b1, lo, hi, act, t, t - 0.1, min(1.0, t + 0.1))
        return (lo, hi, err, thresholds) + T.tardis_range_search(z, b1, thresholds, step, act, want_steps=True)
    s = state
    codes, scale, zero = T.tardis_build_predictor(s["W1"], s["U"], case["bits"], case["group"])
    handle = T.tardis_fold(s["W1"], s["W2"], s["lo"], s["hi"], s["a"], s["c"], codes, scale, zero, case["group"],
                           b1=s["b1"], b2=s["b2"], act=act, pred_bits=case["bits"])
    T.tardis_export_folded(handle, s["Wf"], s["bf"])
    T.tardis_destroy(handle)
    return codes, scale, zero, s["Wf"], s["bf"]


# ---- what a pass cannot do without ------------------------------------------------------------------------------
def _flagged(case):
    """Expected share of flagged neurons: both tails at q, widened by the rounding noise of the predictor."""
    return 2.0 * NormalDist().cdf(NormalDist().inv_cdf(case["q"]) / (1.1 if case["bits"] == 2 else 1.01))


def work(case):
    kind, h, n = case["kind"], case["h"], case.get("n", 0)
    if kind == "search":                     # three calls read the samples; an activation and some sums per sample
        return {"bytes": 3 * 4 * h * n + 44 * h, "flops": 3 * 40 * h * n}
    d = case["d"]
    size = 4 if case.get("dtype") == "f32" else 2
    if kind == "calibrate":                  # the pre-activations pass through memory between the two calls
        return {"bytes": 2 * d * (h + n) + 8 * h * n + 20 * h, "flops": 2 * h * d * n + 40 * h * n}
    predictor = h * d * case["bits"] // 8 + h * (d // case["group"]) * (size + 1)
    if kind == "build":                      # W1, W2, the triangle of U, the tables; the predictor, W_f and b_f
        return {"bytes": 2 * size * h * d + 4 * d * d + 20 * h + predictor + size * d * d + 8 * d,
                "flops": h * d * d + 2 * h * d * d}
    f = _flagged(case)
    union = h * (1.0 - (1.0 - f) ** n)       # neurons whose W1 row and W2 column some token needs
    layers = case.get("layers", 1)
    return {"bytes": layers * (size * d * d + predictor + union * 2 * d * size + 12 * h + 8 * union + 4 * d + 2 * n * d * size),
            "flops": layers * n * (2 * h * d + 2 * d * d + f * h * 4 * d)}


def tolerance(case):
    if case["kind"] in ("calibrate", "search") or (case["kind"] == "forward" and case["dtype"] == "f32"):
        return {"rel": 1e-5}                 # float32 results of wider sums; step counts are whole numbers
    if case["kind"] == "build":              # codes are whole words, bit for bit; W_f is rounded once to its type
        return {"rel": 4e-3 if case["dtype"] == "bf16" else 1e-5}
    return {"rel": 1e-2}
