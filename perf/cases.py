"""The calls that window-attention programs make of this framework, as timed cases.

A case is one forward call of the public Python entry points on tensors that
are already on the GPU: ``nystra`` (plain attention), ``pool_bias`` with
``nystra_biased`` (relative-position bias, shifted-window masks), ``nystra_qkv``
(projections fused in), ``project_qkv`` followed by ``nystra`` (the two-pass
form) and ``exact`` (the attention the method stands in for).  The path is
forward only: it serves pretrained restoration models and has no backward.

Sizes are those of ``paper_2506_08520_gb300/workloads.py`` and of the tests:
8x8, 16x16 and 32x32 windows of feature maps between 64x64 and 1280x720, one
to eight heads of 30 or 32 features, 8 to 64 landmarks, 4 to 6 iterations, in
bf16, fp16 and fp32, and windows of other sizes (12x12 and the like), whose
token count, head width or landmark count is no power of two.
"""
import math

import torch

from paper_2506_08520_gb300 import binding

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _case(name, op, dtype, windows, heads, N, d, m=16, iters=6, landmarks="segments", factors="pairs", bias="",
          inputs="normal"):
    c = {"op": op, "dtype": dtype, "windows": windows, "heads": heads, "N": N, "d": d, "m": m, "iters": iters,
         "landmarks": landmarks, "factors": factors, "bias": bias, "inputs": inputs}
    return {"name": name, **c} if name else c


def listed():
    return [
        # One 64x64 crop of an fp32 model, 8x8 windows: the smallest call, all latency.
        _case("crop64-w8-f32", "nystra", "f32", 64, 6, 64, 30),
        # Denoising a 256x256 image in bf16, 8x8 windows: the ordinary call of the small-window models.
        _case("img256-w8-bf16", "nystra", "bf16", 1024, 6, 64, 30),
        # The same layer given as tokens, weights and biases, as a model's attention module holds them.
        _case("img256-w8-qkv-bf16", "qkv", "bf16", 1024, 6, 64, 30, bias="heads"),
        # Super-resolving a 1280x720 map, 16x16 and 32x32 windows: the largest calls, bound by memory.
        _case("hd-w16-bf16", "nystra", "bf16", 3600, 6, 256, 30),
        _case("hd-w32-f16", "nystra", "f16", 920, 6, 1024, 30),
        # The same map through the projection and then the attention.
        _case("hd-w32-project-bf16", "project", "bf16", 920, 6, 1024, 30),
        # Wide landmark sets for accuracy on correlated tokens: 16x16 windows with 64, 32x32 with 32 landmarks.
        _case("large-w16-m64-bf16", "nystra", "bf16", 1024, 4, 256, 32, m=64, inputs="lowrank"),
        _case("large-w32-m32-bf16", "nystra", "bf16", 256, 4, 1024, 32, m=32, inputs="lowrank"),
        # An fp32 model on 16x16 windows of a 512x512 image.
        _case("img512-w16-f32", "nystra", "f32", 1024, 6, 256, 30),
        # 12x12 windows with square patches: a window size that is no power of two (1849 windows of a padded 512x512).
        _case("img512-w12-f16", "nystra", "f16", 1849, 6, 144, 30, landmarks="patches"),
        # A relative-position bias on 16x16 windows of the 1280x720 map.
        _case("hd-w16-bias-bf16", "biased", "bf16", 3600, 6, 256, 30, bias="heads"),
        # The exact attention of the same layer, which programs compare and fall back to.
        _case("img512-w16-exact-bf16", "exact", "bf16", 1024, 6, 256, 30),
    ]


# No drawn case is larger than the largest listed one, in bytes or in operations.
_MOST_BYTES, _MOST_FLOPS = 1.4e9, 7.5e10


def draw(rng):
    while True:
        c = _draw(rng)
        w = work(c)
        if w["bytes"] <= _MOST_BYTES and w["flops"] <= _MOST_FLOPS:
            return c


def _draw(rng):
    op = rng.choices(["nystra", "biased", "qkv", "project", "exact"], [10, 3, 3, 2, 3])[0]
    square = rng.random() < (0.75 if op in ("nystra", "exact") else 1.0)
    dtype = rng.choices(["f32", "bf16", "f16"], [3, 5, 3])[0]
    if op in ("qkv", "project") and dtype == "f32":
        dtype = "bf16"  # 16-bit tokens and weights only
    landmarks = "segments"
    if square:  # the windows the models use
        w = rng.choice([8, 16, 32])
        d = rng.choice([30, 30, 32, 32, 16, 24, 28])
        if op in ("qkv", "project"):
            m = rng.choice([8, 16, 16, 32]) if w == 32 else rng.choice([8, 16, 16])
        else:
            m = rng.choices([8, 16, 32, 64], [3, 6, 3, 2])[0]
        if m == 16 and rng.random() < 0.25:
            landmarks = "patches"
    else:  # other windows: any token count, head width and landmark count
        w = rng.choice([6, 7, 9, 10, 12, 14, 20, 24, 28])
        d = rng.choice([16, 20, 30, 32, 33, 40, 48, 64])
        m = rng.choice([k for k in range(4, 49) if w * w % k == 0])
        grids = [p * p for p in range(2, 7) if w % p == 0]
        if grids and rng.random() < 0.3:
            landmarks, m = "patches", rng.choice(grids)
    N = w * w
    heads = rng.choice([1, 2, 3, 4, 6, 6, 8])
    windows = max(1, round(math.exp(rng.uniform(math.log(8), math.log(6e6 / N)))))
    bias = ""
    if op == "biased":
        m = min(m, 32)
        # masks of shifted windows come per window, for small windows
        bias = "windows" if w == 8 and rng.random() < 0.4 else "heads"
    if op in ("qkv", "project"):
        bias = rng.choice(["", "heads"]) if op == "qkv" and m <= 16 else ""
    factors = "16" if dtype != "f32" and op != "exact" and rng.random() < 0.15 else "pairs"
    inputs = "lowrank" if op == "nystra" and rng.random() < 0.2 else "normal"
    return _case(None, op, dtype, windows, heads, N, d, m, rng.choice([4, 5, 6, 6, 6]), landmarks, factors, bias, inputs)


# ---------------------------------------------------------------- inputs
def _normal(shape, g, dtype, scale=1.0):
    x = torch.empty(shape, device="cuda", dtype=torch.float32)
    x.normal_(generator=g)
    return (x.mul_(scale) if scale != 1.0 else x).to(DTYPES[dtype])


def _qkv(case, g):
    """Q, K, V of about unit logits: independent tokens, or tokens near an 8-dimensional subspace of each head."""
    nw, h, N, d = (case[k] for k in ("windows", "heads", "N", "d"))
    if case["inputs"] == "normal":
        return tuple(_normal((nw, h, N, d), g, case["dtype"]) for _ in range(3))
    out = []
    for _ in range(2):
        basis = _normal((h, 8, d), g, "f32", 8.0 ** -0.5)
        x = torch.matmul(_normal((nw, h, N, 8), g, "f32"), basis)
        out.append(x.add_(_normal((nw, h, N, d), g, "f32", 0.1)).to(DTYPES[case["dtype"]]))
    return out[0], out[1], _normal((nw, h, N, d), g, case["dtype"])


def _bias(case, g):
    """Relative-position bias [heads, N, N] from a table of offsets; with "windows" every other window of a head also
    has a shifted window's mask (-100 between its two halves): [windows, heads, N, N]."""
    h, N = case["heads"], case["N"]
    w = math.isqrt(N)
    table = _normal((h, (2 * w - 1) ** 2), g, "f32", 0.5)
    t = torch.arange(N, device="cuda")
    r, c = t // w, t % w
    B = table[:, (r[:, None] - r[None, :] + w - 1) * (2 * w - 1) + c[:, None] - c[None, :] + w - 1]
    if case["bias"] == "windows":
        half = (c >= w // 2)
        mask = torch.zeros(case["windows"], 1, N, N, device="cuda")
        mask[::2] = torch.where(half[:, None] == half[None, :], 0.0, -100.0)
        B = B[None] + mask
    return B.contiguous()


def _tokens(case, g):
    nw, h, N, d = (case[k] for k in ("windows", "heads", "N", "d"))
    C = h * d
    return (_normal((nw, N, C), g, case["dtype"]), _normal((3 * C, C), g, case["dtype"], C ** -0.5),
            _normal((3 * C,), g, "f32", 0.1))


def _inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = {"case": case}
    if case["op"] in ("qkv", "project"):
        s["x"], s["w"], s["b"] = _tokens(case, g)
    else:
        s["q"], s["k"], s["v"] = _qkv(case, g)
    if case["bias"]:
        s["bias"] = _bias(case, g)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    if case["bias"]:  # a model pools its bias once
        s["pooled"] = binding.pool_bias(s.pop("bias"), case["m"], case["landmarks"])
    return s


def run(state):
    c = state["case"]
    kw = {"m": c["m"], "iters": c["iters"], "landmarks": c["landmarks"], "factors": c["factors"]}
    if c["op"] == "nystra":
        return binding.nystra(state["q"], state["k"], state["v"], **kw)
    if c["op"] == "biased":
        return binding.nystra_biased(state["q"], state["k"], state["v"], state["pooled"], **kw)
    if c["op"] == "qkv":
        return binding.nystra_qkv(state["x"], state["w"], c["heads"], b_qkv=state["b"], pooled=state.get("pooled"), **kw)
    if c["op"] == "project":
        q, k, v = binding.project_qkv(state["x"], state["w"], c["heads"], state["b"])
        return binding.nystra(q, k, v, **kw)
    return binding.exact(state["q"], state["k"], state["v"])


# ---------------------------------------------------------------- work and results
def work(case):
    """Bytes: inputs read once, the output written once (and Q, K, V stored and read again by the two-pass form).
    Operations: the projections, the products of the method with its m x m iteration, or of exact attention."""
    nw, h, N, d, m = (case[k] for k in ("windows", "heads", "N", "d", "m"))
    es = 4 if case["dtype"] == "f32" else 2
    units, C = nw * h, h * d
    t = units * N * d * es
    if case["op"] == "exact":
        return {"bytes": 4 * t, "flops": 4 * units * N * N * d}
    flops = units * (8 * N * m * d + 2 * m * m * d + case["iters"] * 8 * m ** 3 + 2 * m * m * (d + 1))
    if case["op"] in ("qkv", "project"):
        proj = 2 * nw * N * C * 3 * C
        return {"bytes": (2 if case["op"] == "qkv" else 8) * t + 3 * C * C * es + 12 * C, "flops": flops + proj}
    bias = units if case["bias"] == "windows" else h if case["bias"] else 0
    return {"bytes": 4 * t + bias * (2 * N * m + m * m) * 4, "flops": flops}


def tolerance(case):
    # 16-bit results carry the rounding of the output (0.2% in bf16, 0.02% in fp16) and, amplified by the landmark
    # block's conditioning, that of the derived factors and of stored projections; fp32 ones that of 16-bit pairs
    # (exact attention, 8x8 windows with few landmarks) or of fp32 sums.
    if case["op"] == "exact":
        return {"rel": {"f32": 4e-5, "bf16": 1e-2, "f16": 2e-3}[case["dtype"]], "max": 0.1}
    if case["factors"] == "16" or case["op"] in ("qkv", "project"):
        return {"rel": 2e-2, "max": 0.9}
    if case["dtype"] == "f32":
        return {"rel": 4e-5 if case["N"] == 64 and case["m"] <= 16 else 4e-6, "max": 1e-3}
    return {"rel": 7e-3 if case["dtype"] == "bf16" else 1e-3, "max": 0.5}


def _owner(N, m, landmarks):
    """Landmark of each token."""
    t = torch.arange(N, device="cuda")
    if landmarks == "segments":
        return t // (N // m)
    w, p = math.isqrt(N), math.isqrt(m)
    b = w // p
    return (t // w // b) * p + t % w // b


def _attend64(q, k, v, P, iters, bias):
    """Algorithm 1 in the stabilised form, float64, on [units, N, d]; P averages tokens into landmarks."""
    s = q.shape[-1] ** -0.5
    qb, kb = P @ q, P @ k
    SL, SU, SA = s * q @ kb.mT, s * qb @ k.mT, s * qb @ kb.mT
    if bias is not None:
        SL, SU, SA = SL + bias @ P.mT, SU + P @ bias, SA + P @ bias @ P.mT
    mU = SU.amax(-1, keepdim=True)
    GL, GU, A = (SL - SL.amax(-1, keepdim=True)).exp(), (SU - mU).exp(), (SA - mU).exp()
    Z = A.mT / (A.sum(-2).amax(-1) * A.sum(-1).amax(-1))[:, None, None]
    I = torch.eye(A.shape[-1], dtype=A.dtype, device=A.device)
    for _ in range(iters):
        X = A @ Z
        Z = 0.25 * Z @ (13 * I - X @ (15 * I - X @ (7 * I - X)))
    Y = GL @ Z
    return (Y @ (GU @ v)) / (Y @ GU.sum(-1, keepdim=True))


def exact(case, seed):
    s = _inputs(case, seed)
    nw, h, N, d, m = (case[k] for k in ("windows", "heads", "N", "d", "m"))
    owner = _owner(N, m, case["landmarks"])
    P = torch.nn.functional.one_hot(owner, m).double().mT / (N // m)
    out = torch.empty((nw, h, N, d), dtype=torch.float64, device="cuda")
    step = max(1, int(1.5e8) // (h * N * (N if case["op"] == "exact" or case["bias"] else max(4 * m, 2 * d))))
    for i in range(0, nw, step):
        if "x" in s:
            y = s["x"][i:i + step].double() @ s["w"].double().mT + s["b"].double()
            q, k, v = y.view(-1, N, 3, h, d).permute(2, 0, 3, 1, 4).reshape(3, -1, N, d)
        else:
            q, k, v = (s[n][i:i + step].double().view(-1, N, d) for n in "qkv")
        if case["op"] == "exact":
            o = ((q @ k.mT) * d ** -0.5).softmax(-1) @ v
        else:
            B = None
            if case["bias"] == "windows":
                B = s["bias"][i:i + step].double().view(-1, N, N)
            elif case["bias"]:
                B = s["bias"].double().repeat(q.shape[0] // h, 1, 1)
            o = _attend64(q, k, v, P, case["iters"], B)
        out[i:i + step] = o.view(-1, h, N, d)
    return out
