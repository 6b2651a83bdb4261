"""The work this library is used for, as cases to be timed.

Three kinds of case, each through the public binding (``paper_1905_10759_b200.hbmm``):

* ``linear`` -- inference through fully connected layers.  The weights are binarized once, and their expanded form is
  kept in each layer's workspace, as a program with fixed weights keeps it; a pass binarizes every layer's activations
  and forms the products.  Each layer has activations of its own (what the batch normalisation and the non-linearity
  in front of it left behind; those belong to the caller).
* ``conv`` -- inference through one convolution, or two chained through the fused epilogue.  ``beta_a`` is the group
  size of the activations: 2 and more packs them (packed x packed product), 1 keeps them at full precision.
* ``train`` -- one layer's share of a training step.  The weights have just changed, so nothing about them is kept:
  both operands are binarized, the product is formed, the binarized weights are written out dense (the operand of the
  gradient with respect to the activations), and the weight gradient goes back through the binarization.

Activations are N(0, 1) (batch-norm outputs, which is what the method's layer order feeds the binarizer), weights are
He-normal.
"""
import math

import torch

from paper_1905_10759_b200 import hbmm

DTYPES = {"fp32": (torch.float32, hbmm.F32), "bf16": (torch.bfloat16, hbmm.BF16)}


# --------------------------------------------------------------------------------------------------------------
# Cases
# --------------------------------------------------------------------------------------------------------------
def _linear(M, dims, beta, x="fp32", scales="fp32", beta_w=0):
    return {"kind": "linear", "M": M, "dims": dims, "beta_a": beta, "beta_w": beta_w or beta, "x": x, "scales": scales}


def _conv(B, C, H, W, N, k, stride, beta_a, beta_w, x="fp32", scales="fp32", chain=0):
    return {"kind": "conv", "B": B, "C": C, "H": H, "W": W, "N": N, "k": k, "stride": stride, "beta_a": beta_a,
            "beta_w": beta_w, "x": x, "scales": scales, "chain": chain}


def _train(M, K, N, beta, scales="fp32"):
    return {"kind": "train", "M": M, "K": K, "N": N, "beta": beta, "scales": scales}


def listed():
    return [
        # the fully connected stack of an AlexNet-style classifier answering one request: launches and latency
        dict(_linear(1, "9216-4096-4096-1000", 64), name="fc_stack_b1"),
        # the same stack on a batch
        dict(_linear(256, "9216-4096-4096-1000", 64), name="fc_stack_b256"),
        # the smallest square product of the configurations: a layer of a small network
        dict(_linear(256, "256-256", 32), name="product_256"),
        # layers whose sizes are no multiple of anything, bf16 activations, the paper's own group size
        dict(_linear(333, "1000-720-100", 16, x="bf16"), name="fc_ragged"),
        # the largest square product of the configurations
        dict(_linear(8192, "8192-8192", 32), name="product_8192"),
        # one training step's share of a large layer, scales stored as bf16
        dict(_train(4096, 4096, 4096, 64, "bf16"), name="train_4096"),
        # ResNet-18 3x3 convolution, first stage, both operands packed, batch 64
        dict(_conv(64, 64, 56, 56, 64, 3, 1, 32, 32), name="conv2_x_b64"),
        # second stage at one of the paper's own group sizes
        dict(_conv(64, 128, 28, 28, 128, 3, 1, 4, 4), name="conv3_x_b64_beta4"),
        # last stage, answering one request
        dict(_conv(1, 512, 7, 7, 512, 3, 1, 32, 32), name="conv5_x_b1"),
        # the layer between two stages: stride 2, half a batch
        dict(_conv(32, 64, 56, 56, 128, 3, 2, 32, 32), name="conv_stride2_b32"),
        # activations at full precision (bf16), binarized weights
        dict(_conv(64, 128, 28, 28, 128, 3, 1, 1, 32, x="bf16"), name="conv3_x_b64_dense"),
        # two such layers, the first one's ReLU, batch-norm map and bf16 store in its epilogue
        dict(_conv(16, 256, 14, 14, 256, 3, 1, 1, 32, x="bf16", chain=1), name="conv4_x_b16_chain"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """A layer width: a multiple of 64 half of the time, of 8 a quarter, anything otherwise."""
    v, r = _log_int(rng, lo, hi), rng.random()
    step = 64 if r < 0.5 else 8 if r < 0.75 else 1
    return max(step, v // step * step)


def draw(rng):
    kind = rng.choice(["linear", "linear", "conv", "conv", "conv", "train"])
    beta = rng.choice([2, 4, 8, 16, 32, 32, 64, 64, 128])
    scales = rng.choice(["fp32", "fp32", "fp32", "bf16"])
    # sub-word groups cost the most where the integer pipe has to form them: their cases are kept smaller
    most = 6e9 if beta < 32 else 6e10
    if kind == "linear":
        n = rng.choice([1, 1, 2, 3])
        dims = [_size(rng, 256, 9216) for _ in range(n + 1)]
        M = rng.choice([_log_int(rng, 1, 8), _log_int(rng, 9, 8192)])
        while M * sum(a * b for a, b in zip(dims, dims[1:])) > most:
            M = max(1, M // 2)
        return _linear(M, "-".join(str(d) for d in dims), beta, rng.choice(["fp32", "fp32", "bf16"]), scales)
    if kind == "train":
        M, K, N = (_size(rng, 128, 4096) for _ in range(3))
        while M * K * N > most:
            M = max(1, M // 2)
        return _train(M, K, N, beta, scales)
    mode = rng.choice(["packed", "packed", "dense", "chain"])
    H = rng.choice([7, 8, 13, 14, 16, 27, 28, 32, 55, 56])
    k, stride = rng.choice([(3, 1), (3, 1), (3, 1), (3, 2), (1, 1), (1, 2), (5, 1)])
    B = _log_int(rng, 1, 64)
    if mode == "packed":
        C, N = rng.choice([32, 48, 64, 96, 100, 128, 192, 256, 512]), _size(rng, 32, 512)
        x, beta_a, beta_w = rng.choice(["fp32", "fp32", "fp32", "bf16"]), beta, beta if beta != 2 else 16
    else:
        C, N = rng.choice([64, 128, 192, 256, 512]), _size(rng, 32, 512)
        x, beta_a, beta_w = rng.choice(["bf16", "bf16", "fp32"]), 1, max(beta, 16)
    if mode == "chain":
        k, stride, x = 3, 1, "bf16"
        N = max(64, N // 64 * 64)                 # the second layer reads whole blocks of 64 channels
    while B > 1 and B * H * H * C * k * k * N / stride ** 2 > most:
        B = B // 2
    return _conv(B, C, H, H, N, k, stride, beta_a, beta_w, x, "fp32" if beta_a == 1 else scales, 1 if mode == "chain" else 0)


# --------------------------------------------------------------------------------------------------------------
# Inputs and the state a program keeps
# --------------------------------------------------------------------------------------------------------------
def _normal(shape, gen, dtype=torch.float32, scale=1.0):
    x = torch.randn(shape, generator=gen, device="cuda")
    return (x * scale).to(dtype) if scale != 1.0 or dtype != torch.float32 else x


def _pitch4(n):
    return (n + 3) // 4 * 4


def _out(rows, cols):
    """An fp32 result the product accepts: 16-byte rows."""
    return torch.empty((rows, _pitch4(cols)), dtype=torch.float32, device="cuda")[:, :cols]


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def _binarized_weights(N, K, beta, scales, gen):
    w = _normal((N, K), gen, scale=math.sqrt(2.0 / K))
    return hbmm.quantize(w, hbmm.alloc_operand(N, K, beta, DTYPES[scales][1]))


def _keeps_expanded(M, K, beta_a, beta_w):
    """Products whose expanded weights a caller can keep: the tensor-core path hbmm_gemm itself would pick (more rows than
    the matrix-vector kernel takes, K in whole words, groups of at most 128 elements)."""
    return M > 8 and K % 32 == 0 and min(beta_a, beta_w) <= 128


def _prepare_linear(case, gen):
    dims = [int(d) for d in case["dims"].split("-")]
    dt, sdt = DTYPES[case["x"]][0], DTYPES[case["scales"]][1]
    M, layers = case["M"], []
    for K, N in zip(dims, dims[1:]):
        x = _normal((M, K), gen, dt)
        A = hbmm.alloc_operand(M, K, case["beta_a"], sdt)
        W = _binarized_weights(N, K, case["beta_w"], case["scales"], gen)
        C, ws = _out(M, N), _bytes(hbmm.gemm_workspace_bytes(A, W))
        path = hbmm.PATH_AUTO
        if _keeps_expanded(M, K, case["beta_a"], case["beta_w"]):
            hbmm.gemm_ex(hbmm.quantize(x, A), W, C, hbmm.PATH_FOLDED, ws)      # leaves the expanded weights in ws
            path = hbmm.PATH_FOLDED_PREPARED
        layers.append((x, A, W, C, ws, path))
    return {"run": _run_linear, "layers": layers}


def _run_linear(s):
    out = []
    for x, A, W, C, ws, path in s["layers"]:
        hbmm.quantize(x, A)
        if path == hbmm.PATH_AUTO:
            hbmm.gemm(A, W, C, ws)
        else:
            hbmm.gemm_ex(A, W, C, path, ws)
        out.append(C)
    return out


def _geometry(case):
    k, st, pad = case["k"], case["stride"], case["k"] // 2
    geom = hbmm.make_geom(case["B"], case["C"], case["H"], case["W"], k, k, (st, st), (pad, pad))
    ho, wo = (case["H"] + 2 * pad - k) // st + 1, (case["W"] + 2 * pad - k) // st + 1
    return geom, case["B"] * ho * wo, case["C"] * k * k


def _prepare_conv(case, gen):
    geom, M, K = _geometry(case)
    dt, sdt = DTYPES[case["x"]][0], DTYPES[case["scales"]][1]
    B, C, H, W_, N = case["B"], case["C"], case["H"], case["W"], case["N"]
    s = {"geom": geom, "beta_a": case["beta_a"], "sdt": sdt}
    s["W"] = _binarized_weights(N, K, case["beta_w"], case["scales"], gen)
    s["ws"] = _bytes(hbmm.conv_workspace_bytes(geom, case["beta_a"], sdt, s["W"]))
    if not case["chain"]:
        s["x"], s["C"] = _normal((B, C, H, W_), gen, dt), _out(M, N)
        # the first call leaves the expanded weights in the workspace
        hbmm.conv_im2col(s["x"], geom, case["beta_a"], sdt, s["W"], s["C"], s["ws"])
        s["run"] = _run_conv
        return s
    s["x"] = _normal((B, H, W_, C), gen, torch.bfloat16)                       # NHWC, as a fused layer before left it
    s["geom2"] = hbmm.make_geom(B, N, H, W_, 3, 3, (1, 1), (1, 1))
    s["W2"] = _binarized_weights(N, N * 9, case["beta_w"], case["scales"], gen)
    s["ws2"] = _bytes(hbmm.conv_workspace_bytes(s["geom2"], 1, sdt, s["W2"]))
    s["y1"] = torch.empty((B, H, W_, N), dtype=torch.bfloat16, device="cuda")
    s["y2"] = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    bn = [(torch.rand(N, generator=gen, device="cuda") + 0.5, _normal((N,), gen, scale=0.1)) for _ in range(2)]
    s["ep1"] = hbmm.make_epilogue(hbmm.ACT_RELU, bn[0][0], bn[0][1], out=s["y1"].view(M, N))
    s["ep2"] = hbmm.make_epilogue(hbmm.ACT_RELU, bn[1][0], bn[1][1], out=s["y2"])
    s["flags"] = hbmm.CONV_INPUT_NHWC
    _run_chain(s)                                                              # leaves the expanded weights behind
    s["flags"] = hbmm.CONV_INPUT_NHWC | hbmm.CONV_WEIGHTS_PREPARED
    s["run"] = _run_chain
    return s


def _run_conv(s):
    return hbmm.conv_im2col(s["x"], s["geom"], s["beta_a"], s["sdt"], s["W"], s["C"], s["ws"], flags=hbmm.CONV_WEIGHTS_PREPARED)


def _run_chain(s):
    hbmm.conv_im2col_fused(s["x"], s["geom"], 1, s["sdt"], s["W"], s["ep1"], s["ws"], flags=s["flags"])
    hbmm.conv_im2col_fused(s["y1"], s["geom2"], 1, s["sdt"], s["W2"], s["ep2"], s["ws2"], flags=s["flags"])
    return [s["y1"], s["y2"]]


def _prepare_train(case, gen):
    M, K, N, beta, sdt = case["M"], case["K"], case["N"], case["beta"], DTYPES[case["scales"]][1]
    s = {"run": _run_train, "beta": beta, "x": _normal((M, K), gen), "w": _normal((N, K), gen, scale=math.sqrt(2.0 / K)),
         "gw": _normal((N, K), gen, scale=1e-2), "A": hbmm.alloc_operand(M, K, beta, sdt), "W": hbmm.alloc_operand(N, K, beta, sdt),
         "C": _out(M, N), "wd": torch.empty((N, K), dtype=torch.bfloat16, device="cuda"),
         "gx": torch.empty((N, K), dtype=torch.float32, device="cuda")}
    s["ws"] = _bytes(hbmm.gemm_workspace_bytes(s["A"], s["W"]))
    return s


def _run_train(s):
    hbmm.quantize(s["w"], s["W"])
    hbmm.quantize(s["x"], s["A"])
    hbmm.gemm(s["A"], s["W"], s["C"], s["ws"])
    hbmm.binarize_dense(s["w"], s["beta"], hbmm.BF16, out=s["wd"])
    hbmm.binarize_backward(s["w"], s["gw"], s["beta"], gx=s["gx"])
    return [s["C"], s["wd"], s["gx"]]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return {"linear": _prepare_linear, "conv": _prepare_conv, "train": _prepare_train}[case["kind"]](case, gen)


def run(state):
    return state["run"](state)


# --------------------------------------------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------------------------------------------
def _packed(rows, K, beta, scales):
    return rows * (K / 8 + -(-K // beta) * (2 if scales == "bf16" else 4))


def work(case):
    """Bytes: every input of the pass read once (activations, packed weights), every output written once.  Operations:
    two per output and K-element of a product."""
    size = 2 if case.get("x") == "bf16" else 4
    nbytes = flops = 0.0
    if case["kind"] == "linear":
        dims = [int(d) for d in case["dims"].split("-")]
        for K, N in zip(dims, dims[1:]):
            nbytes += case["M"] * K * size + _packed(N, K, case["beta_w"], case["scales"]) + case["M"] * N * 4
            flops += 2.0 * case["M"] * N * K
    elif case["kind"] == "conv":
        _, M, K = _geometry(case)
        N = case["N"]
        nbytes = case["B"] * case["C"] * case["H"] * case["W"] * size + _packed(N, K, case["beta_w"], case["scales"])
        flops = 2.0 * M * N * K
        if case["chain"]:
            nbytes += _packed(N, N * 9, case["beta_w"], case["scales"]) + 2 * M * N * 2       # both layers' outputs
            flops += 2.0 * M * N * N * 9
        else:
            nbytes += M * N * 4
    else:
        M, K, N = case["M"], case["K"], case["N"]
        nbytes = (M * K + 2 * N * K) * 4 + M * N * 4 + N * K * 2 + N * K * 4                  # x, w, gw; C, dense w, gradient
        flops = 2.0 * M * N * K
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the distance from the same computation in float64 (binarization included):
    fp32 products of K terms, summed in fp32: 1.4e-7 to 1.1e-5, growing with K; full-precision bf16 activations against
    weights of 2^-18: 2.7e-6 to 4.3e-6; scales stored as bf16, or the binarized weights written as bf16: 3.8e-5, a
    group's mean beside a rounding boundary now and then (2^-8 of that group); two layers with bf16 tensors between and
    behind them: 5.7e-4, single values one bf16 step apart."""
    if case["kind"] == "conv" and case["chain"]:
        return {"rel": 2.2e-3, "max": 3.2e-2}
    if case["scales"] == "bf16" or case["kind"] == "train":
        return {"rel": 1.5e-4, "max": 1.2e-2}
    if case["kind"] == "linear":
        K = max(int(d) for d in case["dims"].split("-")[:-1])
    else:
        K = case["C"] * case["k"] ** 2
    return {"rel": max(1.6e-5 if case["beta_a"] == 1 else 2e-6, 5e-9 * K)}


# --------------------------------------------------------------------------------------------------------------
# The same results in 64 bits
# --------------------------------------------------------------------------------------------------------------
def _group_means(x, beta):
    """Mean magnitude of each run of ``beta`` elements of a row (a shorter last run has its own length)."""
    G = -(-x.shape[1] // beta)
    n = torch.full((G,), float(beta), dtype=torch.float64, device=x.device)
    n[-1] = x.shape[1] - (G - 1) * beta
    mag = torch.nn.functional.pad(x.abs(), (0, G * beta - x.shape[1]))
    return mag.view(-1, G, beta).sum(2) / n


def _spread(d, beta, K):
    return d.repeat_interleave(beta, 1)[:, :K]


def _binarized(x, beta, scales):
    """delta (.) Sign(x), Sign(0) = +1; scales stored as bf16 are rounded as stored."""
    x = x.double()
    d = _group_means(x, beta)
    if scales == "bf16":
        d = d.bfloat16().double()
    return torch.where(x < 0, -1.0, 1.0) * _spread(d, beta, x.shape[1])


def _exact_linear(case, gen):
    dims, out = [int(d) for d in case["dims"].split("-")], []
    for K, N in zip(dims, dims[1:]):
        x = _normal((case["M"], K), gen, DTYPES[case["x"]][0])
        w = _normal((N, K), gen, scale=math.sqrt(2.0 / K))
        out.append(_binarized(x, case["beta_a"], case["scales"]) @ _binarized(w, case["beta_w"], case["scales"]).t())
    return out


def _conv64(x, w, case, N):
    """x NCHW in 64 bits, w the binarized filters [N, C kh kw]: the product [B Ho Wo, N], image by image."""
    k, st = case["k"], case["stride"]
    out = []
    for img in x:
        cols = torch.nn.functional.unfold(img[None], k, padding=k // 2, stride=st)[0].t()
        out.append((cols if case["beta_a"] == 1 else _binarized(cols, case["beta_a"], case["scales"])) @ w.t())
    return torch.cat(out)


def _exact_conv(case, gen):
    geom, M, K = _geometry(case)
    B, C, H, W_, N = case["B"], case["C"], case["H"], case["W"], case["N"]
    w = _binarized(_normal((N, K), gen, scale=math.sqrt(2.0 / K)), case["beta_w"], case["scales"])
    if not case["chain"]:
        return _conv64(_normal((B, C, H, W_), gen, DTYPES[case["x"]][0]).double(), w, case, N)
    x = _normal((B, H, W_, C), gen, torch.bfloat16).double()
    w2 = _binarized(_normal((N, N * 9), gen, scale=math.sqrt(2.0 / (N * 9))), case["beta_w"], case["scales"])
    bn = [(torch.rand(N, generator=gen, device="cuda") + 0.5, _normal((N,), gen, scale=0.1)) for _ in range(2)]
    ys = []
    for wd, (scale, shift) in zip((w, w2), bn):                                # each layer's result is stored as bf16
        y = _conv64(x.permute(0, 3, 1, 2), wd, case, N).relu() * scale.double() + shift.double()
        x = y.bfloat16().double().view(B, H, W_, N)
        ys.append(x)
    return [ys[0], ys[1].view(M, N)]


def _exact_train(case, gen):
    M, K, N, beta = case["M"], case["K"], case["N"], case["beta"]
    x, w = _normal((M, K), gen), _normal((N, K), gen, scale=math.sqrt(2.0 / K))
    gw = _normal((N, K), gen, scale=1e-2).double()
    C = _binarized(x, beta, case["scales"]) @ _binarized(w, beta, case["scales"]).t()
    # the gradient of delta (.) Sign(w) with respect to w: through the group's mean, and straight through the sign
    # where |w| <= 1
    w = w.double()
    sign, G = torch.where(w < 0, -1.0, 1.0), -(-K // beta)
    n = torch.full((G,), float(beta), dtype=torch.float64, device=w.device)
    n[-1] = K - (G - 1) * beta
    dot = torch.nn.functional.pad(gw * sign, (0, G * beta - K)).view(N, G, beta).sum(2) / n
    gx = sign * _spread(dot, beta, K) + torch.where(w.abs() <= 1, _spread(_group_means(w, beta), beta, K) * gw, 0.0)
    return [C, _binarized(w, beta, "fp32").bfloat16().double(), gx]


def exact(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return {"linear": _exact_linear, "conv": _exact_conv, "train": _exact_train}[case["kind"]](case, gen)
