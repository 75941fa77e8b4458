"""The work this library is used for, as measurable cases: one pass of the sparse FFN through its public entry points.

Single-token decode (full and low-parameter gate, every storage type of the weights), a layer stack replayed from a CUDA
graph, decode through host buffers, and batches from a few concurrent requests up to a prompt of some hundred tokens.
The dense comparator, the selectable cross-check paths and the offline gate conversion are not in here.
"""
import functools
import math
import statistics

import numpy as np
import torch

from paper_2609_31975_b200 import SparseFFN, g_diagonal, residual_cast

DEV = "cuda:0"
BITS = {"f32": 32, "bf16": 16, "int8": 8, "int4": 4}
RMS_EPS = 1e-5


def case(kind, dtype, B, D, H, r=0, s=0.9, zipf=False, act="relu", act_up="", layers=1, **more):
    """kind: "call" (one FFN call), "host" (x and y in pinned host memory), "stack" (a CUDA graph of dependent layers).
    dtype: storage of the weights (tokens: bf16, or fp32 with fp32 weights).  r: rank of the low-parameter gate, 0 = full
    gate matrix.  s: mean share of neurons that do not fire.  zipf: firing probabilities of the neurons follow a power law
    (else all are equal).  act_up: activation on the up projection ("" = none)."""
    return dict(kind=kind, dtype=dtype, B=B, D=D, H=H, r=r, s=s, zipf=zipf, act=act, act_up=act_up, layers=layers, **more)


def listed():
    return [
        # the smallest model the repository measures: a call is launch and latency, not bytes
        case("call", "f32", 1, 256, 1024, name="decode_small_f32"),
        # one decode step's FFN of a 4096-wide model: the headline workload
        case("call", "bf16", 1, 4096, 14336, name="decode_bf16"),
        # the same for a caller whose activations live on the host and who waits for y
        case("host", "bf16", 1, 4096, 14336, s=0.8, name="decode_bf16_host"),
        # the low-parameter gate, which leaves a call a third of the bytes
        case("call", "bf16", 1, 4096, 14336, r=512, act="sqrelu", name="decode_lopa_bf16"),
        # weight-only int8 and int4 decode, the latter at the paper's width
        case("call", "int8", 1, 4096, 14336, name="decode_int8"),
        case("call", "int4", 1, 3840, 10240, s=0.95, act="rsplus", name="decode_int4"),
        # a token through eight dependent layers of the paper's shape (ragged H, rank 480) in full precision
        case("stack", "f32", 1, 3840, 14230, r=480, layers=8, name="stack_lopa_f32"),
        # a few concurrent requests on 4-bit weights, with a second activation
        case("call", "int4", 5, 4096, 14336, zipf=True, act_up="silu", name="batch5_int4"),
        # a serving batch
        case("call", "bf16", 16, 4096, 14336, zipf=True, name="batch16_bf16"),
        # a large serving batch on int8 weights
        case("call", "int8", 64, 4096, 14336, zipf=True, name="batch64_int8"),
        # the widest model, low-parameter gate, a small batch
        case("call", "bf16", 8, 8192, 28672, r=1024, act="sqrelu", name="batch8_wide_lopa_bf16"),
        # the tokens of a prompt at once
        case("call", "bf16", 200, 4096, 14336, zipf=True, name="prompt200_bf16"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_once(rng):
    kind = rng.choice(["call"] * 8 + ["host", "stack"])
    dtype = rng.choice(["bf16", "bf16", "int8", "int4"] if kind == "call" else ["bf16"] if kind == "host" else ["bf16", "f32"])
    B = 1
    if kind == "call":
        if rng.random() < 0.5:
            B = round(_log_uniform(rng, 2, 256))
        elif rng.random() < 0.25:
            dtype = "f32"
    step = 64 if B == 1 else 128  # widths of models: multiples of 64 and more; batches are run on tensor-core tiles
    D = max(256, round(_log_uniform(rng, 256, 8192) / step) * step)
    H = min(28672, round(D * rng.uniform(2.0, 4.0)))
    if rng.random() < 0.5:
        H = H // 64 * 64
    r = 0
    if rng.random() < (0.7 if kind == "stack" else 0.3):
        r = max(64, round(D * rng.uniform(1 / 16, 1 / 4) / 32) * 32)
        if B > 1:
            r = r // 64 * 64
    return case(kind, dtype, B, D, H, r=r, s=round(rng.uniform(0.7, 0.97), 3), zipf=B > 1 and rng.random() < 0.7,
                act=rng.choice(["relu", "sqrelu", "rsplus"]), act_up=rng.choice(["", "", "", "relu", "silu"]),
                layers=rng.randint(2, 8) if kind == "stack" else 1)


def _price(c):
    w = work(c)
    return w["bytes"] / 6.5e12 + w["flops"] / 1.4e15


def draw(rng):
    most = max(_price(c) for c in listed())
    while True:
        c = _draw_once(rng)
        if _price(c) <= most:
            return c


@functools.lru_cache(maxsize=64)
def _firing(H, zipf, s):
    """Firing probability per rank of neuron: min(0.99, c k^-1.1) with the mean 1 - s, or 1 - s for all."""
    if not zipf:
        return np.full(H, 1.0 - s)
    base = np.arange(1, H + 1, dtype=np.float64) ** -1.1
    lo, hi = 0.0, float(H)
    for _ in range(60):
        c = 0.5 * (lo + hi)
        if np.minimum(0.99, c * base).mean() < 1.0 - s:
            lo = c
        else:
            hi = c
    return np.minimum(0.99, 0.5 * (lo + hi) * base)


def _matrix(c, rows, cols, std, gen):
    """A weight matrix as the handle takes it: a tensor, or codes and row scales as a quantiser leaves them."""
    v = torch.randn((rows, cols), generator=gen, device=DEV)
    if BITS[c["dtype"]] > 8:
        return v.mul_(std).to(torch.float32 if c["dtype"] == "f32" else torch.bfloat16)
    scale = 1.0 + 0.1 * (2.0 * torch.rand(rows, generator=gen, device=DEV) - 1.0)
    if c["dtype"] == "int8":
        return {"q": v.mul_(32.0).round_().clamp_(-127, 127).to(torch.int8), "s": scale * (std / 32.0)}
    q = v.mul_(2.5).round_().clamp_(-7, 7).to(torch.int8).bitwise_and_(15).view(torch.uint8)
    return {"q": q[:, 0::2] | (q[:, 1::2] << 4), "s": scale * (std / 2.5)}


def _layer(c, gen):
    """One FFN: weights N(0, 1 / fan_in), and the gate bias that makes neuron j fire with its probability."""
    D, H, r = c["D"], c["H"], c["r"]
    if r:
        gate = {"V": _matrix(c, r, D, D ** -0.5, gen), "U": _matrix(c, H, r, r ** -0.5, gen), "g_idx": g_diagonal(H, D, DEV),
                "use_rmsnorm": True, "rms_eps": RMS_EPS}
    else:
        gate = {"W_g": _matrix(c, H, D, D ** -0.5, gen)}
    sigma = math.sqrt(2.0) if r else 1.0  # the low-parameter gate adds one entry of the token
    if c["zipf"]:
        p = torch.from_numpy(_firing(H, True, c["s"])).to(DEV)[torch.randperm(H, generator=gen, device=DEV)]
        b_g = (math.sqrt(2.0) * sigma * torch.erfinv(2.0 * p - 1.0)).float()
    else:
        b_g = torch.full((H,), -sigma * statistics.NormalDist().inv_cdf(c["s"]), device=DEV)
    return gate, b_g, _matrix(c, H, D, D ** -0.5, gen), _matrix(c, H, D, D ** -0.5, gen)


def prepare(c, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    D, H, B, L = c["D"], c["H"], c["B"], c["layers"]
    dtype = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    ffn = SparseFFN(D, H, dtype, r_max=c["r"], B_max=B, device=DEV)
    ffn.set_up_activation(c["act_up"] or None)
    layers = [_layer(c, gen) for _ in range(L)]
    st = {"kind": c["kind"], "ffn": ffn, "layers": layers, "act": c["act"]}
    x = torch.randn((B, D), generator=gen, device=DEV).to(dtype)
    if c["kind"] == "host":
        x_host, y_host = x[0].cpu().pin_memory(), torch.empty(D, dtype=torch.float32).pin_memory()
        st["call"] = ffn.prepared(x_host, *layers[0], c["act"], y_host, host=True)
        st["out"], st["x_host"] = y_host, x_host
        st["stream"] = torch.cuda.current_stream()
    elif c["kind"] == "stack":
        # layer l + 1 reads what stands for the attention's output plus a part of layer l's y
        xs = torch.randn((L + 1, D), generator=gen, device=DEV).to(dtype)
        resid, ys = xs.clone(), torch.empty((L, D), dtype=torch.float32, device=DEV)
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())

        def token():
            for l in range(L):
                ffn.sparse_ffn_forward(xs[l], *layers[l], c["act"], ys[l], stream=stream)
                residual_cast(ys[l], resid[l + 1], 0.25, xs[l + 1], stream=stream)

        token()
        stream.synchronize()
        st["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st["graph"], stream=stream):
            token()
        st["out"] = (ys, xs[L])
        st["keep"] = (xs, resid)
    elif B == 1:
        st["out"] = torch.empty(D, dtype=torch.float32, device=DEV)
        st["x"] = x[0].clone()
        if c["dtype"] != "f32":  # a decode loop: the call marshalled once
            st["call"] = ffn.prepared(st["x"], *layers[0], c["act"], st["out"])
    else:
        st["x"] = x
    st["forward"] = {"int8": ffn.sparse_ffn_forward_q8, "int4": ffn.sparse_ffn_forward_q4}.get(c["dtype"], ffn.sparse_ffn_forward)
    return st


def run(st):
    if st["kind"] == "stack":
        st["graph"].replay()
        return st["out"]
    if "call" in st:
        st["call"]()
        if st["kind"] == "host":
            st["stream"].synchronize()  # y is on the host then
        return st["out"]
    return st["forward"](st["x"], *st["layers"][0], st["act"])


def work(c):
    """The gate in full, the rows of W_up / W_down of the union of the fired neurons, scales, biases, tokens and y; the
    products of the gate for every token, those of the up and down projections for the pairs of token and fired neuron."""
    D, H, B, r, bits = c["D"], c["H"], c["B"], c["r"], BITS[c["dtype"]]
    p = _firing(H, c["zipf"], c["s"])
    union = float((1.0 - (1.0 - p) ** B).sum())
    gate = r * D + H * r if r else H * D
    size = (gate + 2.0 * union * D) * bits / 8 + 4 * H + B * D * ((4 if bits == 32 else 2) + 4)
    size += 4 * (H + r + 2 * union if bits < 16 else 0) + (4 * H if r else 0)
    flops = 2.0 * B * gate + 4.0 * B * D * float(p.sum())
    return {"bytes": c["layers"] * size, "flops": c["layers"] * flops}


def tolerance(c):
    """About four times what the path differs by from the same formulas in 64 bits (2-norm, largest): a batch rounds h to
    bf16 for the down projection (1.7e-3, 8e-3); a single token keeps fp32 throughout (2.5e-7; another order of its sums
    of up to 30000 terms shows a few times that), but for the int8 limbs that integer products make of it (8e-5, 3e-4).  A
    stack rounds each layer's token to its type: in bf16 an entry at a boundary may go either way (2^-8 of that entry, or
    2.4e-4 of the smallest token, a few times in eight layers)."""
    if c["kind"] == "stack" and c["dtype"] == "bf16":
        return {"rel": 1e-3, "max": 2e-2}
    if c["B"] > 1:
        return {"rel": 7e-3, "max": 4e-2}
    return {"rel": 3e-4, "max": 1.5e-3} if BITS[c["dtype"]] < 16 else {"rel": 2e-6, "max": 1e-5}


def _wide(m):
    """The matrix that a weight stands for, in 64 bits."""
    if not isinstance(m, dict):
        return m.double()
    q = m["q"]
    if q.dtype == torch.uint8:  # two codes a byte, the even column in the low half
        q = torch.stack([q & 15, q >> 4], dim=2).reshape(q.shape[0], -1).to(torch.int8)
        q = torch.where(q > 7, q - 16, q)
    return q.double() * m["s"].double()[:, None]


def _act(name, z):
    if name == "silu":
        return z * torch.sigmoid(z)
    p = z.clamp(min=0.0)
    return {"relu": lambda: p, "sqrelu": lambda: p * p, "rsplus": lambda: p * torch.sigmoid(p)}[name]()


def _ffn64(c, layer, x):
    gate, b_g, W_up, W_down = layer
    if c["r"]:
        v = x @ _wide(gate["V"]).T
        v = v / torch.sqrt((v * v).mean(dim=1, keepdim=True) + RMS_EPS)
        z = v @ _wide(gate["U"]).T + x[:, torch.arange(c["H"], device=DEV) * c["D"] // c["H"]]
    else:
        z = x @ _wide(gate["W_g"]).T
    u = x @ _wide(W_up).T
    return (_act(c["act"], z + b_g.double()) * (_act(c["act_up"], u) if c["act_up"] else u)) @ _wide(W_down)


def exact(c, seed):
    """The formulas of the path in 64 bits.  A stack rounds each layer's token to its storage type, which is part of it."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    layers = [_layer(c, gen) for _ in range(c["layers"])]
    dtype = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    x = torch.randn((c["B"], c["D"]), generator=gen, device=DEV).to(dtype)
    if c["kind"] != "stack":
        y = _ffn64(c, layers[0], x.double())
        return y.cpu()[0] if c["kind"] == "host" else y if c["B"] > 1 else y[0]
    xs = torch.randn((c["layers"] + 1, c["D"]), generator=gen, device=DEV).to(dtype)
    x, ys = xs[:1], []
    for l, layer in enumerate(layers):
        y = _ffn64(c, layer, x.double())
        ys.append(y[0])
        x = (xs[l + 1].double() + 0.25 * y).to(dtype)
    return torch.stack(ys), x[0].double()
