"""The work a user of the N:M structured-binary linear layer has the library do, as cases to time and to compare.

Sizes are those of the LLaMA-2 7B / 13B / 70B linears the repository is configured for, with ragged ones between them;
N is the paper's 4, 5 or 6 of 8.  Weights follow the repository's recipe (fp16, N(0, 0.02), 1 % of the columns x 10; activations
N(0, 1), 0.5 % of the channels x 20) and go through the quantizer, so that salient columns, regions and scales are the
ones the method makes.
"""
import math
import types

import torch

import paper_2408_01803_b200 as stb

DEV = "cuda"
KINDS = ("gemv", "gemm_f16", "gemm", "mlp", "block", "stack", "layers", "quantize")


def listed():
    return [
        # decode, one linear per call.  The smallest call: a grouped-query k/v projection of 70B at one token.
        dict(name="gemv_1024x8192_4of8_b1", kind="gemv", n=1024, m=8192, N=4, batch=1, out="f32"),
        # a row count that fills no tile, columns of no model in particular, three sequences, fp16 out for the next layer
        dict(name="gemv_5003x2816_5of8_b3_f16", kind="gemv", n=5003, m=2816, N=5, batch=3, out="f16"),
        # the down projection of 7B for sixteen sequences
        dict(name="gemv_4096x11008_6of8_b16", kind="gemv", n=4096, m=11008, N=6, batch=16, out="f32"),
        # decode for 64 sequences, where the tensor-core product takes over from the GEMV (gate / up of 7B)
        dict(name="gemm_f16_11008x4096_6of8_t64", kind="gemm_f16", n=11008, m=4096, N=6, T=64, out="f16"),
        # decode, whole lists of linears in one call: the MLP of a 7B layer (gate, up, silu(gate) * up, down), one token
        dict(name="mlp_7b_6of8_b1", kind="mlp", h=4096, f=11008, N=6, batch=1),
        # the seven linears of a 13B decoder block, one token
        dict(name="block_13b_5of8_b1", kind="block", h=5120, f=13824, N=5, batch=1),
        # a decode step of the whole 7B stack, N per layer from {4, 5, 6}, one token
        dict(name="stack_7b_32_layers_b1", kind="stack", h=4096, f=11008, N=0, batch=1, layers=32),
        # four 7B layers for eight sequences through the call that launches layer by layer
        dict(name="layers_7b_4_layers_b8", kind="layers", h=4096, f=11008, N=0, batch=8, layers=4),
        # prefill: q / o of 70B for 2048 tokens
        dict(name="gemm_8192x8192_4of8_t2048", kind="gemm", n=8192, m=8192, N=4, T=2048, out="bf16"),
        # a short prompt of odd length through the down projection of 13B, fp32 out
        dict(name="gemm_5120x13824_5of8_t333", kind="gemm", n=5120, m=13824, N=5, T=333, out="f32"),
        # the largest prefill: gate / up of 70B
        dict(name="gemm_28672x8192_4of8_t2048", kind="gemm", n=28672, m=8192, N=4, T=2048, out="bf16"),
        # converting a checkpoint: dense fp16 weights through the quantizer, packed, and read back as dense fp16
        dict(name="quantize_4096x4096_6of8", kind="quantize", n=4096, m=4096, N=6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cols(rng, lo, hi):
    """A number of input columns: whole 128-column blocks."""
    return 128 * max(1, round(_log(rng, lo, hi) / 128))


def draw(rng):
    kind = rng.choice(("gemv", "gemv", "gemv", "gemm_f16", "mlp", "block", "stack", "layers", "gemm", "gemm", "gemm", "quantize"))
    N = rng.choice((4, 5, 6))
    if kind == "gemv":
        while True:
            n, m = _log(rng, 256, 28672), _cols(rng, 512, 28672)
            if n * m <= 28672 * 8192:
                return dict(kind=kind, n=n, m=m, N=N, batch=rng.choice((1, 1, 1, _log(rng, 2, 16), _log(rng, 2, 16))), out=rng.choice(("f32", "f16")))
    if kind == "gemm_f16":
        while True:
            n, m = _log(rng, 512, 28672), _cols(rng, 1024, 28672)
            if n * m <= 28672 * 8192:
                return dict(kind=kind, n=n, m=m, N=N, T=_log(rng, 17, 64), out=rng.choice(("f32", "f16")))
    if kind == "gemm":
        while True:
            n, m, T = _log(rng, 512, 28672), _cols(rng, 1024, 28672), _log(rng, 65, 4096)
            if n * m * T <= 28672 * 8192 * 2048 and n * m <= 28672 * 8192:
                return dict(kind=kind, n=n, m=m, N=N, T=T, out=rng.choice(("f32", "bf16")))
    if kind == "quantize":
        while True:
            n, m = _log(rng, 256, 16384), _cols(rng, 512, 16384)
            if n * m <= 4096 * 4096:
                return dict(kind=kind, n=n, m=m, N=N)
    h = _cols(rng, 1024, 8192)
    f = 128 * round(h * rng.uniform(2.5, 3.6) / 128)
    if kind == "mlp":
        return dict(kind=kind, h=h, f=f, N=N, batch=rng.choice((1, 1, 2, 4)))
    if kind == "block":
        return dict(kind=kind, h=h, f=f, N=N, batch=rng.choice((1, 1, 2, 4)))
    per_layer = 4 * h * h + 3 * h * f
    most = (32 if kind == "stack" else 4) * (4 * 4096 * 4096 + 3 * 4096 * 11008) // per_layer
    layers = max(1, min(48, _log(rng, 2, max(2, most)), most))
    if most < 1:                                  # one layer of this width is more than the largest listed call
        h, f = 4096, 11008
    return dict(kind=kind, h=h, f=f, N=0, batch=rng.choice((1, 1, 2, 4)) if kind == "stack" else _log(rng, 2, 16), layers=layers)


# ---------------------------------------------------------------------------------------------------------------------
def _dense(n, m, g):
    W = torch.randn(n, m, generator=g, device=DEV, dtype=torch.float32).mul_(0.02)
    W[:, torch.randperm(m, generator=g, device=DEV)[: round(0.01 * m)]] *= 10.0
    return W.to(torch.float16)


def _activations(T, m, g, dtype=torch.float16):
    x = torch.randn(T, m, generator=g, device=DEV, dtype=torch.float32)
    x[:, torch.randperm(m, generator=g, device=DEV)[: round(0.005 * m)]] *= 20.0
    return x.to(dtype)


def _norms(m, g):
    """Column norms of 256 rows of calibration activations."""
    return _activations(256, m, g, torch.float32).double().square().sum(0).sqrt()


def _pack(q):
    return stb.pack(q["n"], q["m"], q["N"], q["keep"], q["sign"], q["region"], q["sign2"], q["salient"], q["scale"])


def _unit_gain(q, layer):
    """The layer's scales divided by its gain, so that activations keep their size along a chain of linears (in a model the
    norms between them see to that)."""
    gain = stb.dequant(layer, torch.float16).float().square().sum().div(layer.n).sqrt()
    return dict(q, scale=(q["scale"].view(torch.float16) / gain).to(torch.float16).view(torch.int16))


def _layer(n, m, N, g):
    return _pack(stb.quantize(_dense(n, m, g), _norms(m, g), N))


class _Family:
    """Packed layers of a stack, each at an address of its own; one quantizer run per (shape, N)."""

    def __init__(self, g):
        self.g, self.made = g, {}

    def new(self, n, m, N):
        if (n, m, N) not in self.made:
            q = stb.quantize(_dense(n, m, self.g), _norms(m, self.g), N)
            self.made[n, m, N] = _unit_gain(q, _pack(q))
        return _pack(self.made[n, m, N])


def _n_per_layer(case, seed):
    """N of each decoder layer."""
    if case["N"]:
        return [case["N"]] * case.get("layers", 1)
    r = torch.Generator().manual_seed(seed)
    count = case.get("layers", 1)
    # each of 4, 5, 6 as often as the others (nearly), in an order from the seed: every seed is the same amount of work
    order = torch.randperm(count, generator=r).tolist()
    return [4 + (k + 2) % 3 for k in order]


def prepare(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    kind = case["kind"]
    st = types.SimpleNamespace(kind=kind)
    if kind in ("gemv", "gemm_f16", "gemm"):
        st.layer = _layer(case["n"], case["m"], case["N"], g)
        st.out_dtype = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[case["out"]]
        rows = case["batch"] if kind == "gemv" else case["T"]
        st.x = _activations(rows, case["m"], g, torch.bfloat16 if kind == "gemm" else torch.float16)
        if kind == "gemm_f16":                      # a decode loop keeps its output and its workspace
            st.y = torch.empty(rows, case["n"], dtype=st.out_dtype, device=DEV)
            st.ws = torch.empty(max(256, stb.gemm_f16_workspace(case["n"], case["m"], case["N"], rows)), dtype=torch.uint8, device=DEV)
        return st
    if kind == "quantize":
        st.W, st.xnorm, st.N = _dense(case["n"], case["m"], g), _norms(case["m"], g), case["N"]
        return st
    # lists of linears: buffers, steps and workspace are made once and serve every decode step
    h, f, b = case["h"], case["f"], case["batch"]
    Ns = _n_per_layer(case, seed)
    fam = _Family(g)
    L = len(Ns)
    st.x = _activations(b, h, g)
    wide = lambda cols: torch.empty(L, b, cols, dtype=torch.float16, device=DEV)  # noqa: E731
    st.out = {k: wide(h) for k in ("q", "k", "v", "o", "down")}
    st.out.update({k: wide(f) for k in ("gate", "up")})
    if kind == "mlp":
        for k in ("q", "k", "v", "o"):
            del st.out[k]
    steps, cur, o = [], st.x, st.out
    for i, N in enumerate(Ns):
        if kind != "mlp":
            # attention is not part of this path: the output projection reads the queries in its place
            steps += [(fam.new(h, h, N), cur, o[k][i]) for k in ("q", "k", "v")]
            steps.append((fam.new(h, h, N), o["q"][i], o["o"][i]))
            cur = o["o"][i]
        steps += [(fam.new(f, h, N), cur, o[k][i]) for k in ("gate", "up")]
        # the gated activation where one layer stands alone; along a stack (no norms between the layers here) a product of
        # two activations would grow or fade without bound, so there the down projection reads the gate's output
        gated = kind in ("mlp", "block")
        steps.append((fam.new(h, f, N), (o["gate"][i], o["up"][i]) if gated else o["gate"][i], o["down"][i]))
        cur = o["down"][i]
    st.layers = [s[0] for s in steps]
    st.steps = stb.make_steps(steps)
    st.status = torch.zeros(1, dtype=torch.int32, device=DEV)
    if kind != "layers":
        st.ws = stb.resident_workspace(st.steps)
    return st


def run(st):
    if st.kind == "gemv":
        return stb.gemv(st.layer, st.x, out_dtype=st.out_dtype)
    if st.kind == "gemm":
        return stb.gemm(st.layer, st.x, out_dtype=st.out_dtype)
    if st.kind == "gemm_f16":
        return stb.gemm_f16(st.layer, st.x, out=st.y, ws=st.ws)
    if st.kind == "quantize":
        q = stb.quantize(st.W, st.xnorm, st.N)
        return {"logical": {k: q[k] for k in ("keep", "sign", "region", "sign2", "salient", "scale")}, "dense": stb.dequant(_pack(q), torch.float16)}
    if st.kind == "layers":
        stb.layer_stack(None, dev_status=st.status, marshalled=st.steps)
    else:
        stb.layer_stack_resident(None, st.ws, dev_status=st.status, marshalled=st.steps)
    return st.out


def _packed_bytes(n, m, N):
    """A layer as the format defines it, per row and block of 128 columns: 16 bytes of keep masks, 2 N of signs, 4 N of region
    ids, five fp16 scales, and two bits for each salient column (about eight per block)."""
    return n * (m // 128) * (16 + 6 * N + 10 + 2)


def work(case):
    kind = case["kind"]
    if kind in ("gemv", "gemm_f16", "gemm"):
        n, m, N = case["n"], case["m"], case["N"]
        T = case["batch"] if kind == "gemv" else case["T"]
        return {"bytes": _packed_bytes(n, m, N) + 2 * T * m + (4 if case["out"] == "f32" else 2) * T * n, "flops": 2.0 * n * m * T}
    if kind == "quantize":
        n, m, N = case["n"], case["m"], case["N"]
        # dense in, logical fields out, packed layer out and in again, dense out
        logical = n * (m // 8) * 4 + n * (m // 128) * 14 + (m // 128) * 16
        return {"bytes": 2 * n * m + 8 * m + logical + 2 * _packed_bytes(n, m, N) + 2 * n * m, "flops": 0.0}
    h, f, b = case["h"], case["f"], case["batch"]
    nbytes = flops = 0.0
    for N in _n_per_layer(case, 0):
        shapes = [(f, h), (f, h), (h, f)] + ([] if kind == "mlp" else [(h, h)] * 4)
        for n, m in shapes:
            nbytes += _packed_bytes(n, m, N) + 2 * b * n
            flops += 2.0 * n * m * b
        nbytes += 2 * b * (h + f) + (0 if kind == "mlp" else 4 * b * h)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "quantize":
        return "exact"                    # bits, region ids and fp16 scales that the definition fixes
    if kind in ("gemv", "gemm_f16"):
        # exact fp16 operands, fp32 sums of up to 28672 terms; the fp16 result is that sum rounded
        return {"rel": 2e-5 if case["out"] == "f32" else 1e-3}
    if kind == "gemm":
        # the call defines its weights as bf16 roundings of the scales; what is left is the fp32 sum and a bf16 result
        return {"rel": 2e-5 if case["out"] == "f32" else 5e-3}
    # a chain of linears with fp16 between them: every result is rounded to 2^-11, and the roundings add up along the chain
    depth = 4 * len(_n_per_layer(case, 0))
    return {"rel": 1e-3 * math.sqrt(depth)}
