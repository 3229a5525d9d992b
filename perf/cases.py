"""The work a program has this library do, as cases that can be timed and compared.

A case is a dict of plain values; its "kind" says which public entry point a pass goes through:

  linear     one layer's forward pass (AserLinear.__call__)
  block      the seven linears of a decoder block: query/key/value stored fused
             (AserSharedInputCat), output, gate and up sharing their input (AserSharedInput), down
  shared     layers that share their input, one linear launch per layer (AserSharedInput)
  variant    the separate steps with the options of the activation pass: code width and T stored as
             bf16 pairs (quant_act_ws, then linear_w4a8_lr at twice the rank)
  host       a forward pass from pinned host memory to pinned host memory (AserLinear.forward_host)
  pack       a layer's weights quantized and laid out when a model is loaded (pack_w4, repack_w4)
  construct  a layer's int4 weights and low-rank factors built from calibration tokens (construct)

Activations are N(0, 1) in fp16 with 1 % of the channels scaled up, weights N(0, sigma^2), the
smoothing vector is sqrt(max|X_c| / max|W_c|) on those channels and 1 elsewhere, the input of a down
projection is silu(a) b: the distributions of the benchmark's configurations, drawn on the GPU.
Outside `construct` the factors are Gaussian stand-ins of the right shape and size: the low-rank term
is then about a fifth of the output.
"""
import math

import torch

import paper_2411_07762_b200 as aser

HIDDEN, KV, MLP = 4096, 1024, 14336          # the decoder block of the benchmark (8B class)


def _linear(tokens, k, n, rank, **more):
    return dict(kind="linear", tokens=tokens, k=k, n=n, rank=rank, **more)


def listed():
    return [
        # one new token of one sequence through an attention projection: the smallest call
        dict(_linear(1, 4096, 4096, 64, capacity=16), name="decode_1_proj"),
        # a decode step of eight sequences through a whole block (8B class): seven layers, few tokens
        dict(kind="block", tokens=8, rank=128, name="decode_8_block"),
        # a decode step of sixteen sequences, the large projection of a 70B-class layer: weight stream
        dict(_linear(16, 8192, 28672, 64, gain=50.0, sigma=0.015, capacity=16), name="decode_16_70b_up"),
        # a decode step of a full serving batch (odd token count), 70B-class square projection
        dict(_linear(101, 8192, 8192, 32, gain=50.0, sigma=0.015), name="batch_101_70b_proj"),
        # a chunk of a prompt mixed with running sequences: a ragged number of tokens, gate and up
        dict(kind="shared", tokens=333, k=HIDDEN, n=MLP, layers=2, rank=64, name="chunk_333_gate_up"),
        # prefill of one 2048-token prompt, gate projection (the block below has the down projection)
        dict(_linear(2048, HIDDEN, MLP, 64), name="prefill_2048_gate"),
        # prefill of a batch of prompts (8 x 512 tokens) through a whole block
        dict(kind="block", tokens=4096, rank=128, name="prefill_4096_block"),
        # the largest call: 70B-class projection, 4096 tokens, the highest rank
        dict(_linear(4096, 8192, 28672, 256, gain=50.0, sigma=0.015), name="prefill_4096_70b_up"),
        # six-bit activation codes and T as bf16 pairs (the paper's W4A6 rows and outlier split)
        dict(kind="variant", tokens=1500, k=HIDDEN, n=HIDDEN, rank=64, act_bits=6, pair=True, name="w4a6_pair_1500"),
        # activations that live in host memory: copy in, forward pass, copy out
        dict(kind="host", tokens=1024, k=HIDDEN, n=HIDDEN, rank=128, name="host_1024_proj"),
        # loading a model, layer by layer: fp16 weights quantized, packed and laid out
        dict(kind="pack", k=8192, n=28672, sigma=0.015, gain=50.0, name="pack_70b_up"),
        # quantizing a model, layer by layer: weights, whitening and factors from calibration tokens
        dict(kind="construct", k=HIDDEN, n=HIDDEN, rank=64, calibration=512, name="construct_4096"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["linear"] * 8 + ["block", "block", "shared", "shared", "variant", "variant", "host", "pack", "construct"])
    tokens = min(4096, _log(rng, 1, 5000))
    rank = 16 * rng.choice([0, 1, 2, 3, 4, 4, 6, 8, 8, 12, 16])
    if kind == "block":
        return dict(kind=kind, tokens=tokens, rank=16 * rng.choice([1, 2, 4, 6, 8]))
    if kind == "linear":
        k = 128 * _log(rng, 4, 112)
        n = 8 * _log(rng, 64, 3584)
        if rng.random() < 0.5:
            k, n = rng.choice([(4096, 4096), (4096, 1024), (4096, 14336), (14336, 4096), (8192, 8192), (8192, 28672)])
        n = min(n, 8 * (8192 * 3584 // k))                   # no layer above the largest listed one
        big = k >= 8192
        return _linear(tokens, k, n, rank, gain=50.0 if big else 30.0, sigma=0.015 if big else 0.02,
                       gated=k == MLP)
    if kind == "shared":
        return dict(kind=kind, tokens=tokens, k=128 * _log(rng, 4, 64), n=8 * _log(rng, 128, 1792),
                    layers=rng.choice([2, 3]), rank=16 * rng.choice([1, 2, 4, 6, 8]))
    if kind == "variant":
        return dict(kind=kind, tokens=tokens, k=128 * _log(rng, 4, 64), n=8 * _log(rng, 64, 1024),
                    rank=16 * rng.choice([1, 2, 4, 6, 8]), act_bits=rng.choice([6, 8]), pair=rng.random() < 0.5)
    if kind == "host":
        return dict(kind=kind, tokens=min(tokens, 2048), k=HIDDEN, n=rng.choice([1024, 4096, 4104]), rank=16 * rng.randint(1, 8))
    if kind == "pack":
        return dict(kind=kind, k=128 * _log(rng, 8, 112), n=8 * _log(rng, 128, 3584))
    return dict(kind="construct", k=128 * rng.randint(6, 30), n=8 * rng.randint(96, 500), rank=16 * rng.randint(1, 4),
                calibration=rng.randint(100, 512))


# ----------------------------------------------------------------------------
# what a program has in hand
# ----------------------------------------------------------------------------
class _Maker:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed) & 0x7FFFFFFF)

    def normal(self, *shape, scale=1.0):
        return torch.randn(*shape, device="cuda", dtype=torch.float16, generator=self.g) * scale

    def outliers(self, k):
        return torch.randperm(k, device="cuda", generator=self.g)[:max(1, k // 100)]

    def activations(self, tokens, k, idx, gain, gated=False):
        x = self.normal(tokens, k)
        if gated:
            x = torch.nn.functional.silu(x) * self.normal(tokens, k)
        x[:, idx] *= gain
        return x

    def smoothing(self, x, w, idx):
        s = torch.ones(x.shape[1], device="cuda", dtype=torch.float32)
        s[idx] = (x[:, idx].abs().amax(0).float() / w[:, idx].abs().amax(0).float()).sqrt().clamp_min(1e-3)
        return s

    def factors(self, k, n, rank):
        if rank == 0:
            return None, None
        return self.normal(rank, k, scale=0.02), self.normal(n, rank, scale=0.02)


def _group(m, tokens, k, ns, rank, gain, sigma, gated=False):
    """Layers that read one x [tokens, K]: x, its smoothing vector, and each layer's weights and factors."""
    idx = m.outliers(k)
    x = m.activations(tokens, k, idx, gain, gated)
    s, layers = None, []
    for n in ns:
        w = m.normal(n, k, scale=sigma)
        if s is None:
            s = m.smoothing(x, w, idx)
        layers.append((w, *m.factors(k, n, rank)))
    return x, s, layers


def _inputs(case, seed):
    """The groups of layers that a pass goes through, one after the other."""
    m = _Maker(seed)
    gain, sigma, rank = case.get("gain", 30.0), case.get("sigma", 0.02), case.get("rank", 0)
    if case["kind"] == "block":
        for k, ns in ((HIDDEN, (HIDDEN, KV, KV)), (HIDDEN, (HIDDEN,)), (HIDDEN, (MLP, MLP)), (MLP, (HIDDEN,))):
            yield _group(m, case["tokens"], k, ns, rank, gain, sigma, gated=k == MLP)
    elif case["kind"] in ("pack", "construct"):
        yield _group(m, case.get("calibration", 64), case["k"], (case["n"],), 0, gain, sigma)
    else:
        yield _group(m, case["tokens"], case["k"], (case["n"],) * case.get("layers", 1), rank, gain, sigma,
                     case.get("gated", False))


def prepare(case, seed):
    kind = case["kind"]
    tokens, rank = case.get("tokens", 0), case.get("rank", 0)
    st = {"kind": kind}

    def built(group, capacity):
        x, s, layers = group
        return x, [aser.AserLinear(w, s, la, lb, capacity) for w, la, lb in layers]

    if kind == "block":
        (x_qkv, qkv), (x_o, o), (x_mlp, mlp), (x_down, down) = [built(g, tokens) for g in _inputs(case, seed)]
        st["steps"] = [(aser.AserSharedInputCat(qkv, tokens), x_qkv), (o[0], x_o),
                       (aser.AserSharedInput(mlp, tokens), x_mlp), (down[0], x_down)]
        return st
    k, n = case["k"], case["n"]
    group, = _inputs(case, seed)
    if kind in ("pack", "construct"):
        st.update(W=group[2][0][0], s=group[1], X=group[0], rank=rank)
        return st
    x, layers = built(group, case.get("capacity", tokens))
    st["X"] = x
    if kind == "shared":
        st["call"] = aser.AserSharedInput(layers, tokens)
        return st
    layer = layers[0]
    st["call"] = layer
    if kind == "host":
        st["X_host"] = x.cpu().pin_memory()
        st["Y_host"] = torch.zeros((tokens, n), dtype=torch.float16).pin_memory()
    elif kind == "variant":
        pair = case["pair"]
        r2 = 2 * rank if pair else rank
        st.update(bits=case["act_bits"], pair=pair, n=n,
                  L_B=aser.pair_up_projection(layer.L_B) if pair else layer.L_B,
                  scratch=torch.empty((max(1024, aser.quant_workspace_bytes(tokens, k, rank)),), dtype=torch.uint8, device="cuda"),
                  ws=aser.new_workspace(tokens, n, k, r2),
                  out=(torch.empty((tokens, k), dtype=torch.int8, device="cuda"),
                       torch.empty((tokens,), dtype=torch.float32, device="cuda"),
                       torch.empty((tokens, r2), dtype=torch.bfloat16, device="cuda")),
                  Y=torch.empty((tokens, n), dtype=torch.float16, device="cuda"))
    return st


def run(st):
    kind = st["kind"]
    if kind == "block":
        return [call(x) for call, x in st["steps"]]
    if kind in ("linear", "shared"):
        return st["call"](st["X"])
    if kind == "host":
        st["call"].forward_host(st["X_host"], st["Y_host"])
        torch.cuda.current_stream().synchronize()        # the result is in host memory when the pass ends
        return st["Y_host"]
    if kind == "variant":
        layer = st["call"]
        codes, scale, t = aser.quant_act_ws(st["X"], layer.s, layer.L_A, ws=st["scratch"], out=st["out"],
                                            act_bits=st["bits"], t_pair=st["pair"])
        y = aser.linear_w4a8_lr(codes, scale, layer.Wk, layer.w_scale, t, st["L_B"], st["n"], st["ws"], Y=st["Y"])
        return {"Y": y, "codes": codes, "scale": scale}
    if kind == "pack":
        wq, scale = aser.pack_w4(st["W"], st["s"])
        return {"Wq": wq, "scale": scale, "Wk": aser.repack_w4(wq)}
    out = aser.construct(st["W"], st["s"], st["X"], st["rank"])
    # the factors are determined up to sign and rotation: their product is what a layer uses
    return {"Wq": out["Wq"], "scale": out["w_scale"], "sigma": out["sigma"],
            "product": out["L_B"].float() @ out["L_A"].float()}


# ----------------------------------------------------------------------------
# the same outputs in plain torch: codes and their scales by single fp32 steps, as the format
# defines them, everything summed in fp64
# ----------------------------------------------------------------------------
def _codes(v, qmax, low):
    scale = v.abs().amax(1) / float(qmax)
    q = (v / torch.where(scale > 0, scale, 1.0)[:, None]).round_().clamp_(low, qmax)
    return q, scale


def _exact_pass(x, s, layers, qmax=127):
    xs = x.float() / s
    q, a_scale = _codes(xs, qmax, -qmax)
    out = []
    for w, la, lb in layers:
        wq, w_scale = _codes(w.float() * s, 7, -8)
        y = q.double() @ wq.double().T * a_scale.double()[:, None] * w_scale.double()
        if la is not None:
            y += (xs.double() @ la.double().T) @ lb.double().T
        out.append(y)
    return out, a_scale


def exact(case, seed):
    kind = case["kind"]
    groups = _inputs(case, seed)
    if kind == "block":
        outs = [_exact_pass(*g)[0] for g in groups]
        return [outs[0], outs[1][0], outs[2], outs[3][0]]
    (x, s, layers), = groups
    if kind in ("linear", "host"):
        return _exact_pass(x, s, layers)[0][0]
    if kind == "shared":
        return _exact_pass(x, s, layers)[0]
    if kind == "variant":
        y, a_scale = _exact_pass(x, s, layers, 2 ** (case["act_bits"] - 1) - 1)
        return {"Y": y[0], "codes": None, "scale": a_scale.double()}
    ws = layers[0][0].float() * s
    if kind == "pack":
        return {"Wq": None, "scale": ws.double().abs().amax(1) / 7, "Wk": None}
    q, scale = _codes(ws, 7, -8)
    error = ws.double() - q.double() * scale.double()[:, None]
    xs = (x.float() / s).double()
    gram = xs.T @ xs
    gram.diagonal().add_(0.01 * gram.trace() / gram.shape[0])
    a = error @ torch.linalg.cholesky(gram)
    values, u = torch.linalg.eigh(a @ a.T)               # ascending: the squared singular values of E S
    u = u[:, -case["rank"]:]
    # U_r U_r^T (E S) S^-1
    return {"Wq": None, "scale": scale.double(), "sigma": values[-case["rank"]:].flip(0).sqrt(), "product": u @ (u.T @ error)}


# ----------------------------------------------------------------------------
# what a pass cannot do without, and how far two correct passes may lie apart
# ----------------------------------------------------------------------------
def _pass(tokens, k, ns, rank):
    r = rank * len(ns)
    n = sum(ns)
    b = 2 * tokens * k + 4 * k + 2 * r * k                       # X, s, L_A
    b += n * k // 2 + 4 * n + 2 * n * rank + 2 * tokens * n      # weights, scales, L_B, Y
    return b, 2 * tokens * k * n + 2 * tokens * r * k + 2 * tokens * rank * n


def work(case):
    kind = case["kind"]
    if kind == "block":
        t, r = case["tokens"], case["rank"]
        parts = [_pass(t, HIDDEN, (HIDDEN, KV, KV), r), _pass(t, HIDDEN, (HIDDEN,), r),
                 _pass(t, HIDDEN, (MLP, MLP), r), _pass(t, MLP, (HIDDEN,), r)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    k, n = case["k"], case["n"]
    if kind == "pack":
        return {"bytes": 2 * n * k + 4 * k + n * k // 2 + 4 * n + n * k // 2, "flops": 2 * n * k}
    if kind == "construct":
        c, r = case["calibration"], case["rank"]
        # Gram matrix (symmetric), Cholesky factor, E S (triangular), one two-sided projection on
        # the singular subspace, the solve for L_A, the product of the factors
        flops = c * k * k + k ** 3 / 3 + n * k * k + 4 * n * k * r + r * k * k + 2 * n * k * r
        return {"bytes": 2 * n * k + 2 * c * k + n * k // 2 + 2 * r * (n + k) + 4 * n * k, "flops": flops}
    b, f = _pass(case["tokens"], k, (n,) * case.get("layers", 1), case["rank"])
    if kind == "variant":
        b += case["tokens"] * k + 4 * case["tokens"]             # codes and scales are outputs too
    return {"bytes": b, "flops": f}


def tolerance(case):
    if case["kind"] == "pack":
        return "exact"
    if case["kind"] == "construct":
        # 4e-4 and 1.4e-2 seen between 48 subspace iterations and the exact triplets, factors in fp16
        return {"rel": 2e-3, "max": 0.05, "differ": 0.0}
    # against fp64 sums: rel 2.1e-4 .. 2.5e-4 (fp16 result, bf16 T), largest 1.1e-3
    return {"rel": 1e-3, "max": 4e-3, "differ": 0.0}
