"""The measured workloads of the pQuant layer: quantisation-aware training steps of one linear, forward passes of
training size without a backward (prefill), and decode from packed sign bits.

A case is a dict of sizes and options; `prepare` makes a user's buffers on the GPU from a seed, `run` is one pass through
the library's entry points (`PQLinear`, `pq_linear_forward_hp8`, `pq_ffn_forward`, `pq_decode_batch`).  Inputs follow the
distributions of `paper_2602_22592_b200/inputs.py` (activations N(0, 1), weights N(0, 0.02), a Zipf(1.1) expert planted
per token), drawn on the device.
"""
import math

import torch

from paper_2602_22592_b200 import binding as pqb
from paper_2602_22592_b200.inputs import zipf_shares
from paper_2602_22592_b200.layer import PQLinear

DEV = "cuda:0"
PLANT = 6.0          # router margin of the planted expert
NORM_EPS = 1e-5


def listed():
    return [
        # ---- one quantisation-aware training step of a linear: pack the latent weights, forward, straight-through backward
        # the smallest layer: 256 tokens, 512 -> 512, one dense branch of width 32, per-feature scales (launches and latency)
        dict(name="train_256x512", kind="train", T=256, K=512, N=512, r=32, E=1, vector=True),
        # a short batch on sizes that are multiples of 32 and of nothing larger: partial tiles in every direction, three experts
        dict(name="train_1000_ragged_e3", kind="train", T=1000, K=2080, N=992, r=40, E=3, vector=True),
        # attention-shaped projection of a 1.3B model with eight experts (four of the seven linears of a decoder block)
        dict(name="train_8192_attn_e8", kind="train", T=8192, K=2048, N=2048, r=128, E=8, vector=False),
        # gate / up projection of a 1.3B model, dense high-precision branch
        dict(name="train_8192_up_dense", kind="train", T=8192, K=2048, N=5632, r=128, E=1, vector=False),
        # down projection of the same model with eight experts and skewed routing: the long contraction of the forward
        dict(name="train_8192_down_e8", kind="train", T=8192, K=5632, N=2048, r=128, E=8, vector=False),
        # ---- forward only, many tokens (a prompt), nothing kept for a backward
        # up projection of a 3B model, experts in INT8
        dict(name="prefill_2048_up_hp8", kind="prefill_hp8", T=2048, K=3200, N=8640, r=128, E=8, vector=False),
        # the whole gated FFN of a 1.3B model in the FFN-level form (1-bit FFN beside an INT8 FFN of width 128)
        dict(name="prefill_2048_ffn", kind="prefill_ffn", T=2048, K=2048, N=5504, r=128, E=1, vector=False),
        # ---- decode from packed sign bits, up to 16 tokens
        # one call for one attention-shaped linear of a 1.3B model, one token: what a lone call costs
        dict(name="decode_one_m1", kind="decode", M=1, K=2048, N=2048, r=128, E=8, layers=1, form="single", hp8=False, norm=False),
        # one token through the MLP projections of a 26-layer 3B model, in the order a sequence needs them: gate and up of a
        # layer in one call (same activations, RMSNorm in front), then down
        dict(name="decode_step_m1", kind="decode", M=1, K=3200, N=8640, r=160, E=8, layers=26, form="mlp", hp8=False, norm=True),
        # the same for a batch of 16 sequences
        dict(name="decode_step_m16", kind="decode", M=16, K=3200, N=8640, r=160, E=8, layers=26, form="mlp", hp8=False, norm=True),
        # four tokens, INT8 experts, a shorter model
        dict(name="decode_step_m4_hp8", kind="decode", M=4, K=3200, N=8640, r=160, E=8, layers=8, form="mlp", hp8=True, norm=True),
        # all 78 linears as independent work in one call (several replicas or speculative branches side by side), four tokens each
        dict(name="decode_all_m4", kind="decode", M=4, K=3200, N=8640, r=160, E=8, layers=26, form="together", hp8=False, norm=False),
    ]


def _log(rng, lo, hi, step):
    """A multiple of `step`, spread evenly over the logarithm of [lo, hi]."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi // step * step, max(step, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "prefill_hp8", "prefill_ffn", "decode", "decode", "decode", "decode"])
    if kind == "decode":
        form = rng.choice(["single", "mlp", "mlp", "together"])
        while True:
            K, N = _log(rng, 512, 4096, 32), _log(rng, 512, 8640, 32)
            if K * N <= 3200 * 8640:
                break
        hp8 = rng.random() < 0.3
        layers = 1 if form == "single" else _log(rng, 2, 26, 1)
        return dict(kind="decode", M=_log(rng, 1, 16, 1), K=K, N=N, r=rng.choice([32, 64, 96, 128, 160] if hp8 else [0, 32, 40, 96, 128, 160]),
                    E=rng.choice([1, 4, 8]), layers=layers, form=form, hp8=hp8, norm=rng.random() < 0.5)
    most = 8192 * 2048 * 5632
    while True:
        T = rng.randint(128, 8192) if rng.random() < 0.5 else _log(rng, 128, 8192, 1)
        K, N = _log(rng, 256, 5632, 32), _log(rng, 256, 8640, 32)
        if T * K * N <= (most // 3 if kind == "prefill_ffn" else most):
            break
    if kind == "train":
        r = rng.choice([0, 32, 40, 64, 128, 128])
        return dict(kind=kind, T=T, K=K, N=N, r=r, E=rng.choice([1, 3, 8, 8]), vector=rng.random() < 0.3)
    return dict(kind=kind, T=T, K=K, N=N, r=rng.choice([32, 64, 128]), E=1 if kind == "prefill_ffn" else rng.choice([1, 4, 8]), vector=False)


# --------------------------------------------------------------------------- inputs
def _normal(g, shape, dtype=torch.bfloat16, std=1.0):
    return (torch.randn(shape, generator=g, device=DEV, dtype=torch.float32) * std).to(dtype)


def _tokens(g, T, K, Wr):
    """Activations [T, K] and, with a router, an expert planted per token (shares ~ Zipf(1.1))."""
    x = torch.randn((T, K), generator=g, device=DEV, dtype=torch.float32)
    if Wr is not None:
        share = torch.tensor(zipf_shares(Wr.shape[0]), dtype=torch.float32, device=DEV)
        x += PLANT * Wr.float()[torch.multinomial(share, T, replacement=True, generator=g)]
    return x.to(torch.bfloat16)


def _fill(L, g, X=None, latent=True):
    """Weights, experts, router and scales of one layer; its activations are X, or drawn to suit its router."""
    E = max(L.E, 1)
    L.W = _normal(g, (L.N, L.K), torch.float32, 0.02) if latent else None
    if L.r > 0:
        L.A = _normal(g, (E, L.r, L.K), std=0.02)
        L.B = _normal(g, (E, L.N, L.r), std=0.02)
        L.Wr = _normal(g, (E, L.K), std=L.K ** -0.5) if L.E > 1 else None
    n = L.N if L.scale_vector else 1
    spread = torch.rand((2, n), generator=g, device=DEV) * 0.2 + 0.9 if L.scale_vector else torch.ones((2, 1), device=DEV)
    L.alpha, L.beta = (2.0 * spread[0]).contiguous(), (0.2 * spread[1]).contiguous()
    L.X = _tokens(g, L.T, L.K, L.Wr) if X is None else X
    return L


def _prepare_train(c, g):
    L = _fill(PQLinear(c["T"], c["K"], c["N"], c["r"], c["E"], scale_vector=c["vector"], device=DEV), g)
    L.dY = _normal(g, (L.T, L.N))
    return L


def _prepare_hp8(c, g):
    """A packed layer with INT8 experts; forward only, so no buffer is kept for a backward."""
    T, K, N, r, E = c["T"], c["K"], c["N"], c["r"], c["E"]
    L = _fill(PQLinear(16, K, N, r, E, device=DEV, training=False), g, X=torch.empty(0, device=DEV))   # weights only
    pqb.pq_pack_weights(L.desc, L.W, L.w_bits, L.w_s8, L.w_scales, L.ws_pack)
    L.pack_experts()
    L.W = None
    d = pqb.make_desc(T, K, N, r, L.E)
    return dict(L=L, d=d, X=_tokens(g, T, K, L.Wr), Y=torch.empty((T, N), dtype=torch.bfloat16, device=DEV),
                ws=torch.empty(pqb.pq_workspace_bytes(d, pqb.PQ_PHASE_FWD), dtype=torch.uint8, device=DEV))


def _prepare_ffn(c, g):
    T, D, F1, r = c["T"], c["K"], c["N"], c["r"]
    s = dict(d=pqb.make_ffn_desc(T, D, F1, r), X=_tokens(g, T, D, None), Y=torch.empty((T, D), dtype=torch.bfloat16, device=DEV))
    for name, n, k in (("gate", F1, D), ("up", F1, D), ("down", D, F1)):
        L = PQLinear(16, k, n, device=DEV, training=False)
        pqb.pq_pack_weights(L.desc, _normal(g, (n, k), torch.float32, 0.02), L.w_bits, L.w_s8, L.w_scales, L.ws_pack)
        s[name] = (L.w_s8, L.w_scales)
    G, U, Dn = _normal(g, (1, r, D), std=0.02), _normal(g, (1, r, D), std=0.02), _normal(g, (1, D, r), std=0.02)
    desc, ws = pqb.make_desc(T, D, D, r, 1), torch.empty(1 << 16, dtype=torch.uint8, device=DEV)

    def pack8(a, b):
        a8, b8, sc = torch.empty_like(a, dtype=torch.int8), torch.empty_like(b, dtype=torch.int8), torch.empty((1, 2), device=DEV)
        pqb.pq_pack_experts(desc, a, b, a8, b8, sc, ws)
        return a8, b8, sc
    G8, D8, gd = pack8(G, Dn)
    U8, _, ud = pack8(U, Dn)
    s.update(G8=G8, U8=U8, D8=D8, scales=torch.stack([gd[0, 0], ud[0, 0], gd[0, 1]]).contiguous(), alpha=torch.full((1,), 2.0, device=DEV),
             beta=torch.full((1,), 0.2, device=DEV), ws=torch.empty(pqb.pq_ffn_workspace_bytes(s["d"]), dtype=torch.uint8, device=DEV))
    return s


def _decode_layer(c, g, K, N, Y, X=None, norm=False):
    L = _fill(PQLinear(c["M"], K, N, c["r"], c["E"], device=DEV, training=False), g, X)
    L.Y = Y
    L.pack(bits_only=True)          # also lays the weights out for the streaming kernel
    if c["hp8"]:
        L.pack_decode_hp8()
    if norm:
        L.norm_weight, L.norm_eps = _normal(g, (K,), std=0.1) + 1.0, NORM_EPS
    L.W = L.w_s8 = None             # a decoder keeps the packed form only
    return L


def _prepare_decode(c, g):
    """The layers' outputs are slices of one tensor per projection; `calls` holds the argument arrays, one per library call."""
    M, K, N, n = c["M"], c["K"], c["N"], c["layers"]

    def out(width):
        return torch.empty((n, M, width), dtype=torch.bfloat16, device=DEV)
    if c["form"] == "single":
        Y = out(N)
        layers = [[_decode_layer(c, g, K, N, Y[0], norm=c["norm"])]]
        outs = [Y]
    else:
        outs = [out(N), out(N), out(K)]
        layers = []
        for i in range(n):
            gate = _decode_layer(c, g, K, N, outs[0][i], norm=c["norm"])
            up = _decode_layer(c, g, K, N, outs[1][i], X=gate.X)
            if c["norm"]:
                up.norm_weight, up.norm_eps = gate.norm_weight, gate.norm_eps
            layers += [[gate, up], [_decode_layer(c, g, N, K, outs[2][i])]]
        if c["form"] == "together":
            layers = [[L for call in layers for L in call]]
    return dict(layers=layers, outs=outs, calls=[pqb.make_decode_items([L.decode_entry() for L in call]) for call in layers])


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return case["kind"], {"train": _prepare_train, "prefill_hp8": _prepare_hp8, "prefill_ffn": _prepare_ffn, "decode": _prepare_decode}[case["kind"]](case, g)


# --------------------------------------------------------------------------- one pass
def run(state):
    kind, s = state
    if kind == "train":
        s.pack()
        s.forward()
        s.backward()
        grads = dict(dX=s.dX, dW=s.dW, dbeta=s.dbeta)
        if s.r > 0:
            grads.update(dA=s.dA, dB=s.dB, dWr=s.dWr, dalpha=s.dalpha)
        return dict(Y=s.Y, bits=s.w_bits, scales=s.w_scales, **grads)
    if kind == "prefill_hp8":
        L = s["L"]
        pqb.pq_linear_forward_hp8(s["d"], s["X"], L.w_s8, L.w_scales, L.A8, L.B8, L.hp_scales, L.Wr, L.alpha, L.beta, s["Y"], None, s["ws"])
        return s["Y"]
    if kind == "prefill_ffn":
        pqb.pq_ffn_forward(s["d"], s["X"], *s["gate"], *s["up"], *s["down"], s["G8"], s["U8"], s["D8"], s["scales"], s["alpha"], s["beta"], s["Y"], s["ws"])
        return s["Y"]
    for items in s["calls"]:
        pqb.pq_decode_batch(items)
    return s["outs"]


# --------------------------------------------------------------------------- what a pass cannot do without
def _decode_linear_work(c, K, N, reads_x):
    M, r, E = c["M"], c["r"], c["E"] if c["r"] > 0 else 0
    used = sum(1 - (1 - p) ** M for p in zipf_shares(E)) if E > 1 else min(E, 1)      # experts that some token is routed to
    width = 1 if c["hp8"] else 2
    by = N * K / 8 + used * width * r * (K + N) + (2 * E * K if E > 1 else 0) + (2 * M * K if reads_x else 0) + 2 * M * N
    return by, 2 * M * (N * K + r * (K + N) + (E * K if E > 1 else 0))


def work(case):
    c = case
    if c["kind"] == "decode":
        K, N = c["K"], c["N"]
        parts = [_decode_linear_work(c, K, N, True)]
        if c["form"] != "single":
            parts += [_decode_linear_work(c, K, N, False), _decode_linear_work(c, N, K, True)]
        return dict(bytes=c["layers"] * sum(p[0] for p in parts), flops=c["layers"] * sum(p[1] for p in parts))
    T, K, N, r, E = c["T"], c["K"], c["N"], c["r"], max(c["E"], 1) if c["r"] > 0 else 0
    router = E * K if E > 1 else 0
    if c["kind"] == "train":
        # read X, dY, W, A, B, Wr; write Y, dX, the packed words, dW, dA, dB, dWr.  Three products of the 1-bit branch, six of the experts'
        by = 2 * T * (2 * K + 2 * N) + N * K * (4 + 4 + 1 / 8) + 6 * E * r * (K + N) + 6 * router
        return dict(bytes=by, flops=6 * T * N * K + 6 * T * r * (K + N) + 6 * T * router)
    if c["kind"] == "prefill_hp8":
        return dict(bytes=2 * T * (K + N) + N * K + E * r * (K + N) + 2 * router, flops=2 * T * (N * K + r * (K + N) + router))
    return dict(bytes=4 * T * K + 3 * N * K + 3 * r * K, flops=2 * T * 3 * K * (N + r))


def tolerance(case):
    # Measured against the same layer in 64-bit arithmetic: outputs and gradients that pass through bf16 (Y, dX, dW, dA,
    # dWr, dbeta) are off by 1.7e-3 .. 2.5e-3 of their norm and by at most 1.5e-2 of a value's scale; dB and dalpha by
    # 2e-6 .. 3e-5.  About four times the larger ones.  Packed sign words are whole numbers and have to be the same.
    return {"rel": 1e-2, "max": 5e-2}
