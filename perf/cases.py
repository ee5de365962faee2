"""The work that users of this package have it do, as cases that can be timed and compared.

A case is a dict of plain values.  Six kinds of work, all through the public entry points:

  linear    one quantised FC layer, fp32 in and fp32 out (`q8_linear`)
  ffn       the two FC layers of a feed-forward block chained in Int8 (`q8_linear_requant` + `q8_linear_q`)
  fc_set    embedding gather plus the four FC layers of one encoder block on independent inputs (the benchmark step)
  encoder   a whole encoder forward: static scales, dynamic scales, or a captured CUDA graph of the static forward
  weights   quantisation of a weight matrix or embedding table when a model is loaded (`q8_quantize_weight`)
  training  one fake-quantised tensor of quantisation-aware training, forward and backward (`q8_calibrate`,
            `q8_fake_quantize`, `q8_ste_backward`)

Inputs follow paper_1910_06188_b200/synth.py: weights, biases and tables ~ N(0, 0.02), activations ~ N(0, 1) with one
entry in a hundred multiplied by 8, token ids uniform.  FC inputs are drawn on the GPU (the same distributions); the
encoder draws its own weights.
"""
import math

import torch

from paper_1910_06188_b200 import binding as q8
from paper_1910_06188_b200 import synth
from paper_1910_06188_b200.encoder import Q8BertEncoder, random_ids

DIMS = {"base": synth.BERT_BASE, "large": synth.BERT_LARGE}
DECAY = 0.9999


def listed():
    return [
        # one layer on one short sequence, scale taken from the incoming tensor: the smallest call there is
        dict(name="linear_dynamic_128x768", kind="linear", M=128, K=768, N=768, act=0, scale="dynamic"),
        # a layer whose width is not a multiple of 16, on a token count that is not a multiple of any tile
        dict(name="linear_odd_1000x300", kind="linear", M=1000, K=300, N=1200, act=1, scale="dynamic"),
        # feed-forward block on one unpadded 509-token batch, Int8 between its two layers
        dict(name="ffn_large_509", kind="ffn", M=509, H=1024, F=4096),
        # the benchmark's FC sets: BERT-Base on 32 x 128 tokens, BERT-Large on 64 x 384 tokens
        dict(name="fc_set_base_4096", kind="fc_set", model="base", M=4096),
        dict(name="fc_set_large_24576", kind="fc_set", model="large", M=24576),
        # a served model answering one query at a time, replayed from a graph.  (The encoder cases run a few of the
        # models' 12 or 24 identical layers: see tolerance())
        dict(name="encoder_base_1x128_graph", kind="encoder", model="base", layers=6, B=1, S=128, mode="graph"),
        # a served model on a full batch
        dict(name="encoder_base_32x128", kind="encoder", model="base", layers=6, B=32, S=128, mode="static"),
        # dynamic quantisation (no calibration data), sequences of a length that fills no tile
        dict(name="encoder_base_7x203_dynamic", kind="encoder", model="base", layers=4, B=7, S=203, mode="dynamic"),
        # the longest sequences the models take (512 positions)
        dict(name="encoder_base_16x512", kind="encoder", model="base", layers=4, B=16, S=512, mode="static"),
        # question answering at throughput: BERT-Large blocks on 64 x 384 tokens
        dict(name="encoder_large_64x384", kind="encoder", model="large", layers=3, B=64, S=384, mode="static"),
        # loading a model: the word table of BERT-Large is its largest tensor
        dict(name="weights_30522x1024", kind="weights", N=30522, K=1024),
        # quantisation-aware training: the widest activation of a BERT-Base batch of 32 x 128 tokens
        dict(name="training_4096x3072", kind="training", M=4096, K=3072),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _width(rng, lo, hi):
    """A layer width: mostly a multiple of 64 as models have it, sometimes only of 16, seldom anything at all."""
    w = _log_int(rng, lo, hi)
    step = rng.choice((64, 64, 64, 16, 1))
    return max(step, w // step * step)


def draw(rng):
    kind = rng.choice(("linear", "linear", "ffn", "fc_set", "encoder", "encoder", "encoder", "weights", "training"))
    if kind == "linear":
        return dict(kind=kind, M=_log_int(rng, 1, 8192), K=_width(rng, 64, 4096), N=_width(rng, 64, 4096),
                    act=rng.randrange(2), scale=rng.choice(("static", "dynamic")))
    if kind == "ffn":
        H = rng.choice((512, 768, 1024))
        return dict(kind=kind, M=_log_int(rng, 16, 16384), H=H, F=4 * H)
    if kind == "fc_set":
        return dict(kind=kind, model=rng.choice(("base", "large")), M=_log_int(rng, 64, 16384))
    if kind == "encoder":
        S = _log_int(rng, 16, 512)
        B = _log_int(rng, 1, max(1, 16384 // S))
        return dict(kind=kind, model=rng.choice(("base", "large")), layers=rng.randint(2, 3), B=B, S=S,
                    mode=rng.choice(("static", "dynamic", "graph")))
    if kind == "weights":
        return dict(kind=kind, N=_log_int(rng, 512, 30522), K=_width(rng, 256, 1024))
    return dict(kind=kind, M=_log_int(rng, 64, 16384), K=_width(rng, 256, 3072))


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _activation(g, *shape):
    x = torch.randn(shape, generator=g, device="cuda")
    outlier = torch.rand(shape, generator=g, device="cuda") < synth.OUTLIER_PROB
    return x.mul_(1.0 + (synth.OUTLIER_GAIN - 1.0) * outlier)


def _weight(g, *shape):
    return torch.randn(shape, generator=g, device="cuda").mul_(synth.WEIGHT_SIGMA)


def _calibrated(x):
    """Eq. 4 state after one calibration batch, and the scale a static layer takes from it."""
    state = q8.new_calibrate_state()
    q8.q8_calibrate(x, DECAY, state)
    return state, q8.calibrate_S_x(state)


def _layer(g, M, K, N, act, static):
    """A loaded layer, its input and what a serving program keeps beside it."""
    X = _activation(g, M, K)
    Wq, S_w = q8.q8_quantize_weight(_weight(g, N, K))
    lay = dict(X=X, Wq=Wq, S_w=S_w, bias=_weight(g, N), act=act, S_x=None, workspace=q8.new_workspace(M, N, K))
    if static:
        lay["state"], lay["S_x"] = _calibrated(_activation(g, M, K))
    return lay


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind == "linear":
        return dict(case=case, layer=_layer(g, case["M"], case["K"], case["N"], case["act"], case["scale"] == "static"))
    if kind == "ffn":
        M, H, F = case["M"], case["H"], case["F"]
        up, down = _layer(g, M, H, F, 1, True), _layer(g, M, F, H, 0, True)
        return dict(case=case, up=up, down=down)
    if kind == "fc_set":
        dims, M = DIMS[case["model"]], case["M"]
        layers = [_layer(g, M, K, N, act, True) for _, K, N, act in synth.fc_set(dims["hidden"], dims["ffn"])]
        for lay in layers:
            lay["Y"] = torch.empty((M, lay["Wq"].shape[0]), device="cuda")
        Eq, S_e = q8.q8_quantize_weight(_weight(g, dims["vocab"], dims["hidden"]))
        ids = torch.randint(dims["vocab"], (M,), generator=g, device="cuda", dtype=torch.int32)
        return dict(case=case, layers=layers, Eq=Eq, S_e=S_e, ids=ids, rows=torch.empty((M, dims["hidden"]), device="cuda"))
    if kind == "encoder":
        B, S = case["B"], case["S"]
        enc = Q8BertEncoder(DIMS[case["model"]], config=seed, layers=case["layers"])
        ids = random_ids(B * S, enc.V, seed)
        if case["mode"] != "dynamic":
            enc.forward(random_ids(B * S, enc.V, seed + 1), B, S, scales="calibrate", decay=DECAY)
        state = dict(case=case, encoder=enc, ids=ids, B=B, S=S)
        if case["mode"] == "graph":
            state["graph"], state["out"] = enc.capture(ids, B, S)
        return state
    if kind == "weights":
        return dict(case=case, W=_weight(g, case["N"], case["K"]))
    X = _activation(g, case["M"], case["K"])
    state, _ = _calibrated(_activation(g, case["M"], case["K"]))
    grad = torch.randn(X.shape, generator=g, device="cuda")
    return dict(case=case, X=X, grad=grad, start=state, state=state.clone())


# ------------------------------------------------------------------ one pass
def run(state):
    kind = state["case"]["kind"]
    if kind == "linear":
        a = state["layer"]
        return q8.q8_linear(a["X"], a["Wq"], a["S_w"], a["S_x"], a["bias"], a["act"], workspace=a["workspace"])
    if kind == "ffn":
        a, b = state["up"], state["down"]
        mid = q8.q8_linear_requant(a["X"], a["Wq"], a["S_w"], a["S_x"], a["bias"], a["act"], b["S_x"],
                                   workspace=a["workspace"])
        return q8.q8_linear_q(mid, b["S_x"], b["Wq"], b["S_w"], b["bias"], b["act"]), mid
    if kind == "fc_set":
        q8.q8_embedding(state["ids"], state["Eq"], state["S_e"], out=state["rows"])
        for a in state["layers"]:
            q8.q8_linear(a["X"], a["Wq"], a["S_w"], a["S_x"], a["bias"], a["act"], Y=a["Y"], workspace=a["workspace"])
        return [state["rows"]] + [a["Y"] for a in state["layers"]]
    if kind == "encoder":
        mode = state["case"]["mode"]
        if mode == "graph":
            state["graph"].replay()
            return state["out"]
        forward = state["encoder"].forward_fused if mode == "static" else state["encoder"].forward_dynamic_fused
        return forward(state["ids"], state["B"], state["S"])
    if kind == "weights":
        return q8.q8_quantize_weight(state["W"])
    state["state"].copy_(state["start"])  # every pass is the same training step
    q8.q8_calibrate(state["X"], DECAY, state["state"])
    S = q8.calibrate_S_x(state["state"])
    xhat = q8.q8_fake_quantize(state["X"], S)
    return xhat, q8.q8_ste_backward(state["grad"]), S


# ------------------------------------------------------------------ the same results in 64 bits, in plain torch
def _plain_scale(x):
    m = x.abs().max().float()
    return torch.full_like(m, 127.0) / m  # (127.0 / m would be computed as 127 times the rounded reciprocal)


def _plain_quantize(x, S):
    """Integers of Eq. 1 as float64.  The paper's product x * S is formed in the precision of x."""
    return torch.clamp(torch.round(x * S.to(x.dtype)), -127, 127).double()


def _plain_linear(Xq, S_x, Wq, S_w, bias, act):
    """Integer operands held as float64: the matrix product is exact."""
    S = S_x * S_w
    y = (Xq @ Wq.T + torch.round(bias * S).double()) / S.double()
    return torch.nn.functional.gelu(y) if act else y


def _plain_layer(g, M, K, N, act, static):
    """The draws of _layer(), in its order."""
    X, W = _activation(g, M, K), _weight(g, N, K)
    S_w = _plain_scale(W)
    lay = dict(X=X, Wq=_plain_quantize(W, S_w), S_w=S_w, bias=_weight(g, N), act=act)
    lay["S_x"] = _plain_scale(_activation(g, M, K) if static else X)
    return lay


def _plain_encoder(case, seed):
    """The whole forward in float64.  A value next to a rounding boundary of a quantiser may fall on its other side here,
    as it may in any other implementation: the results agree to the size of that noise (see tolerance())."""
    dims, B, S = DIMS[case["model"]], case["B"], case["S"]
    H, heads = dims["hidden"], dims["heads"]

    def draw_weight(n, k, index):
        w = torch.from_numpy(synth.weight(n, k, synth.seed_for(seed, index))).cuda()
        S_w = _plain_scale(w)
        return _plain_quantize(w, S_w), S_w

    tables = [draw_weight(n, H, 100 + i) for i, n in enumerate((dims["vocab"], dims["max_pos"], 2))]
    layers = [[draw_weight(N, K, 200 + 20 * l + 2 * i)
               + (torch.from_numpy(synth.bias(N, synth.seed_for(seed, 200 + 20 * l + 2 * i + 1))).cuda(), act)
               for i, (_, K, N, act) in enumerate(synth.fc_set(H, dims["ffn"]))] for l in range(case["layers"])]

    def norm(x):
        x = x - x.mean(1, keepdim=True)
        return x / torch.sqrt((x * x).mean(1, keepdim=True) + 1e-12)

    def forward(ids, scales):
        seen = iter(scales) if scales is not None else None
        taken = []

        def fc(x, layer):
            S_x = next(seen) if seen is not None else _plain_scale(x)
            taken.append(S_x)
            return _plain_linear(_plain_quantize(x, S_x), S_x, *layer)

        places = torch.arange(S, device="cuda").repeat(B)
        rows = (ids.long(), places, torch.zeros_like(places))
        h = norm(sum(E[r] / S_e.double() for (E, S_e), r in zip(tables, rows)))
        for qkv, attn_out, ffn1, ffn2 in layers:
            q, k, v = fc(h, qkv).view(B, S, 3, heads, H // heads).permute(2, 0, 3, 1, 4)
            ctx = torch.softmax(q @ k.transpose(2, 3) / math.sqrt(H // heads), dim=3) @ v
            h = norm(fc(ctx.transpose(1, 2).reshape(B * S, H), attn_out) + h)
            h = norm(fc(fc(h, ffn1), ffn2) + h)
        return h, taken

    ids = random_ids(B * S, dims["vocab"], seed)
    if case["mode"] == "dynamic":
        return forward(ids, None)[0]
    # the first calibration batch sets the running maximum
    return forward(ids, forward(random_ids(B * S, dims["vocab"], seed + 1), None)[1])[0]


def exact(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind == "linear":
        a = _plain_layer(g, case["M"], case["K"], case["N"], case["act"], case["scale"] == "static")
        return _plain_linear(_plain_quantize(a["X"], a["S_x"]), a["S_x"], a["Wq"], a["S_w"], a["bias"], a["act"])
    if kind == "ffn":
        M, H, F = case["M"], case["H"], case["F"]
        a, b = _plain_layer(g, M, H, F, 1, True), _plain_layer(g, M, F, H, 0, True)
        mid = _plain_linear(_plain_quantize(a["X"], a["S_x"]), a["S_x"], a["Wq"], a["S_w"], a["bias"], a["act"])
        mid = _plain_quantize(mid.float(), b["S_x"])
        return _plain_linear(mid, b["S_x"], b["Wq"], b["S_w"], b["bias"], b["act"]), mid.to(torch.int8)
    if kind == "fc_set":
        dims, M = DIMS[case["model"]], case["M"]
        outs = []
        for _, K, N, act in synth.fc_set(dims["hidden"], dims["ffn"]):
            a = _plain_layer(g, M, K, N, act, True)
            outs.append(_plain_linear(_plain_quantize(a["X"], a["S_x"]), a["S_x"], a["Wq"], a["S_w"], a["bias"], a["act"]))
        E = _weight(g, dims["vocab"], dims["hidden"])
        ids = torch.randint(dims["vocab"], (M,), generator=g, device="cuda", dtype=torch.int32)
        S_e = _plain_scale(E)
        return [_plain_quantize(E[ids.long()], S_e) / S_e.double()] + outs
    if kind == "encoder":
        return _plain_encoder(case, seed)
    if kind == "weights":
        W = _weight(g, case["N"], case["K"])
        S_w = _plain_scale(W)
        return _plain_quantize(W, S_w).to(torch.int8), S_w.double().reshape(1)
    X = _activation(g, case["M"], case["K"])
    ema = _activation(g, case["M"], case["K"]).abs().max().double()
    grad = torch.randn(X.shape, generator=g, device="cuda")
    S = _plain_scale(ema + (1.0 - DECAY) * (X.abs().max().double() - ema))
    return _plain_quantize(X, S) / S.double(), grad.double(), S.double().reshape(1)


# ------------------------------------------------------------------ what a pass cannot do without
def _linear_work(M, K, N, in_bytes=4, out_bytes=4):
    return M * K * in_bytes + N * K + 4 * N + M * N * out_bytes, 2 * M * N * K


def work(case):
    kind = case["kind"]
    if kind == "linear":
        b, f = _linear_work(case["M"], case["K"], case["N"])
    elif kind == "ffn":
        up = _linear_work(case["M"], case["H"], case["F"], out_bytes=1)
        down = _linear_work(case["M"], case["F"], case["H"], in_bytes=0)
        b, f = up[0] + down[0], up[1] + down[1]
    elif kind == "fc_set":
        dims, M = DIMS[case["model"]], case["M"]
        parts = [_linear_work(M, K, N) for _, K, N, _ in synth.fc_set(dims["hidden"], dims["ffn"])]
        # each table row is read once, however often it is asked for
        b = sum(p[0] for p in parts) + 4 * M + min(M, dims["vocab"]) * dims["hidden"] + 4 * M * dims["hidden"]
        f = sum(p[1] for p in parts)
    elif kind == "encoder":
        dims, T, L = DIMS[case["model"]], case["B"] * case["S"], case["layers"]
        H, F = dims["hidden"], dims["ffn"]
        b = 4 * T + min(T, dims["vocab"]) * H + min(case["S"], dims["max_pos"]) * H + 4 * T * H
        b += L * sum(N * K + 4 * N for _, K, N, _ in synth.fc_set(H, F))
        f = L * (sum(2 * T * N * K for _, K, N, _ in synth.fc_set(H, F)) + 4 * T * case["S"] * H)
    elif kind == "weights":
        n = case["N"] * case["K"]
        b, f = 5 * n, 3 * n
    else:
        n = case["M"] * case["K"]
        b, f = 16 * n, 4 * n  # X and the gradient in, the fake-quantised X and the passed-on gradient out
    return dict(bytes=b, flops=f)


def tolerance(case):
    kind = case["kind"]
    if kind == "weights":
        return "exact"
    if kind == "training":
        return dict(rel=1e-7, max=4e-7)  # one fp32 division; seen within 2.3e-8 (5.6e-8) of 64 bits
    if kind == "encoder":
        # Attention computed by the two kernels of this package (tensor cores, CUDA cores), both within 4e-6 of a
        # 64-bit result: a last-bit difference turns some roundings to Int8 the other way in the next layer, and
        # after four layers the outputs differ by 1.2e-2 (base) and 1.9e-2 (large), after twelve by 2.8e-2, in
        # single values by 0.14: the size of the quantisation noise, which limits the depth that can be compared.
        return dict(rel=3e-2, max=5e-1)
    # The integers are exact; fp32 values seen within 5e-8 (largest 2.4e-7) of the layer evaluated in 64 bits.
    return dict(rel=4e-7, max=2e-6, differ=1e-4)
