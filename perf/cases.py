"""The work a user of this framework has it do, as measurable cases.

Every case is one pass through the public entry points: a whole encoder (layer after layer, the
way a model is run), the model around it (ids -> embedding -> layers -> classifier) on padded and
on packed batches, a captured graph replayed, a layer composed from the single operators, and the
integer non-linearities on their own.  Shapes are the ones of this repository's configurations
(RoBERTa-Base and -Large), its tests and its benchmark; weights, tables and inputs are seeded
random tensors of the distributions `synth` uses, drawn on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2101_01321_b200 import binding, synth

MODELS = {"base": {"H": 768, "heads": 12, "F": 3072, "layers": 12},
          "large": {"H": 1024, "heads": 16, "F": 4096, "layers": 24}}
VOCAB, LABELS = synth.VOCAB, synth.N_LABELS
S_INPUT = 4.5 / 127.0            # static scale of a unit-variance int8 activation


def listed() -> list[dict]:
    return [
        # one sentence at a time: interactive use, where launches and latency count
        {"name": "base_b1_l128", "kind": "encoder", "model": "base", "B": 1, "L": 128, "p_max": 255},
        # a few short sentences of a service that captured its fixed shape once (L not a multiple of 16)
        {"name": "base_graph_b4_l50", "kind": "graph", "model": "base", "B": 4, "L": 50, "p_max": 255},
        # a small batch padded to an odd length
        {"name": "base_b8_l77", "kind": "encoder", "model": "base", "B": 8, "L": 77, "p_max": 255},
        # sentence classification on a padded batch: ids in, logits out, key-padding mask
        {"name": "base_model_b32_l128", "kind": "model", "model": "base", "B": 32, "L": 128, "p_max": 255},
        # the benchmark's default workload
        {"name": "base_b128_l128", "kind": "encoder", "model": "base", "B": 128, "L": 128, "p_max": 255},
        # the same sentence mix without padding: packed rows and offsets, ids in, logits out
        {"name": "base_packed_b128_l128", "kind": "packed", "model": "base", "B": 128, "L": 128, "p_max": 255},
        # the larger model on paragraphs
        {"name": "large_b32_l256", "kind": "encoder", "model": "large", "B": 32, "L": 256, "p_max": 255},
        # the larger model on full-length documents: the largest workload configured
        {"name": "large_b64_l512", "kind": "encoder", "model": "large", "B": 64, "L": 512, "p_max": 255},
        # a layer composed from the single operators (a caller with its own graph), odd token count,
        # 7-bit probabilities
        {"name": "ops_base_b10_l101", "kind": "ops", "model": "base", "B": 10, "L": 101, "p_max": 127},
        # the non-linearities on their own, at the benchmark's sizes
        {"name": "gelu_16m", "kind": "gelu", "n": 1 << 24},
        {"name": "softmax_r196608_l128", "kind": "softmax", "rows": 196608, "L": 128, "p_max": 255},
        {"name": "layernorm_r16384_c768", "kind": "layernorm", "rows": 16384, "C": 768, "bits": 32},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    kind = rng.choice(["encoder", "encoder", "encoder", "graph", "model", "packed", "packed", "ops",
                       "gelu", "softmax", "layernorm"])
    if kind == "gelu":
        return {"kind": kind, "n": _log_int(rng, 1 << 14, 1 << 24)}
    if kind == "softmax":
        L = rng.randint(16, 512)
        return {"kind": kind, "rows": _log_int(rng, 1000, min(196608, (1 << 26) // L)), "L": L,
                "p_max": rng.choice([255, 127])}
    if kind == "layernorm":
        return {"kind": kind, "rows": _log_int(rng, 100, 32768), "C": rng.choice([256, 512, 768, 1024]),
                "bits": rng.choice([16, 32])}
    model = rng.choice(["base", "large"])
    L = rng.randint(16, 512) if rng.random() < 0.6 else rng.choice([32, 64, 128, 256, 384, 512])
    most = {"graph": 2048, "ops": 8192}.get(kind, 16384)
    B = _log_int(rng, 1, max(1, min(128, most // L)))
    return {"kind": kind, "model": model, "B": B, "L": L, "p_max": rng.choice([255, 255, 127])}


# --------------------------------------------------------------------------- inputs
def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(g, *shape) -> torch.Tensor:
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)


def _int8_activation(g, rows: int, cols: int) -> torch.Tensor:
    return (_normal(g, rows, cols) / S_INPUT).round_().clamp_(-127, 127).to(torch.int8)


def _weight(g, n_out: int, n_in: int):
    """W ~ N(0, 0.02^2) with one symmetric int8 scale per output channel."""
    w = _normal(g, n_out, n_in) * 0.02
    s = w.abs().amax(dim=1).double() / 127.0
    q = (w / s.float()[:, None]).round_().clamp_(-127, 127).to(torch.int8)
    return q, s.cpu().numpy()


def _bias(g, S_in: float, S_w: np.ndarray) -> np.ndarray:
    b = (_normal(g, S_w.size) * 0.02).double().cpu().numpy()
    return np.rint(b / (S_in * S_w)).astype(np.int32)


def _affine(g, n: int):
    v = _normal(g, 2, n).double().cpu().numpy()
    return 1.0 + 0.1 * v[0], 0.1 * v[1]


def _scales(case: dict) -> dict:
    m = MODELS[case["model"]]
    return synth.static_activation_scales(m["H"], m["F"], case["L"], S_INPUT)


def _layer_params(g, case: dict, scales: dict) -> dict:
    """One layer's integer parameters and static scales, as `Layer` takes them."""
    m = MODELS[case["model"]]
    H, F = m["H"], m["F"]
    p = {"H": H, "heads": m["heads"], "F": F, "p_max": case["p_max"], **scales}
    for nm, n_out, n_in, S_in in (("qkv", 3 * H, H, "S_x"), ("o", H, H, "S_ctx"), ("f1", F, H, "S_h1"), ("f2", H, F, "S_go")):
        w, S_w = _weight(g, n_out, n_in)
        p[f"w_{nm}"], p[f"S_w_{nm}"], p[f"bias_{nm}"] = w.cpu().numpy(), S_w, _bias(g, scales[S_in], S_w)
    p["gamma1"], p["beta1"] = _affine(g, H)
    p["gamma2"], p["beta2"] = _affine(g, H)
    return p


def _stack(g, case: dict, ctx) -> list:
    """The model's layers; layer l + 1 reads layer l's output."""
    scales = _scales(case)
    layers = []
    for _ in range(MODELS[case["model"]]["layers"]):
        layers.append(ctx.ibert_layer_create(_layer_params(g, case, scales)))
        scales = {**scales, "S_x": scales["S_out"]}
    return layers


def _lengths(seed: int, B: int, L: int) -> np.ndarray:
    """A sentence-length mix: half of the batch in [L/8, L/2], half in [L/2, L], one full sequence.
    The lengths belong to the case (a packed batch's size follows from them), their order to the seed."""
    rng = np.random.default_rng(1000 * B + L)
    short, long_ = rng.integers(max(L // 8, 1), L // 2 + 1, B), rng.integers(L // 2, L + 1, B)
    lens = np.where(rng.random(B) < 0.5, short, long_).astype(np.int32)
    lens[0] = L
    return np.random.default_rng(seed).permutation(lens)


def prepare(case: dict, seed: int) -> dict:
    g = _gen(seed)
    kind = case["kind"]
    st = {"case": case}
    if kind == "graph":
        st["stream"] = torch.cuda.Stream()
        st["ctx"] = binding.Context(0, st["stream"])
    else:
        st["ctx"] = binding.Context(0)
    ctx = st["ctx"]
    if kind == "gelu":
        x = _normal(g, case["n"])
        amax = float(x.abs().max())
        st.update(q=(x * (32767.0 / amax)).round_().clamp_(-32767, 32767).to(torch.int32), S=amax / 32767.0, S_out=amax / 127.0)
        return st
    if kind == "softmax":
        st.update(q=(_normal(g, case["rows"], case["L"]) * 16384.0).round_().to(torch.int32), S=1.0 / 16384.0)
        return st
    if kind == "layernorm":
        rows, C = case["rows"], case["C"]
        x = _normal(g, rows, C) + 0.5 * _normal(g, rows, 1)
        r = 0.25 * _normal(g, rows, C)
        S, S_r = float((x + r).abs().max()) / 32767.0, float(r.abs().max()) / 127.0
        gamma, beta = _affine(g, C)
        st.update(q=(x / S).round_().clamp_(-32767, 32767).to(torch.int16 if case["bits"] == 16 else torch.int32), S=S,
                  r=(r / S_r).round_().clamp_(-127, 127).to(torch.int8), S_r=S_r, gamma=gamma, beta=beta, S_out=4.5 * 1.01 / 127.0)
        return st

    m = MODELS[case["model"]]
    H, B, L = m["H"], case["B"], case["L"]
    if kind in ("encoder", "graph"):
        st.update(layers=_stack(g, case, ctx), x=_int8_activation(g, B * L, H))
        if kind == "graph":
            st["out"] = torch.empty((B * L, H), dtype=torch.int8, device="cuda")
            torch.cuda.synchronize()
            st["graph"] = binding.Graph(ctx, st["layers"], st["x"], B, L, st["out"])
        return st
    if kind == "ops":
        p = _layer_params(g, case, _scales(case))
        for nm in ("qkv", "o", "f1", "f2"):
            p[f"w_{nm}"] = torch.from_numpy(p[f"w_{nm}"]).cuda()
            p[f"bias_{nm}"] = torch.from_numpy(p[f"bias_{nm}"]).cuda()
        # the calls take one output scale: Q, K and V share theirs
        st.update(p=p, x=_int8_activation(g, B * L, H))
        return st

    # ids -> embedding -> layers -> classifier
    lens = _lengths(seed, B, L)
    scales = _scales(case)
    word, S_word = _normal(g, VOCAB, H) * 0.02, 0.02 * 5.0 / 127.0
    pos = _normal(g, L + 2, H) * 0.02
    gamma, beta = _affine(g, H)
    tokens = B * L if kind == "model" else int(lens.sum())
    w, S_w = _weight(g, LABELS, H)
    st.update(layers=_stack(g, case, ctx), lens=torch.from_numpy(lens).cuda(),
              cu=torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)).cuda(),
              ids=torch.randint(0, VOCAB, (tokens,), generator=g, device="cuda", dtype=torch.int32),
              word=(word / S_word).round_().clamp_(-127, 127).to(torch.int8), S_word=S_word,
              pos=(pos / S_word).round_().clamp_(-127, 127).to(torch.int8), S_pos=S_word, gamma=gamma, beta=beta,
              head_w=w, head_S_w=S_w, head_bias=torch.from_numpy(_bias(g, scales["S_out"], S_w)).cuda(), S_last=scales["S_out"])
    return st


# --------------------------------------------------------------------------- one pass
def run(st: dict):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "gelu":
        return ctx.ibert_gelu_i(st["q"], st["S"], st["S_out"])[0]
    if kind == "softmax":
        return ctx.ibert_softmax_i(st["q"], st["S"], case["p_max"])[0]
    if kind == "layernorm":
        return ctx.ibert_layernorm_i(st["q"], st["S"], st["r"], st["S_r"], st["gamma"], st["beta"], st["S_out"])[0]
    B, L = case["B"], case["L"]
    if kind == "encoder":
        h = st["x"]
        for layer in st["layers"]:
            h, _ = ctx.ibert_encoder_layer(layer, h, B, L)
        return h
    if kind == "graph":
        here = torch.cuda.current_stream()
        st["stream"].wait_stream(here)
        out = st["graph"].launch()
        here.wait_stream(st["stream"])
        return out
    if kind == "ops":
        p, x = st["p"], st["x"]
        H, heads = p["H"], p["heads"]
        qkv, _ = ctx.ibert_linear_i8(x, p["S_x"], p["w_qkv"], p["S_w_qkv"], p["bias_qkv"], 0, p["S_q"])
        c, _ = ctx.ibert_attention_i8(qkv, B, L, H, heads, p["S_q"], p["S_q"], p["S_q"], p["S_ctx"], p["p_max"])
        h1, _ = ctx.ibert_linear_layernorm_i8(c, p["S_ctx"], p["w_o"], p["S_w_o"], p["bias_o"], p["S_r1"], x, p["S_x"],
                                              p["gamma1"], p["beta1"], p["S_h1"])
        f, _ = ctx.ibert_linear_gelu_i8(h1, p["S_h1"], p["w_f1"], p["S_w_f1"], p["bias_f1"], p["S_gi"], p["S_go"])
        r2, _ = ctx.ibert_linear_i8(f, p["S_go"], p["w_f2"], p["S_w_f2"], p["bias_f2"], 3, p["S_r2"])
        out, _ = ctx.ibert_layernorm_i(r2, p["S_r2"], h1, p["S_h1"], p["gamma2"], p["beta2"], p["S_out"])
        return {"qkv": qkv, "context": c, "h1": h1, "ffn": f, "sum": r2, "out": out}
    if kind == "model":
        h, _ = ctx.ibert_embedding_i8(st["ids"], L, st["word"], st["S_word"], st["pos"], st["S_pos"], st["gamma"],
                                      st["beta"], S_INPUT)
        for layer in st["layers"]:
            h, _ = ctx.ibert_encoder_layer_masked(layer, h, B, L, st["lens"])
        logits, _ = ctx.ibert_classifier_i8(h, B, L, st["S_last"], st["head_w"], st["head_S_w"], st["head_bias"])
    else:
        h, _ = ctx.ibert_embedding_packed_i8(st["ids"], st["cu"], L, st["word"], st["S_word"], st["pos"], st["S_pos"],
                                             st["gamma"], st["beta"], S_INPUT)
        for layer in st["layers"]:
            h, _ = ctx.ibert_encoder_layer_packed(layer, h, st["cu"], L)
        logits, _ = ctx.ibert_classifier_packed_i8(h, st["cu"], st["S_last"], st["head_w"], st["head_S_w"], st["head_bias"])
    return {"hidden": h, "logits": logits}


# --------------------------------------------------------------------------- what a pass cannot do without
def work(case: dict) -> dict:
    kind = case["kind"]
    if kind == "gelu":
        return {"bytes": 5 * case["n"], "flops": 0}
    if kind == "softmax":
        return {"bytes": 5 * case["rows"] * case["L"], "flops": 0}
    if kind == "layernorm":
        return {"bytes": case["rows"] * case["C"] * (case["bits"] // 8 + 2), "flops": 0}
    m = MODELS[case["model"]]
    H, F, L = m["H"], m["F"], case["L"]
    T = case["B"] * L
    pairs = T * L                                       # (query, key) pairs per head
    if kind == "packed":
        lens = _lengths(0, case["B"], L).astype(np.int64)
        T, pairs = int(lens.sum()), int((lens * lens).sum())
    weights = 4 * H * H + 2 * H * F
    layers = 1 if kind == "ops" else m["layers"]
    flops = layers * (2 * T * weights + 4 * pairs * H)
    nbytes = layers * (weights + 4 * (5 * H + F)) + 2 * T * H
    if kind == "ops":                                   # every operator's result is handed out
        nbytes += T * (3 * H + H + H + F + 2 * H)
    if kind in ("model", "packed"):
        nbytes += T * (4 + H) + 4 * case["B"] * (1 + LABELS)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case: dict):
    return "exact"                                      # integer arithmetic throughout: bytes and whole numbers
