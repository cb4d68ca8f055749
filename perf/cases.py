"""Performance cases of the decoding library: what its users run, from one short command to a full batch.

A case is one call of a public entry point on one model:

  entry  "decode"  wind_decode_greedy on device buffers (the model served next to its encoder)
         "host"    wind_decode_greedy_host on pinned host buffers (the encoder runs elsewhere)
         "refill"  wind_decode_greedy_refill: a set of utterances on fewer batch rows (offline transcription)
         "beam"    wind_beam_search on one utterance
  model  one of the decoder shapes this repository is configured for (MODELS)
  n      utterances;  rows  batch rows they are decoded on ("refill");  lo, hi  their lengths in frames (uniform)
  W      window (1 is frame-by-frame greedy decoding);  beam  hypotheses kept ("beam", else 0)

The weights stand for a trained transducer: an encoder frame either carries a label or does not, the joint network answers
with that label or with the blank by a clear margin, and the prediction network remembers the last label, so that a label is
emitted once (`trained_like`).  With independent random weights every decision would be close to a tie and a frame would
emit several labels, which no trained model does.  The share of frames that carry a label is the one of the repository's
configurations (0.25 to 0.40).
"""
import math

import numpy as np
import torch

import paper_2505_13765_b200 as wind

# Decoder shapes of the repository's configurations: D encoder, E embedding, P prediction network (L layers), H joint,
# V labels; rate: share of the frames that carry a label; S: most symbols per frame.
MODELS = {
    "tiny": dict(D=64, E=64, P=64, L=1, H=64, V=32, act=0, rate=0.30, S=5),
    "large": dict(D=512, E=640, P=640, L=1, H=640, V=1024, act=0, rate=0.35, S=10),
    "xl": dict(D=1024, E=640, P=640, L=2, H=640, V=1024, act=0, rate=0.25, S=10),
    "bigvocab": dict(D=1024, E=1024, P=1024, L=1, H=1024, V=8192, act=1, rate=0.40, S=10),
}


def case(name, entry, model, dtype, n, lo, hi, W, rows=0, beam=0):
    c = dict(entry=entry, model=model, dtype=dtype, n=n, lo=lo, hi=hi, W=W, rows=rows, beam=beam)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest model and utterance (8 s), in fp32: fixed costs and launches
        case("tiny_f32", "decode", "tiny", "f32", 1, 100, 100, 4),
        # an fp32 checkpoint of the large model, a handful of short utterances
        case("large_f32_b4", "decode", "large", "f32", 4, 60, 203, 8),
        # one 100 s recording: latency of a single stream
        case("large_b1", "decode", "large", "bf16", 1, 1250, 1250, 8),
        # a small batch of voice commands, 3 to 24 s, odd sizes
        case("large_b7_short", "decode", "large", "bf16", 7, 37, 301, 5),
        # frame-by-frame greedy decoding (no window), the baseline every user compares with
        case("large_b32_w1", "decode", "large", "bf16", 32, 125, 1000, 1),
        # the full batch: 128 utterances of 10 to 200 s
        case("large_b128", "decode", "large", "bf16", 128, 125, 2500, 8),
        # encoder outputs arrive in host memory: copies in, transcripts out
        case("large_host_b24", "host", "large", "bf16", 24, 100, 900, 8),
        # offline transcription: 300 utterances on 64 rows
        case("large_refill_300", "refill", "large", "bf16", 300, 50, 800, 8, rows=64),
        # the two-layer model on a small batch, and its full batch of long utterances
        case("xl_b6", "decode", "xl", "bf16", 6, 90, 610, 4),
        case("xl_b64", "decode", "xl", "bf16", 64, 500, 5000, 8),
        # the large vocabulary with its wide window
        case("bigvocab_b32", "decode", "bigvocab", "bf16", 32, 250, 3000, 16),
        # beam search over a 20 s utterance
        case("large_beam4", "beam", "large", "bf16", 1, 250, 250, 8, beam=4),
    ]


def draw(rng):
    """One more case of the listed kinds; sizes over their whole range, evenly in their logarithm."""
    def size(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    def lengths(lo, hi):
        top = size(lo, hi)
        return max(1, int(top * rng.uniform(0.05, 1.0))), top

    window = rng.choice([1, 2, 3, 4, 5, 8, 8, 8, 11, 16])
    kind = rng.choice(["tiny", "f32", "large", "large", "large", "large", "host", "refill", "xl", "xl", "bigvocab", "beam"])
    if kind == "tiny":
        lo, hi = lengths(40, 600)
        return case(None, "decode", "tiny", "f32", size(1, 16), lo, hi, window)
    if kind == "f32":
        lo, hi = lengths(40, 300)
        return case(None, "decode", "large", "f32", size(1, 16), lo, hi, window)
    if kind == "host":
        lo, hi = lengths(60, 1250)
        return case(None, "host", "large", "bf16", size(1, 64), lo, hi, window)
    if kind == "refill":
        rows = size(4, 128)
        lo, hi = lengths(60, 800)
        return case(None, "refill", "large", "bf16", size(rows + 1, 400), lo, hi, window, rows=rows)
    if kind == "beam":
        t = size(40, 300)
        return case(None, "beam", "large", "bf16", 1, t, t, rng.choice([1, 4, 8, 16]), beam=rng.choice([2, 3, 4]))
    if kind == "xl":
        lo, hi = lengths(100, 3000)
        return case(None, "decode", "xl", "bf16", size(1, 64), lo, hi, window)
    if kind == "bigvocab":
        lo, hi = lengths(100, 1500)
        return case(None, "decode", "bigvocab", "bf16", size(1, 32), lo, hi, window)
    lo, hi = lengths(50, 2500)
    return case(None, "decode", "large", "bf16", size(1, 128), lo, hi, window)


# ---------------------------------------------------------------------------------------------------------------------
# a model that is as sure of its labels as a trained one
# ---------------------------------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _orthonormal(g, rows, cols):
    return torch.linalg.qr(_normal(g, rows, cols))[0]


def trained_like(name, dtype):
    """Weights (numpy, fp32) and the frame direction of every label [V, D].

    Label k has a code v_k; the frame direction, the embedding and (through the LSTM's cell input) the hidden state after
    label k are images of it, W_pred maps that hidden state to minus the encoder projection of label k's frame, and row k
    of W_out is the encoder projection of label k's frame.  So a frame that carries label k scores k high unless k was the
    label before it, and everything else scores below the blank's bias.  The other gates are random with open input and
    output gates and a mostly closed forget gate.
    """
    m = MODELS[name]
    D, E, P, L, H, V = (m[k] for k in "DEPLHV")
    g = _gen(20250513 + len(name) * 1000 + V)
    act = torch.relu if m["act"] == 0 else torch.tanh
    d = min(D, E, P, H)
    code = _normal(g, V, d) if V > d else _orthonormal(g, d, V).T * math.sqrt(d)
    frames = code @ _orthonormal(g, D, d).T * math.sqrt(D / d)
    emb = torch.zeros(V + 1, E, device="cuda", dtype=torch.float64)
    s_e = _orthonormal(g, E, d)
    emb[:V] = code @ s_e.T
    w_ih, w_hh, b_ih, b_hh = [], [], [], []
    h = emb[:V]
    for l in range(L):
        fan = E if l == 0 else P
        wi = _normal(g, 4 * P, fan) * (0.3 * fan ** -0.5)
        wh = _normal(g, 4 * P, P) * (0.3 * P ** -0.5)
        wi[2 * P: 3 * P] = 0.7 * _orthonormal(g, P, d) @ s_e.T if l == 0 else 1.5 * _orthonormal(g, P, P)
        bi = torch.zeros(4 * P, device="cuda", dtype=torch.float64)
        bi[:P], bi[P: 2 * P], bi[3 * P:] = 3.0, -3.0, 3.0
        gates = (h @ wi.T + bi).split(P, dim=1)
        h = torch.sigmoid(gates[3]) * torch.tanh(torch.sigmoid(gates[0]) * torch.tanh(gates[2]))
        w_ih.append(wi), w_hh.append(wh), b_ih.append(bi), b_hh.append(torch.zeros_like(bi))
    w_enc = _orthonormal(g, H, D) * math.sqrt(H / D) if H >= D else _orthonormal(g, D, H).T
    x = frames @ w_enc.T                                         # [V, H] what the joint sees of label k's frame
    ridge = 1e-3 * h.square().sum(0).mean() * torch.eye(P, device="cuda", dtype=torch.float64)
    w_pred = -torch.linalg.solve(h.T @ h + ridge, h.T @ x).T     # hidden state after label k -> minus that
    other = x.roll(1, 0) + h @ w_pred.T                          # frame of another label after label k
    signal = (act(other) * x.roll(1, 0)).sum(1).mean()
    w_out = torch.zeros(V + 1, H, device="cuda", dtype=torch.float64)
    w_out[:V] = x * (12.0 / signal)
    w_out[V] = _normal(g, H) * (0.1 * H ** -0.5)
    b_out = torch.zeros(V + 1, device="cuda", dtype=torch.float64)
    b_out[V] = 6.5
    zero = torch.zeros(H)

    def host(t):
        return t.to(torch.float32).cpu().numpy()

    weights = dict(D=D, E=E, P=P, L=L, H=H, V=V, blank_id=V, act=m["act"], dtype=dtype, emb=host(emb),
                   w_ih=[host(t) for t in w_ih], w_hh=[host(t) for t in w_hh], b_ih=[host(t) for t in b_ih],
                   b_hh=[host(t) for t in b_hh], w_enc=host(w_enc), b_enc=host(zero), w_pred=host(w_pred), b_pred=host(zero),
                   w_out=host(w_out), b_out=host(b_out))
    return weights, frames.to(torch.float32)


_models = {}


def loaded(name, dtype):
    """The model a program keeps: (WindModel, frame directions)."""
    if (name, dtype) not in _models:
        weights, frames = trained_like(name, dtype)
        _models[name, dtype] = wind.WindModel(weights), frames
    return _models[name, dtype]


def utterances(c, frames, dtype, seed):
    """Encoder outputs [n, hi, D] with lengths in [lo, hi]: a frame carries a label with the model's rate (never the label
    carried before it), plus noise; the others are weaker noise; padding is zero."""
    m = MODELS[c["model"]]
    n, T, D, V = c["n"], c["hi"], m["D"], m["V"]
    g = _gen(seed)
    lens = torch.randint(c["lo"], c["hi"] + 1, (n,), generator=g, device="cuda", dtype=torch.int32)
    emits = torch.rand(n, T, generator=g, device="cuda") < m["rate"]
    steps = torch.randint(1, V, (n, T), generator=g, device="cuda")
    label = torch.cumsum(emits * steps, 1) % V
    enc = torch.empty(n, T, D, dtype=dtype, device="cuda")
    for b in range(n):
        f = torch.randn(T, D, generator=g, device="cuda")
        f = torch.where(emits[b, :, None], frames[label[b]] + 0.2 * f, 0.5 * f)
        f.masked_fill_((torch.arange(T, device="cuda") >= lens[b])[:, None], 0.0)
        enc[b] = f
    return enc, lens


def prepare(case, seed):
    c = dict(case)
    m = MODELS[c["model"]]
    model, frames = loaded(c["model"], c["dtype"])
    enc, lens = utterances(c, frames, model.torch_dtype, seed)
    n, T, W = c["n"], c["hi"], c["W"]
    s = dict(c=c, model=model, enc=enc, lens=lens, S=m["S"])
    if c["entry"] == "beam":
        s["enc"] = enc[0].float().cpu().numpy()
        return s
    max_out = 2 * T + 16
    out = dict(tokens=torch.full((n, max_out), -1, dtype=torch.int32, device="cuda"),
               frames=torch.full((n, max_out), -1, dtype=torch.int32, device="cuda"),
               lengths=torch.zeros(n, dtype=torch.int32, device="cuda"))
    if c["entry"] == "refill":
        need = wind.binding.wind_refill_workspace_bytes(model, n, T, c["rows"], W)
        s["workspace"] = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
    elif c["entry"] == "host":
        s["workspace"] = wind.alloc_workspace(model, n, T, W, host_staging_max_out=max_out)
        s["enc"], s["lens"] = enc.cpu().pin_memory(), lens.cpu().pin_memory()
        out = {k: v.cpu().pin_memory() for k, v in out.items()}
    else:
        s["workspace"] = wind.alloc_workspace(model, n, T, W)
    s["out"] = out
    return s


def run(state):
    s, c = state, state["c"]
    if c["entry"] == "beam":
        hyps, steps, _ = wind.binding.wind_beam_search(s["model"], s["enc"], c["W"], c["beam"], s["S"], max_hyps=c["beam"])
        out = dict(tokens=np.full((c["beam"], c["hi"] * s["S"]), -1, np.int32), lengths=np.zeros(c["beam"], np.int32),
                   scores=np.zeros(c["beam"]))
        out["frames"] = out["tokens"].copy()
        for k, (tokens, frames, score) in enumerate(hyps):
            out["tokens"][k, :len(tokens)], out["frames"][k, :len(frames)] = tokens, frames
            out["lengths"][k], out["scores"][k] = len(tokens), score
        return out
    o = s["out"]
    if c["entry"] == "refill":
        wind.wind_decode_greedy_refill(s["model"], s["enc"], s["lens"], c["rows"], c["W"], s["S"], o["tokens"], o["frames"],
                                       o["lengths"], s["workspace"])
    elif c["entry"] == "host":
        wind.wind_decode_greedy_host(s["model"], s["enc"], s["lens"], c["W"], s["S"], o["tokens"], o["frames"], o["lengths"],
                                     s["workspace"])
        # entries behind a transcript's end are unspecified here: a user reads up to it
        behind = torch.arange(o["tokens"].shape[1])[None, :] >= o["lengths"][:, None]
        return dict(lengths=o["lengths"], tokens=o["tokens"].masked_fill(behind, -1), frames=o["frames"].masked_fill(behind, -1))
    else:
        wind.wind_decode_greedy(s["model"], s["enc"], s["lens"], c["W"], s["S"], o["tokens"], o["frames"], o["lengths"],
                                s["workspace"])
    return o


def work(case):
    """Every valid frame and every weight read once, every token and its frame written once; the projection of every frame,
    one decoder update per token, the joint once per frame and once more on the frame of every token (per hypothesis for
    beam search), the embedding's input term once per token or once per label, whichever is less."""
    m = MODELS[case["model"]]
    D, E, P, L, H, V = (m[k] for k in "DEPLHV")
    es = 2 if case["dtype"] == "bf16" else 4
    valid = case["n"] * (case["lo"] + case["hi"]) / 2
    hyps = max(1, case["beam"])
    tokens = m["rate"] * valid * hyps
    weights = (V + 1) * E + 4 * P * (E + P) + (L - 1) * 8 * P * P + H * (D + P) + (V + 1) * H
    update = 8 * P * P + (L - 1) * 16 * P * P + 2 * P * H
    flops = 2 * valid * D * H + tokens * update + min(tokens, V + 1) * 8 * P * E + 2 * H * (V + 1) * (valid * hyps + tokens)
    return {"bytes": es * (valid * D + weights) + 8 * tokens + 4 * case["n"], "flops": flops}


def tolerance(case):
    """Transcripts are whole numbers and the margins of the decisions are far above rounding: they stay the same.  A beam
    score is a sum of log-probabilities from bf16 activations."""
    return {"rel": 1e-2, "differ": 0.0} if case["entry"] == "beam" else "exact"
