"""Performance cases: what a user of this library has it do, through its public calls.

A program that decodes loads a model once, keeps one session for the batch shape it serves, and for every new batch of
sources calls ``bpd_encode`` and a decode call that returns the ids to the host.  That is one pass here: host ids in,
host ids out.  Two further kinds stand for a scheduler that steps a session itself (``bpd_iteration``) and for programs
that embed the single operators.

Model shapes are those of ``bpd_inputs/workloads.py`` (the paper's translation and super-resolution settings).  The
weights are random as there, with one addition: the embeddings, the output projection and the proposal heads carry a
planted next-token rule, so that the model predicts with the confidence of a trained one and its proposals hold for
runs of about five tokens.  Without it every next token of a random model is a near tie and ids would depend on the
order of a sum.  The rule: the vocabulary is cut into bands of ``M`` ids; a source is drawn from one band (a subject, a
brightness) and the output stays in that band; inside a band the ids form one cycle made of shuffled runs of
consecutive ids.  Head i predicts i tokens ahead as if the current run went on, which is right until the run ends.
"""
import math
from dataclasses import replace

import numpy as np
import torch

import paper_1811_03115_b200 as bpd
from bpd_inputs import WORKLOADS
from bpd_inputs.blob import DTYPE_F32, HEAD_BLOCKDIAG, tensor_specs, write_blob

RUN = 5.0     # mean length of a run of consecutive ids: the mean accepted block size the repository's benchmark uses
SIGNAL = 4.0  # strength of the planted part of the decoder's stream, against about 1.5 from everything else in it

# name -> (configuration, std of the random draws)
MODELS = {
    "tiny": (WORKLOADS["C1"].cfg, WORKLOADS["C1"].sigma),              # fp32, CUDA-core kernels
    "base": (WORKLOADS["C2"].cfg, WORKLOADS["C2"].sigma),              # translation, base size, 4 heads
    "big": (WORKLOADS["C3"].cfg, WORKLOADS["C3"].sigma),               # translation, big size, 8 heads
    "big10": (WORKLOADS["C4"].cfg, WORKLOADS["C4"].sigma),             # the same with 10 heads
    "big_blockdiag": (replace(WORKLOADS["C3"].cfg, head_layout=HEAD_BLOCKDIAG), WORKLOADS["C3"].sigma),
    "image": (WORKLOADS["C5"].cfg, WORKLOADS["C5"].sigma),             # super-resolution, intensities 0..255
    "image_local": (WORKLOADS["C5L"].cfg, WORKLOADS["C5L"].sigma),     # the same with 1D local self-attention
}


def listed():
    def decode(name, model, batch, src_lo, src_hi, tgt, k, how="blockwise", accept=0):
        return {"name": name, "kind": "decode", "model": model, "batch": batch, "src_lo": src_lo, "src_hi": src_hi,
                "tgt": tgt, "k": k, "how": how, "accept": accept}
    return [
        # the smallest decode: a toy-sized fp32 model, nothing but launches and latency
        decode("tiny_fp32", "tiny", 1, 16, 16, 32, 4),
        # one sentence at a time, interactive use: base and big translation models
        decode("base_sentence", "base", 1, 32, 32, 64, 4),
        decode("big_sentence", "big", 1, 40, 40, 128, 8),
        # the same model without proposals: what users run for comparison and with k = 1 models
        decode("big_greedy", "big", 1, 40, 40, 128, 1, how="greedy"),
        # a few ragged sentences in one call, odd counts: more rows than the one-sentence paths take
        decode("base_ragged5", "base", 5, 7, 61, 51, 4),
        # top-2 acceptance with independent head layers, three sentences
        decode("big_blockdiag_top2", "big_blockdiag", 3, 9, 45, 77, 8, accept=bpd.BPD_ACCEPT_TOPN(2)),
        # offline translation: full batches
        decode("big_batch32", "big10", 32, 10, 80, 128, 10),
        # super-resolution of an 8x8 image to 32x32, exact acceptance; and with local attention, where intensities
        # within 2 of the base model's are taken
        decode("image_3072", "image", 1, 192, 192, 3072, 10),
        decode("image_local_dist2", "image_local", 1, 192, 192, 3072, 10, accept=bpd.BPD_ACCEPT_DISTANCE(2)),
        # a scheduler that looks at every iteration: encode, then ten single iterations read back one by one
        {"name": "base_stepwise", "kind": "step", "model": "base", "batch": 4, "src_lo": 20, "src_hi": 50, "steps": 10, "k": 4},
        # single operators in a program of the user's own: next-token top-1 for a batch of states, and a projection
        {"name": "top1_operator", "kind": "top1", "rows": 64, "d": 1024, "vocab": 32768, "dtype": "bf16"},
        {"name": "linear_operator", "kind": "linear", "rows": 37, "d": 1024, "out": 4096, "dtype": "bf16"},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["sentence", "sentence", "batch", "batch", "batch", "greedy", "image", "step", "top1", "linear"])
    if kind == "top1":
        return {"kind": "top1", "rows": _log_int(rng, 1, 256), "d": 8 * rng.randint(16, 128), "vocab": _log_int(rng, 250, 50000),
                "dtype": rng.choice(["bf16", "bf16", "fp32"])}
    if kind == "linear":
        return {"kind": "linear", "rows": _log_int(rng, 1, 300), "d": 8 * rng.randint(32, 256), "out": _log_int(rng, 256, 8192),
                "dtype": rng.choice(["bf16", "bf16", "fp32"])}
    if kind == "image":
        side = rng.randint(4, 8)
        tgt = 48 * side * side
        return {"kind": "decode", "model": rng.choice(["image", "image_local"]), "batch": 1, "src_lo": 3 * side * side,
                "src_hi": 3 * side * side, "tgt": tgt - rng.randint(0, tgt // 2), "k": rng.randint(4, 10), "how": "blockwise",
                "accept": rng.choice([0, bpd.BPD_ACCEPT_DISTANCE(2)])}
    model = rng.choice(["tiny", "base", "base", "big", "big", "big10", "big_blockdiag"])
    kmax = MODELS[model][0].k_model
    src_hi = _log_int(rng, 10, 96)
    src_lo = max(1, src_hi // rng.randint(1, 6))
    batch = {"sentence": 1, "greedy": _log_int(rng, 1, 16), "batch": _log_int(rng, 2, 32), "step": _log_int(rng, 1, 16)}[kind]
    if kind == "step":
        return {"kind": "step", "model": model, "batch": batch, "src_lo": src_lo, "src_hi": src_hi, "steps": rng.randint(5, 20),
                "k": rng.randint(2, kmax)}
    if kind == "greedy":
        return {"kind": "decode", "model": model, "batch": batch, "src_lo": src_lo, "src_hi": src_hi, "tgt": _log_int(rng, 12, 96),
                "k": 1, "how": "greedy", "accept": 0}
    return {"kind": "decode", "model": model, "batch": batch, "src_lo": src_lo, "src_hi": src_hi, "tgt": _log_int(rng, 16, 128),
            "k": rng.randint(max(2, kmax // 2), kmax), "how": "blockwise", "accept": rng.choice([0, 0, 0, bpd.BPD_ACCEPT_TOPN(2)])}


# ---------------------------------------------------------------------- models
def _bands(cfg):
    """(bands, ids per band): no more ids than the width of the model tells apart with ease."""
    return (64, cfg.vocab // 64) if cfg.vocab >= 8192 else (8, min(cfg.vocab // 8, cfg.d_model // 4))


def _cycles(cfg):
    """order[g]: the cycle of band g's classes, runs of consecutive classes (mean length RUN) in a shuffled order."""
    bands, m = _bands(cfg)
    rng = np.random.default_rng(7)
    order = np.empty((bands, m), np.int64)
    for g in range(bands):
        cuts = np.flatnonzero(rng.random(m - 1) < 1.0 / RUN) + 1
        runs = np.split(np.arange(m), cuts)
        order[g] = np.concatenate([runs[i] for i in rng.permutation(len(runs))])
    return order


def make_blob(name, device="cuda"):
    """The weight container of a model: random draws plus the planted next-token rule."""
    cfg, sigma = MODELS[name]
    gen = torch.Generator(device=device)
    gen.manual_seed(11)
    d, fh, half = cfg.d_model, cfg.d_hidden, cfg.d_model // 2
    signal = SIGNAL * max(1.0, math.sqrt(512 / d))
    fill = {"gain": torch.ones, "shift": torch.zeros}
    t = {n: fill[kind](shape, device=device) if kind in fill else
         torch.randn(shape, generator=gen, device=device) * sigma for n, shape, kind in tensor_specs(cfg)}
    bands, m = _bands(cfg)
    order = torch.from_numpy(_cycles(cfg)).to(device)
    # a class is a point of a torus (the first half of the dimensions, pairs): one class on is one fixed rotation
    omega = torch.rand(half // 2, generator=gen, device=device) * (2 * math.pi)
    ang = torch.arange(m, device=device)[:, None] * omega[None, :]
    cls = torch.stack([torch.cos(ang), torch.sin(ang)], -1).reshape(m, half) * math.sqrt(2.0)
    band = torch.randn((bands, d), generator=gen, device=device)
    ids = torch.arange(bands * m, device=device)
    t["src_embed"][:bands * m] += band[ids // m] * (2 * signal / math.sqrt(d))
    t["tgt_embed"][:bands * m, :half] += cls[ids % m] * (signal / math.sqrt(d))
    # what the source's band becomes on its way through the decoder's cross-attention (values, then output projection)
    seen = torch.zeros((bands, d), device=device)
    for l in range(cfg.n_dec):
        t["dec.%d.cross.wo" % l][half:] *= 0.3 * signal / (sigma * sigma * d)
        seen += (band @ t["dec.%d.cross.wkv" % l][d:].T) @ t["dec.%d.cross.wo" % l].T
    seen = seen[:, half:] / seen[:, half:].square().mean(-1, keepdim=True).sqrt()
    # output row of class c in band g: the class before c in the band's cycle, and the band
    before = torch.empty_like(order)
    before.scatter_(1, order, order.roll(1, 1))
    t["out_proj"][:bands * m, :half] += cls[before.reshape(-1)] * (3 * sigma)
    t["out_proj"][:bands * m, half:] += seen[ids // m] * (3 * sigma)
    # head i carries its input over (max(x, 0) - max(-x, 0)) and turns it i - 1 classes on
    w1, b1 = t["head.w1"].view(cfg.k_model, fh, d), t["head.b1"].view(cfg.k_model, fh)
    eye = torch.eye(d, device=device)
    t["head.w2"] *= 0.5     # what a head adds at random stays below what it carries over
    for i in range(cfg.k_model):
        w1[i, :2 * d] = torch.cat([eye, -eye])
        b1[i, :2 * d] = 0
        turn = torch.zeros((d, d), device=device)
        c, s = torch.cos(i * omega), torch.sin(i * omega)
        even = torch.arange(0, half, 2, device=device)
        turn[even, even], turn[even, even + 1] = c - 1, -s
        turn[even + 1, even], turn[even + 1, even + 1] = s, c - 1
        w2 = t["head.w2"][i] if cfg.head_layout == HEAD_BLOCKDIAG else t["head.w2"][i * d:(i + 1) * d, i * fh:(i + 1) * fh]
        w2[:, :2 * d] = torch.cat([turn, -turn], 1)
    if cfg.dtype == DTYPE_F32:
        host = {n: v.cpu().numpy() for n, v in t.items()}
    else:
        host = {n: v.to(torch.bfloat16).view(torch.int16).cpu().numpy().view(np.uint16) for n, v in t.items()}
    return write_blob(cfg, host)


_models = {}     # name -> loaded model: a program loads its models once
_session = {}    # shape -> session: one at a time, kept over the sources that come in


def _model(name):
    if name not in _models:
        while len(_models) >= 3:
            _close_session()
            _models.pop(next(iter(_models))).close()
        _models[name] = bpd.Model(make_blob(name))
    return _models[name]


def _close_session():
    while _session:
        _session.popitem()[1].close()


def _session_for(shape):
    s = _session.get(shape)
    if s is None:
        _close_session()
        s = _session[shape] = bpd.Session(_model(shape[0]), shape[1], shape[2], shape[3])
    return s


# ---------------------------------------------------------------------- cases
def _shape(case):
    tgt = case["steps"] * case["k"] if case["kind"] == "step" else case["tgt"]
    return case["model"], case["batch"], case["src_hi"], tgt


def prepare(case, seed):
    if case["kind"] in ("top1", "linear"):
        _close_session()
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        n = case["vocab"] if case["kind"] == "top1" else case["out"]
        x = torch.randn((case["rows"], case["d"]), generator=gen, device="cuda").to(dtype)      # normalised states
        w = (torch.randn((n, case["d"]), generator=gen, device="cuda") * 0.02).to(dtype)
        bias = (torch.randn(n, generator=gen, device="cuda") * 0.02).to(dtype)
        return {"case": case, "x": x, "w": w, "bias": bias}
    bands, m = _bands(MODELS[case["model"]][0])
    rng = np.random.default_rng(seed)
    src = np.zeros((case["batch"], case["src_hi"]), np.int32)
    lens = rng.integers(case["src_lo"], case["src_hi"] + 1, case["batch"]).astype(np.int32)
    lens[rng.integers(case["batch"])] = case["src_hi"]
    for b, n in enumerate(lens):
        first = int(rng.integers(bands)) * m
        if case["model"].startswith("image"):       # a smooth image of one brightness, raster order, RGB interleaved
            side = int(round(math.sqrt(n / 3)))
            img = np.pad(rng.integers(0, m, (side, side, 3)), ((1, 1), (1, 1), (0, 0)), mode="edge")
            img = sum(img[i:i + side, j:j + side] for i in range(3) for j in range(3)) // 9
            src[b, :n] = first + img.reshape(-1)
        else:                                       # a sentence on one subject
            src[b, :n] = first + rng.integers(0, m, n)
    _session_for(_shape(case))
    return {"case": case, "src": src, "lens": lens}


def run(state):
    case = state["case"]
    if case["kind"] == "top1":
        return bpd.bpd_op_vocab_argmax(state["x"], state["w"], want_val=True)
    if case["kind"] == "linear":
        return bpd.bpd_op_linear(state["x"], state["w"], state["bias"], relu=True)
    s = _session_for(_shape(case))
    s.bpd_encode(state["src"], state["lens"])
    if case["kind"] == "step":
        steps = [s.bpd_iteration(case["k"], case["steps"] * case["k"]) for _ in range(case["steps"])]
        return {"accepted": np.stack([r["accepted"] for r in steps]), "next": np.stack([r["next_block"] for r in steps])}
    if case["how"] == "greedy":
        ids, lens, _ = s.bpd_decode_greedy(case["tgt"])
    else:
        ids, lens, _ = s.bpd_decode_blockwise(case["k"], case["tgt"], accept_mode=case["accept"])
    return {"ids": ids, "lens": lens}


def _iterations(case):
    """Model invocations of the slowest row after the first, for rows of random bands (exact acceptance; the other
    criteria take a little more per iteration)."""
    cfg = MODELS[case["model"]][0]
    if case["how"] == "greedy":
        return case["tgt"]
    order = _cycles(cfg)
    bands, m = order.shape
    need = []
    for g in range(bands):
        on = np.append(np.diff(order[g]) == 1, order[g][0] == order[g][-1] + 1)     # does the run go on after this place?
        at, done, n = int(np.flatnonzero(order[g] == 0)[0]), 0, 0
        while done < case["tgt"]:
            took = 1
            while took < case["k"] and on[(at + took - 1) % m]:
                took += 1
            at, done, n = (at + took) % m, done + took, n + 1
        need.append(n)
    return float(np.mean(np.random.default_rng(1).choice(need, (200, case["batch"])).max(1)))


def work(case):
    """Every decoder pass reads the decoder's, the heads' and the output projection's weights once (a pass needs the
    tokens of the one before, and the weights of the models that matter do not fit on the chip) and the cached keys and
    values; the encoder reads its weights once.  Heads beyond the first are needed at one position per row."""
    if case["kind"] in ("top1", "linear"):
        e = 2 if case["dtype"] == "bf16" else 4
        n = case["vocab"] if case["kind"] == "top1" else case["out"]
        out = 8 * case["rows"] if case["kind"] == "top1" else 4 * case["rows"] * n + e * n
        return {"bytes": e * case["d"] * (case["rows"] + n) + out, "flops": 2 * case["rows"] * n * case["d"]}
    cfg = MODELS[case["model"]][0]
    e, d, f, km, fh = cfg.elem_bytes, cfg.d_model, cfg.d_ff, cfg.k_model, cfg.d_hidden
    B, k = case["batch"], case["k"]
    S = (case["src_lo"] + case["src_hi"]) / 2
    if case["kind"] == "step":
        iters, tgt = case["steps"], case["steps"] * min(k, RUN)
    else:
        iters, tgt = _iterations(case), case["tgt"]
    enc = cfg.n_enc * (4 * d * d + 2 * d * f) + cfg.n_dec * 2 * d * d
    dec = cfg.n_dec * (6 * d * d + 2 * d * f)
    heads1 = k if cfg.head_layout == HEAD_BLOCKDIAG else km          # hidden slices a head reads
    w1, voc = heads1 * fh * d, cfg.vocab * d
    w2 = k * d * (fh if cfg.head_layout == HEAD_BLOCKDIAG else km * fh)
    one = d * (fh if cfg.head_layout == HEAD_BLOCKDIAG else km * fh)
    keys = min(tgt / 2, cfg.local_q / 2 + cfg.local_m) if cfg.local_q else tgt / 2
    kv = B * cfg.n_dec * (2 * d * e * keys + 2 * d * e * S)
    byt = e * enc + iters * (e * (dec + w1 + w2 + voc) + kv) + 4 * B * (case["src_hi"] + tgt)
    rows = B * k
    attn = rows * cfg.n_dec * 4 * d * (keys + S)
    per = 2 * rows * (dec + w1 + one + voc) + attn + (2 * B * (w2 + (k - 1) * voc) if k > 1 else 0)
    return {"bytes": byt, "flops": 2 * B * S * enc + 4 * B * S * S * d * cfg.n_enc + iters * per}


def tolerance(case):
    if case["kind"] == "linear":
        return {"rel": 1e-5}                    # products of the inputs summed in fp32
    if case["kind"] == "top1":
        return {"rel": 1e-5, "differ": 0.01}    # values as above; an index may differ where two entries tie
    return "exact"                              # ids: the planted rule keeps every choice far from a tie
