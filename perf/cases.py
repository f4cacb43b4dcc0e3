"""What a user of this framework has it do, as cases that can be timed and compared.

Three kinds, told apart by ``case["kind"]``:

  layer   one denoising step of an attention layer (``Layer.step`` / ``Layer.step_quantile``), on a handle that has
          already run its first pass: the step alternates between two hidden states of which ``changed`` per cent of
          the rows differ, the others by N(0, 1e-3^2).  With ``first`` it is the first pass itself (reset, then a step).
  stack   the transformer stack: one block-wise decoding step over the generation window, or (``first``) the first
          forward pass over the whole sequence.
  scores  drift scores, reuse-rate quantile and compaction of many tokens at once (calibration, batch scoring).

Layer and stack sizes are the repository's benchmark configurations and generic ones between and around them.
"""
from __future__ import annotations

import math

import torch

from paper_2605_08134_b200 import dare
from paper_2605_08134_b200 import workloads as wl

MODES = {"dense": dare.MODE_DENSE, "kv": dare.MODE_KV, "o": dare.MODE_O, "both": dare.MODE_BOTH}
TAU = 0.1          # between the two modes of the drift scores: about 1e-6 for unchanged rows, about 1 for redrawn ones
NOISE = 1e-3


def _layer(name, dtype, d, hd, batch, seq, mode, changed, window=0, clustered=False, quantile=False, first=False):
    c = {"kind": "layer", "dtype": dtype, "d": d, "hd": hd, "batch": batch, "seq": seq, "window": window, "mode": mode,
         "changed": changed, "clustered": clustered, "quantile": quantile, "first": first}
    return {"name": name, **c} if name else c


def _stack(name, layers, d, ff, vocab, batch, prompt, gen, first):
    c = {"kind": "stack", "layers": layers, "d": d, "ff": ff, "vocab": vocab, "batch": batch, "prompt": prompt, "gen": gen,
         "first": first}
    return {"name": name, **c} if name else c


def _scores(name, rows, hd):
    c = {"kind": "scores", "rows": rows, "hd": hd}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest layer of the benchmark (configuration 1): single precision, latency and launches are what counts
        _layer("f32_d256_s128_both", "f32", 256, 64, 1, 128, "both", 20),
        # single precision at an ordinary width, as in a checking run of a small model
        _layer("f32_d1024_b2_s384_kv", "f32", 1024, 64, 2, 384, "kv", 20),
        # bf16 with 64-wide heads, the other common head width
        _layer("bf16_hd64_d2048_b2_s512_both", "bf16", 2048, 64, 2, 512, "both", 13),
        # configuration 2, the headline: an 8B-class layer, batch 1, 87 % of the tokens reused
        _layer("bf16_d4096_b1_s512_both", "bf16", 4096, 128, 1, 512, "both", 13),
        # ... and the same layer recomputed in full (a refresh step of the schedule)
        _layer("bf16_d4096_b1_s512_dense", "bf16", 4096, 128, 1, 512, "dense", 13),
        # semi-autoregressive decoding of the active block only: 32 rows a sequence against a frozen prefix, reuse rate
        # given as a quantile, ragged sizes
        _layer("bf16_d4096_b2_w32_both_quantile", "bf16", 4096, 128, 2, 1003, "both", 50, window=32, quantile=True),
        # configuration 3: batch 8, output reuse, changes clustered in the active block
        _layer("bf16_d4096_b8_s1024_o", "bf16", 4096, 128, 8, 1024, "o", 13, clustered=True),
        # configuration 5: long context
        _layer("bf16_d4096_b4_s4096_both", "bf16", 4096, 128, 4, 4096, "both", 15),
        # the first pass over a prompt (nothing cached), ragged
        _layer("bf16_d2048_b3_s1331_first", "bf16", 2048, 128, 3, 1331, "both", 0, first=True),
        # configuration 4: one decoding step of the whole 32-layer stack, 256 prompt + 256 generated tokens
        _stack("stack_32l_decode", 32, 4096, 12288, 126464, 1, 256, 256, False),
        # first pass of a batch through (a quarter of) that stack: all positions, hidden states out
        _stack("stack_8l_b2_first", 8, 4096, 12288, 126464, 2, 256, 256, True),
        # scoring, quantile and compaction of a million tokens
        _scores("scores_1m_hd128", 1 << 20, 128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "hd64", "f32", "stack", "scores"])
    changed = rng.choice([5, 13, 20, 30, 50, 70, 100])
    mode = rng.choice(["both", "both", "kv", "o", "dense"])
    quantile = mode != "dense" and rng.random() < 0.3
    if kind == "scores":
        return _scores("", _log(rng, 1 << 14, 1 << 20), rng.choice([64, 128]))
    if kind == "stack":
        d, batch = rng.choice([1024, 2048, 4096]), rng.randint(1, 4)
        prompt, gen = _log(rng, 32, 512), 32 * rng.randint(1, 8)
        layers = min(rng.randint(2, 8), 8192 // (batch * (prompt + gen)))
        return _stack("", layers, d, 3 * d, 256 * rng.randint(125, 494), batch, prompt, gen, rng.random() < 0.3)
    if kind == "f32":
        hd = rng.choice([32, 64, 128])
        d = 128 * rng.randint(1, 8)
        batch, seq = rng.randint(1, 4), _log(rng, 32, 400)
        window = rng.choice([0, 0, min(seq, 32)])
        return _layer("", "f32", d, hd, batch, seq, mode, changed, window, rng.random() < 0.3, quantile)
    if kind == "hd64":
        d = 256 * rng.randint(2, 8)
        batch, seq = rng.randint(1, 4), _log(rng, 48, 512)
        window = rng.choice([0, 0, min(seq, 32)])
        return _layer("", "bf16", d, 64, batch, seq, mode, changed, window, rng.random() < 0.3, quantile)
    d = 256 * rng.choice([4, 6, 8, 12, 16])
    batch = rng.randint(1, 8)
    seq = _log(rng, 64, min(4096, 16384 // batch))
    window = rng.choice([0, 0, min(seq, 32), min(seq, 32 * rng.randint(1, 8))])
    first = rng.random() < 0.2
    if first:
        return _layer("", "bf16", d, 128, batch, seq, "both", 0, 0, False, False, True)
    return _layer("", "bf16", d, 128, batch, seq, mode, changed, window, rng.random() < 0.3, quantile)


# ---------------------------------------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(g, shape, std=1.0, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=g)


def _rows(case):
    """Rows of each sequence that a step covers, and how many of them change."""
    act = case["window"] or case["seq"]
    return act, min(act, max(1, round(act * case["changed"] / 100)))


def _prepare_layer(case, seed):
    g = _generator(seed)
    d, hd, batch, seq = case["d"], case["hd"], case["batch"], case["seq"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    shape = wl.LayerShape("case", d, d // hd, hd, batch, seq, seq // 2, 5e5 if dt == torch.bfloat16 else 1e4,
                          wl.DTYPE_BF16 if dt == torch.bfloat16 else wl.DTYPE_F32)
    weights = {k: _normal(g, (d, d), 0.02, dt) for k in ("w_q", "w_k", "w_v", "w_o")}
    weights["rms_gain"] = torch.ones(d, device="cuda")
    layer = dare.Layer(shape, weights)
    x0 = _normal(g, (batch, seq, d), 1.0, torch.float32)
    if case["first"]:
        return {"case": case, "layer": layer, "x": x0.to(dt)}
    layer.step(x0.to(dt), dare.MODE_DENSE, TAU)                       # the first pass, over the whole sequence
    act, n = _rows(case)
    begin = seq - act
    xa = x0[:, begin:].contiguous()
    if case["clustered"]:                                             # a run at the start of the window's second half
        order = (act // 2 + torch.arange(act, device="cuda")) % act
        pick = order[:n].expand(batch, n)
    else:
        pick = torch.rand((batch, act), generator=g, device="cuda").argsort(1)[:, :n]
    changed = torch.zeros((batch, act), dtype=torch.bool, device="cuda").scatter_(1, pick, True)
    xb = torch.where(changed[:, :, None], _normal(g, xa.shape, 1.0, torch.float32),
                     xa + _normal(g, xa.shape, NOISE, torch.float32))
    return {"case": case, "layer": layer, "x": [xb.to(dt), xa.to(dt)], "turn": 0, "begin": begin,
            "reuse": batch * (act - n), "mode": MODES[case["mode"]]}


def _run_layer(s):
    layer, case = s["layer"], s["case"]
    if case["first"]:
        layer.reset()
        return layer.step(s["x"], MODES[case["mode"]], TAU)
    x = s["x"][s["turn"]]
    s["turn"] ^= 1
    if case["quantile"]:
        return layer.step_quantile(x, s["mode"], s["reuse"], pos_begin=s["begin"])
    return layer.step(x, s["mode"], TAU, pos_begin=s["begin"])


def _prepare_stack(case, seed):
    g = _generator(seed)
    d, f, vocab, batch = case["d"], case["ff"], case["vocab"], case["batch"]
    seq = case["prompt"] + case["gen"]
    lay = wl.LayerShape("case", d, d // 128, 128, batch, seq, case["prompt"], 5e5, wl.DTYPE_BF16)
    shape = wl.StackShape("case", case["layers"], lay, f, vocab, case["gen"])
    ones = torch.ones(d, device="cuda")
    # embeddings of unit size, residual branches scaled by depth, and a head that follows the embeddings (the row of
    # token j looks like the embedding of token j + 1): the model is decided about its tokens, as a trained one is
    emb = _normal(g, (vocab, d))
    w = {"emb": emb, "head": emb.roll(-1, 0).mul_(0.05), "final_gain": ones, "layers": []}
    deep = 0.02 / math.sqrt(2 * case["layers"])
    for _ in range(case["layers"]):
        w["layers"].append({"w_q": _normal(g, (d, d), 0.02), "w_k": _normal(g, (d, d), 0.02),
                            "w_v": _normal(g, (d, d), 0.02), "w_o": _normal(g, (d, d), deep), "rms_gain": ones,
                            "gain2": ones, "w_gate": _normal(g, (f, d), 0.02), "w_up": _normal(g, (f, d), 0.02),
                            "w_down": _normal(g, (d, f), deep)})
    stack = dare.Stack(shape, w, batch)
    tokens = torch.randint(0, vocab - 2, (batch, seq), generator=g, device="cuda", dtype=torch.int32)
    taus = [TAU] * case["layers"]
    if case["first"]:
        tokens[:, case["prompt"]:] = shape.mask_id
        return {"case": case, "stack": stack, "tokens": tokens, "taus": taus}
    # two consecutive states of a generation: blocks before the active one are decoded, half of the active one is,
    # and the second state has one token more than the first
    active = case["gen"] // 32 // 2
    lo = case["prompt"] + 32 * active
    now = tokens.clone()
    now[:, lo + 32:] = shape.mask_id
    masked = torch.rand((batch, 32), generator=g, device="cuda").argsort(1)[:, :16] + lo
    now.scatter_(1, masked, shape.mask_id)
    later = now.clone()
    later.scatter_(1, masked[:, :1], tokens.gather(1, masked[:, :1].long()))
    out = (torch.empty(batch, dtype=torch.int32, device="cuda"), torch.empty(batch, dtype=torch.int32, device="cuda"),
           torch.empty(batch, dtype=torch.float32, device="cuda"))
    stack.forward(now, seq, 0, dare.MODE_DENSE, taus)
    return {"case": case, "stack": stack, "states": [later, now], "turn": 0, "tokens": now.clone(), "active": active,
            "taus": taus, "out": out}


def _run_stack(s):
    stack, case = s["stack"], s["case"]
    if case["first"]:
        stack.reset()
        return stack.forward(s["tokens"], case["prompt"] + case["gen"], 0, dare.MODE_BOTH, s["taus"])
    s["tokens"].copy_(s["states"][s["turn"]])          # (the step writes its token; the next pass is another state)
    s["turn"] ^= 1
    pos, tok, prob = stack.decode_step_enqueue(s["tokens"], case["prompt"], s["active"], False, dare.MODE_BOTH, s["taus"],
                                               out=s["out"])
    return {"pos": pos, "tok": tok, "prob": prob, "tokens": s["tokens"]}


def _prepare_scores(case, seed):
    g = _generator(seed)
    n, hd = case["rows"], case["hd"]
    q_prev = _normal(g, (n, hd), 1.28, torch.float32)
    changed = torch.rand((n, 1), generator=g, device="cuda") < 0.13
    q_now = torch.where(changed, _normal(g, (n, hd), 1.28, torch.float32), q_prev + _normal(g, (n, hd), NOISE, torch.float32))
    scratch = dare.dare_select_compact_scratch_bytes(n)
    return {"q_now": q_now, "q_prev": q_prev, "n": n, "hd": hd, "scratch_bytes": scratch, "k": int(0.93 * n),
            "scores": torch.empty(n, device="cuda"), "tau": torch.empty(1, device="cuda"),
            "idx": torch.full((n,), -1, dtype=torch.int32, device="cuda"),
            "count": torch.zeros(1, dtype=torch.int32, device="cuda"),
            "scratch": torch.empty(scratch, dtype=torch.uint8, device="cuda")}


def _check(status, what):
    if status != dare.OK:
        raise dare.DareError(status, what)


def _run_scores(s):
    st = torch.cuda.current_stream().cuda_stream
    _check(dare.dare_drift_scores(s["q_now"].data_ptr(), s["q_prev"].data_ptr(), s["n"], s["hd"], s["scores"].data_ptr(), st),
           "dare_drift_scores")
    _check(dare.dare_score_kth(s["scores"].data_ptr(), s["n"], s["k"], s["tau"].data_ptr(), st), "dare_score_kth")
    _check(dare.dare_select_compact(s["scores"].data_ptr(), s["n"], TAU, s["idx"].data_ptr(), s["count"].data_ptr(),
                                    s["scratch"].data_ptr(), s["scratch_bytes"], st), "dare_select_compact")
    return {"scores": s["scores"], "tau": s["tau"], "idx": s["idx"], "count": s["count"]}


_PREPARE = {"layer": _prepare_layer, "stack": _prepare_stack, "scores": _prepare_scores}


def prepare(case, seed):
    s = _PREPARE[case["kind"]](case, seed)
    s["kind"] = case["kind"]
    torch.cuda.synchronize()
    return s


def run(state):
    if state["kind"] == "layer":
        return _run_layer(state)
    return _run_stack(state) if state["kind"] == "stack" else _run_scores(state)


# ---------------------------------------------------------------------------------------------------------------
def _layer_work(e, d, hd, batch, kv_len, act, n, kv, o):
    """One step over `act` rows a sequence of which `n` are refreshed: kv / o tell which of the two reuse rules apply.
    Every weight, hidden state, key, value and reused output once; only refreshed rows are projected and attended."""
    t, r = batch * act, batch * n
    rk, ro = (r if kv else t), (r if o else t)
    size = e * (4 * d * d + 2 * t * d + 2 * batch * kv_len * d + 2 * rk * d + (t - ro) * d) + 8 * t * hd
    flops = 2 * t * d * d + 4 * rk * d * d + 4 * ro * kv_len * d + 2 * ro * d * d
    return size, flops


def work(case):
    if case["kind"] == "scores":
        n, hd = case["rows"], case["hd"]
        return {"bytes": 8 * n * hd + 12 * n + 0.13 * 4 * n, "flops": 6 * n * hd}
    if case["kind"] == "layer":
        e = 2 if case["dtype"] == "bf16" else 4
        act, n = _rows(case)
        mode = MODES[case["mode"]]
        if case["first"]:
            act, n, mode = case["seq"], case["seq"], 0
        size, flops = _layer_work(e, case["d"], case["hd"], case["batch"], case["seq"], act, n, mode & 1, mode & 2)
        return {"bytes": size, "flops": flops}
    d, f, batch = case["d"], case["ff"], case["batch"]
    seq = case["prompt"] + case["gen"]
    act = seq if case["first"] else case["gen"]
    n = act if case["first"] else 1
    size, flops = _layer_work(2, d, 128, batch, seq, act, n, not case["first"], not case["first"])
    t = batch * act
    size += 2 * 3 * d * f
    flops += 6 * t * d * f
    size, flops = case["layers"] * size, case["layers"] * flops
    if not case["first"]:
        size += 2 * case["vocab"] * d
        flops += 2 * 16 * batch * case["vocab"] * d
    return {"bytes": size, "flops": flops}


def tolerance(case):
    if case["kind"] == "scores":
        return {"rel": 1e-5, "max": 1e-5}
    if case["kind"] == "stack":
        # bf16 residual stream rounded twice a layer; the chosen positions and tokens are the same
        return {"rel": 2e-2, "max": 0.2}
    # bf16: 8-bit mantissas of x_norm, Q, K, V and the attention output; single precision: sums of up to 1024 products
    return {"rel": 1e-2, "max": 0.1} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 1e-4}
