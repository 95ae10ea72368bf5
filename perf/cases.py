"""What a program that uses this library has it do, as cases that can be timed and compared.

A case is a dict of plain values.  Its "kind" is the public entry point it goes through:

  fused       cmsd.FusedCall / cmsd.confidence_verify: confidence and verification in one pass
  confidence  cmsd.confidence: the drafter's signals and the next draft length
  verify      cmsd.verify: verification with signals the caller already has
  lmhead      cmsd.lmhead_confidence: the drafter's LM head with the signals
  loop        decode_sim.DecodeSim: the decode loop, replayed from a CUDA graph

Inputs are made on the GPU from the seed alone, after the recipes of
paper_2508_15371_gb300/workloads.py.
"""
import math

import torch

from paper_2508_15371_gb300 import cmsd, decode_sim

LAM = (1.0 / 3.0, 1.0 / 3.0, 1.0 / 3.0)     # the library's default ensemble weights and sigmoid sharpness
BETA_SIG = 1.0
MAX_BYTES = 2 * 256 * 16 * 152064 * 2        # logit bytes of the largest listed case
MEAN_WINDOW = 4.9                            # drafted positions per sequence and iteration of the listed loop


def _fused(name, B, K, V, dtype, rule, recipe, signals, ragged=False, bonus=False, masked=0.0):
    return dict(name=name, kind="fused", B=B, K=K, V=V, dtype=dtype, rule=rule, recipe=recipe, signals=signals,
                ragged=ragged, bonus=bonus, masked=masked)


def listed():
    return [
        # one interactive sequence, a short window: latency of a call in a decode loop that wants decisions only
        _fused("one_sequence", 1, 4, 32000, "f32", "sampled", "spike", False),
        # a small translation batch under the paper's own rule, with the signals logged, 30 % of the vocabulary masked
        _fused("small_batch_paper", 8, 8, 32128, "bf16", "paper", "spread", True, masked=0.3),
        # the serving batch of the benchmark: decisions only, residual draws
        _fused("serve_sampled", 64, 8, 128256, "bf16", "sampled", "zipf", False),
        # the same batch under the paper's rule, signals logged
        _fused("serve_paper", 64, 8, 128256, "bf16", "paper", "zipf", True),
        # the largest batch and window: offline generation
        _fused("large_sampled", 256, 16, 152064, "bf16", "sampled", "mixture", True),
        # speculative sampling with the verifier's extra row: a token more when all drafts are accepted
        _fused("bonus_sampled", 32, 8, 128256, "bf16", "sampled", "mixture", True, bonus=True),
        # verification apart from the drafter's pass: ragged windows, odd vocabulary (rows off 16-byte boundaries)
        dict(name="verify_ragged_odd", kind="verify", B=48, K=12, V=32001, dtype="bf16", rule="sampled",
             recipe="spread", ragged=True),
        # the drafter's own step: one new position per sequence, its signals
        dict(name="draft_step", kind="confidence", B=64, K=1, V=128256, dtype="bf16", recipe="mixture",
             ragged=False, masked=0.0),
        # the drafter's LM head: a small drafter, the serving batch, and a batch of several positions per sequence
        dict(name="lmhead_small", kind="lmhead", R=16, d=1024, V=32000, logits=False),
        dict(name="lmhead_serve", kind="lmhead", R=64, d=2048, V=128256, logits=False),
        dict(name="lmhead_wide", kind="lmhead", R=256, d=2048, V=128256, logits=False),
        # the device-resident decode loop: generation and pass of 64 iterations, adaptive windows
        dict(name="decode_loop", kind="loop", B=32, K=16, V=32000, iterations=64, rule="sampled"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng, lo=8000, hi=152064):
    v = _log(rng, lo, hi)
    how = rng.randrange(3)
    return max(lo, v - v % 128) if how == 0 else (v | 1) if how == 1 else v


def draw(rng):
    kind = rng.choice(["fused", "fused", "fused", "fused", "verify", "confidence", "lmhead", "lmhead", "loop"])
    if kind == "lmhead":
        return dict(kind=kind, R=_log(rng, 4, 256), d=64 * _log(rng, 8, 48), V=min(128256, _vocab(rng)),
                    logits=rng.random() < 0.2)
    if kind == "loop":
        return dict(kind=kind, B=_log(rng, 4, 32), K=rng.randint(4, 16), V=min(32000, _vocab(rng, 4000, 32000)),
                    iterations=rng.choice([16, 32, 64]), rule=rng.choice(["sampled", "paper"]))
    dtype = rng.choice(["bf16", "bf16", "f32"])
    es = 4 if dtype == "f32" else 2
    V = _vocab(rng)
    K = rng.choice([1, 2, 4, 8, 16, rng.randint(1, 24)])
    B = max(1, min(_log(rng, 1, 256), MAX_BYTES // (2 * (K + 1) * V * es)))
    c = dict(kind=kind, B=B, K=K, V=V, dtype=dtype, ragged=rng.random() < 0.4,
             recipe=rng.choice(["spike", "spread", "zipf", "mixture"]))
    if kind != "confidence":
        c["rule"] = rng.choice(["sampled", "sampled", "paper"])
    if kind != "verify":
        c["masked"] = rng.choice([0.0, 0.0, 0.0, 0.3])
    if kind == "fused":
        c["signals"] = rng.random() < 0.5
        c["bonus"] = (V * es) % 16 == 0 and rng.random() < 0.4
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _rows(c, seed):
    """Drafter logits [B, K, V], target logits [B, K (+1), V], drafted tokens [B, K] and windows [B] (or None)."""
    B, K, V = c["B"], c["K"], c["V"]
    Kt = K + 1 if c.get("bonus") else K
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
    draft = torch.empty((B, K, V), dtype=dt, device="cuda")
    target = torch.empty((B, Kt, V), dtype=dt, device="cuda")
    tokens = torch.empty((B, K), dtype=torch.int32, device="cuda")
    recipe = c["recipe"]
    sig = {"spike": 0.5, "spread": 1.0, "zipf": 1.0, "mixture": 2.0}[recipe]
    if recipe == "zipf":
        prof = 4.0 * torch.arange(1, V + 1, device="cuda", dtype=torch.float32) ** -1.1
    step = max(1, 16_000_000 // (Kt * V))
    for b0 in range(0, B, step):
        b1 = min(B, b0 + step)
        n = (b1 - b0) * Kt
        z = torch.randn((n, V), generator=g, device="cuda")
        rows = torch.arange(n, device="cuda")
        at = torch.randint(0, V, (n,), generator=g, device="cuda")
        u = torch.rand((n, 3), generator=g, device="cuda")
        if recipe == "spike":
            z[rows, at] += 12.0 * u[:, 0]
        elif recipe == "spread":
            z *= 1.5
            z[rows, at] += 10.0 * u[:, 0]
        elif recipe == "zipf":
            order = torch.argsort(torch.rand((n, V), generator=g, device="cuda"), dim=1)
            z = 0.5 * z + prof[order]
        else:                                            # half peaked, 30 % flat, 20 % with two near maxima
            flat, two = (u[:, 0] >= 0.5) & (u[:, 0] < 0.8), u[:, 0] >= 0.8
            z[flat] *= 0.3
            h = torch.where(flat, torch.zeros_like(u[:, 1]), 8.0 + 6.0 * u[:, 1])
            z[rows, at] += h
            z[rows[two], (at[two] + 1) % V] += h[two] - 0.5 * u[two, 2]
        t = torch.randn((n, V), generator=g, device="cuda")
        if recipe == "spread":                           # agreement differs from sequence to sequence
            s = torch.tensor([0.2, 1.0, 3.0], device="cuda")[(b0 + rows // Kt) % 3][:, None]
            t = z + s * t
        else:
            t = z + sig * t
        if c.get("masked"):                              # entries that no sequence may use
            gm = torch.Generator(device="cuda").manual_seed(seed + 5)
            off = torch.rand((V,), generator=gm, device="cuda") < c["masked"]
            off[:2] = False
            z[:, off] = -math.inf
            t[:, off] = -math.inf
        z, t = z.to(dt).view(b1 - b0, Kt, V), t.to(dt).view(b1 - b0, Kt, V)
        draft[b0:b1] = z[:, :K]
        target[b0:b1] = t
        w = z[:, :K].float()
        if recipe != "spike":                            # sampled from the drafter; else its argmax
            e = torch.rand(w.shape, generator=g, device="cuda").clamp_(1e-12, 1 - 1e-7)
            w = w - torch.log(-torch.log(e))
        tokens[b0:b1] = w.argmax(dim=2).to(torch.int32)
    k_row = None
    if c["ragged"]:
        k_row = torch.randint(0, K + 1, (B,), generator=g, device="cuda").to(torch.int32)
        k_row[0] = K
    return draft, target, tokens, k_row


def _lmhead_inputs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 29)
    R, d, V = c["R"], c["d"], c["V"]
    w = torch.empty((V, d), dtype=torch.bfloat16, device="cuda")
    for v0 in range(0, V, 16384):
        v1 = min(V, v0 + 16384)
        w[v0:v1] = (torch.randn((v1 - v0, d), generator=g, device="cuda") / math.sqrt(d)).to(torch.bfloat16)
    h = 0.7 * torch.randn((R, d), generator=g, device="cuda")
    at = torch.randint(0, V, (R,), generator=g, device="cuda")
    a = 16.0 * torch.rand((R, 1), generator=g, device="cuda")
    a[torch.rand((R, 1), generator=g, device="cuda") > 0.7] = 0.0   # 30 % of rows point at no token
    a[0] = 0.0
    p = w[at].float()
    h = h + a * p / (p * p).sum(dim=1, keepdim=True)
    return h.to(torch.bfloat16), w


def _buffers(names, B, K, Ko):
    """Zeroed outputs: entries past a ragged window are left as they are by the calls."""
    z = lambda shape, dt: torch.zeros(shape, dtype=dt, device="cuda")  # noqa: E731
    shapes = dict(H=((B, K), torch.float32), margin=((B, K), torch.float32), conf=((B, K), torch.float32),
                  lse=((B, K), torch.float32), argmax=((B, K), torch.int32), accept=((B, K), torch.uint8),
                  k_next=((B,), torch.int32), n_accept=((B,), torch.int32), out_tokens=((B, Ko), torch.int32))
    return {n: z(*shapes[n]) for n in names}


SIGNALS = ("H", "margin", "conf", "lse", "argmax")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "loop":
        p = cmsd.params(case["K"], case["rule"])
        sim = decode_sim.DecodeSim(case["B"], case["K"], case["V"], case["iterations"], p, seed=1000 + seed)
        sim.step(0)                                      # the one-time set-up of the kernels, before the capture
        torch.cuda.synchronize()
        return dict(kind=kind, sim=sim, graph=sim.capture())
    if kind == "lmhead":
        h, w = _lmhead_inputs(case, seed)
        out = {n: torch.zeros(case["R"], dtype=torch.float32, device="cuda") for n in ("H", "margin", "conf", "lse")}
        out["argmax"] = torch.zeros(case["R"], dtype=torch.int32, device="cuda")
        if case["logits"]:
            out["logits"] = torch.zeros((case["R"], case["V"]), dtype=torch.float32, device="cuda")
        return dict(kind=kind, hidden=h, weight=w, out=out, logits=case["logits"], p=cmsd.params(1),
                    ws=cmsd.lmhead_workspace(case["R"], case["d"], case["V"]))
    B, K, V = case["B"], case["K"], case["V"]
    draft, target, tokens, k_row = _rows(case, seed)
    if kind == "confidence":
        return dict(kind=kind, draft=draft, k_row=k_row, p=cmsd.params(K), ws=cmsd.workspace(B, K, V),
                    out=_buffers(SIGNALS + ("k_next",), B, K, K))
    if kind == "verify":
        p = cmsd.params(K, case["rule"])
        sig = cmsd.confidence(draft, k_row=k_row, p=p, out=_buffers(SIGNALS + ("k_next",), B, K, K))
        return dict(kind=kind, draft=draft, target=target, tokens=tokens, k_row=k_row, p=p, conf=sig["conf"],
                    lse=sig["lse"], seed=seed, ws=cmsd.workspace(B, K, V),
                    out=_buffers(("n_accept", "out_tokens", "accept"), B, K, K))
    p = cmsd.params(K, case["rule"], bonus=case["bonus"])
    names = ("k_next", "n_accept", "out_tokens") + (SIGNALS + ("accept",) if case["signals"] else ())
    out = _buffers(names, B, K, K + 1 if case["bonus"] else K)
    call = cmsd.FusedCall(draft, target, tokens, p, seed=seed, iteration=1, k_row=k_row, out=out,
                          signals=case["signals"])
    return dict(kind=kind, call=call)


def run(state):
    kind = state["kind"]
    if kind == "fused":
        out = state["call"]()
        return {n: t for n, t in out.items() if t is not None}
    if kind == "lmhead":
        return cmsd.lmhead_confidence(state["hidden"], state["weight"], p=state["p"], logits=state["logits"],
                                      out=state["out"], ws=state["ws"])
    if kind == "confidence":
        return cmsd.confidence(state["draft"], k_row=state["k_row"], p=state["p"], out=state["out"], ws=state["ws"])
    if kind == "verify":
        return cmsd.verify(state["draft"], state["target"], state["tokens"], state["conf"], draft_lse=state["lse"],
                           k_row=state["k_row"], p=state["p"], seed=state["seed"], iteration=1, out=state["out"],
                           ws=state["ws"])
    state["graph"].replay()
    sim = state["sim"]
    return {"k": sim.hist_k, "n_accept": sim.hist_n, "out_tokens": sim.hist_tok}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "lmhead":
        R, d, V = case["R"], case["d"], case["V"]
        return {"bytes": 2 * d * (V + R) + 20 * R + (4 * R * V if case["logits"] else 0), "flops": 2 * R * d * V}
    if kind == "loop":                                   # each logit of a window's rows written once and read once
        rows = case["B"] * (case["K"] + (case["iterations"] - 1) * min(MEAN_WINDOW, 0.35 * case["K"]))
        return {"bytes": 2 * rows * 2 * case["V"] * 4, "flops": 30 * rows * 2 * case["V"]}
    B, K, V = case["B"], case["K"], case["V"]
    es = 4 if case["dtype"] == "f32" else 2
    rows = B * K * (0.5 if case["ragged"] else 1.0)      # windows uniform in 0 .. K
    if kind == "confidence":
        return {"bytes": rows * V * es, "flops": 15 * rows * V}
    if kind == "verify":                                 # the drafter's logits: at the drafted token only
        return {"bytes": rows * V * es, "flops": 10 * rows * V}
    return {"bytes": 2 * rows * V * es, "flops": 30 * rows * V}


def tolerance(case):
    # Sums and logarithms in 32 bits.  Against `exact` the signals of the streaming calls are off by up to 1.1e-7
    # (2-norm over the rows), those of the LM head, whose logits carry the rounding of a 32-bit dot product of d
    # terms, by up to 3.4e-6; a few rows average less.  Decisions and tokens are whole values and stay the same.
    if case["kind"] in ("loop", "verify") or (case["kind"] == "fused" and not case["signals"]):
        return "exact"
    if case["kind"] == "lmhead":
        return {"rel": 1.5e-5, "max": 1e-4} if case["R"] >= 16 else {"rel": 4e-5, "max": 2e-4}
    return {"rel": 5e-7, "max": 5e-6} if case["B"] * case["K"] >= 16 else {"rel": 4e-6, "max": 2e-5}


# ---------------------------------------------------------------------------
# the signals in 64 bits
# ---------------------------------------------------------------------------

def _signals64(z):
    """H, margin, conf, lse and argmax of rows z (float64)."""
    V = z.shape[1]
    top = z.topk(2, dim=1).values
    m = top[:, :1]
    e = torch.exp(z - m)
    s = e.sum(dim=1, keepdim=True)
    p = e / s
    H = -torch.special.xlogy(p, p).sum(dim=1)
    margin = top[:, 0] - top[:, 1]
    soft = (1.0 - torch.exp(top[:, 1] - top[:, 0])) / s[:, 0]
    C = (LAM[0] * (1.0 - H / math.log(V)) + LAM[1] * torch.sigmoid(BETA_SIG * margin)
         + LAM[2] * soft / (1.0 - 1.0 / V)).clamp(0.0, 1.0)
    return dict(H=H, margin=margin, conf=C, lse=(m + torch.log(s))[:, 0], argmax=z.argmax(dim=1).to(torch.int32))


def exact(case, seed):
    kind = case["kind"]
    if kind == "lmhead":
        h, w = _lmhead_inputs(case, seed)
        h = h.double()
        z = torch.cat([h @ w[v:v + 8192].double().T for v in range(0, case["V"], 8192)], dim=1)
        out = _signals64(z)
        if case["logits"]:
            out["logits"] = z
        return out
    if kind in ("loop", "verify") or (kind == "fused" and not case["signals"]):
        return None                                      # decisions and tokens only
    B, K, V = case["B"], case["K"], case["V"]
    draft, _, _, k_row = _rows(case, seed)
    z = draft.view(B * K, V)
    step = max(1, 20_000_000 // V)
    parts = [_signals64(z[r:r + step].double()) for r in range(0, B * K, step)]
    out = {n: torch.cat([q[n] for q in parts]).view(B, K) for n in SIGNALS}
    if k_row is not None:
        past = torch.arange(K, device="cuda")[None, :] >= k_row[:, None]
        out = {n: t.masked_fill(past, 0) for n, t in out.items()}
    out["k_next"] = None
    if kind == "fused":
        out.update(n_accept=None, out_tokens=None, accept=None)
    return out
