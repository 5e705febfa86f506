"""Performance cases: the calls a serving program makes of this library, over the
range of sizes it makes them at.

A case is a dict of plain values. `listed()` names the cases, `draw(rng)` gives
one more of the same ranges, `prepare(case, seed)` builds what a program holds
before the call (plan, pool, inputs) on the GPU, `run(state)` makes one pass
through the public entry points and returns every output, `work(case)` states
the bytes and flops one pass cannot do without, and `exact(case, seed)` gives
the outputs in 64 bits by plain torch where they are computed numbers (page
codes are not: they are decisions, and come back as bytes).

Kinds of pass:
  decode    one token through the layers of a slot pool (fused step per layer)
  split     the same token as readout and writeback per layer
  state32   one token on the FP32-state pool; intb: on the rowwise INT-b pool
  prefill   a prompt of `tokens` tokens on FP32 states, one layer
  pages     unpack every layer of `batch` slots to dense states (a checkpoint,
            a continued prompt), and pack dense states into pages (the prefill
            boundary)
  calibrate the calibration protocol on a recorded trace
"""
import math

import numpy as np
import torch

import paper_2609_38169_gb300 as P

D = 128
RING = 4                       # tokens of inputs a decode state cycles through

# Fractions of FP16 pivot units of the paper's two models (heads, key rows).
PIVOT_HEADS, PIVOT_ROWS = 32 / 2304, 512 / 81920


def _decode(name, kind="decode", gate="scalar", layers=1, hk=32, hv=32, batch=1, slots=0, bits=6,
            pivots=0, fit_iters=1):
    return {"name": name, "kind": kind, "gate": gate, "layers": layers, "hk": hk, "hv": hv,
            "batch": batch, "slots": slots or batch, "bits": bits, "pivots": pivots,
            "fit_iters": fit_iters}


def listed():
    return [
        # One request on a small model, one layer: the smallest call, all latency.
        _decode("decode_tiny", hk=4, hv=4, batch=1),
        # A GQA layer (16 key heads, 32 value heads) at an ordinary batch.
        _decode("decode_gqa", hk=16, hv=32, batch=64),
        # The serving pool: 1024 slots in random order, four layers, FP16 pivot heads.
        _decode("decode_pool", layers=4, batch=1024, pivots=2),
        # The side-stream form of the step (readout, then writeback) on the GQA layer.
        _decode("split_gqa", kind="split", hk=16, hv=32, batch=256),
        # Channel gates, 4-bit plan with widths {2, 4, 6, 8} per key row and pivot rows.
        _decode("decode_channel", gate="channel", batch=256, bits=4, pivots=26),
        # Channel gates at 6 bits over four layers: the long-generation workload.
        _decode("decode_drift", gate="channel", layers=4, batch=128, bits=6, pivots=102),
        # The uncompressed serving default: FP32 states on the GQA layer.
        _decode("state32_gqa", kind="state32", hk=16, hv=32, batch=64, bits=32),
        # Uniform rowwise INT8 states on the channel-gate layer.
        _decode("int8_channel", kind="intb", gate="channel", batch=256, bits=8),
        # Prompts of 512 tokens for a full batch, scalar gates.
        {"name": "prefill_gqa", "kind": "prefill", "gate": "scalar", "hk": 16, "hv": 32,
         "batch": 128, "tokens": 512},
        # A few prompts of an odd length, channel gates: fewer heads than SMs.
        {"name": "prefill_channel", "kind": "prefill", "gate": "channel", "hk": 32, "hv": 32,
         "batch": 3, "tokens": 333},
        # Pages to dense states and back for 64 slots of a four-layer pool.
        {"name": "pages_pool", "kind": "pages", "gate": "scalar", "layers": 4, "hk": 32, "hv": 32,
         "batch": 64, "bits": 6, "pivots": 2},
        # Calibration of the four-layer channel-gate model: 8 sequences of 256 tokens.
        {"name": "calibrate_drift", "kind": "calibrate", "gate": "channel", "layers": 4, "hk": 32,
         "hv": 32, "batch": 8, "tokens": 256, "every": 8, "bits": 6, "pivots": 102},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode"] * 5 + ["split", "state32", "intb", "prefill", "prefill", "pages", "calibrate"])
    gate = rng.choice(["scalar", "scalar", "scalar", "channel", "channel"])
    hv = rng.choice([4, 6, 8, 12, 16, 24, 32])
    hk = hv // rng.choice([g for g in (1, 2, 4) if hv % g == 0])
    layers = rng.choice([1, 1, 2, 3, 4])
    bits = rng.choice([6, 6, 4, 8])
    frac = PIVOT_ROWS * D if gate == "channel" else PIVOT_HEADS
    pivots = int(layers * hv * frac + rng.random())
    if kind == "prefill":
        tokens = _log(rng, 16, 2048)
        most = max(1, min(128, 128 * 512 * 32 // (tokens * hv)))
        return {"kind": kind, "gate": gate, "hk": hk, "hv": hv, "batch": _log(rng, 1, most), "tokens": tokens}
    if kind == "pages":
        return {"kind": kind, "gate": gate, "layers": layers, "hk": hk, "hv": hv,
                "batch": _log(rng, 1, 128), "bits": bits, "pivots": pivots}
    if kind == "calibrate":
        return {"kind": kind, "gate": gate, "layers": layers, "hk": hk, "hv": hv,
                "batch": rng.randint(1, 8), "tokens": _log(rng, 16, 256), "every": rng.choice([4, 8, 16]),
                "bits": bits, "pivots": pivots}
    batch = _log(rng, 1, 1024)
    if kind == "state32":
        bits, pivots, batch = 32, 0, min(batch, 24576 // (layers * hv))
    if kind == "intb":
        bits, pivots = rng.choice([8, 6, 4]), 0
    c = _decode("", kind, gate, layers, hk, hv, batch, batch + rng.choice([0, 0, rng.randint(1, 64)]), bits,
                pivots, rng.choice([1, 1, 1, 2]) if kind in ("decode", "split") else 1)
    del c["name"]
    return c


# ------------------------------------------------------------------ preparation
def _candidates(c):
    return (2, 4, 6, 8) if c["bits"] == 4 else (4, 6, 8)


def _config(c):
    return P.Config(n_layers=c.get("layers", 1), n_key_heads=c["hk"], n_value_heads=c["hv"],
                    gate_kind=P.GATE_CHANNEL if c["gate"] == "channel" else P.GATE_SCALAR,
                    nominal_bits=c["bits"] if c.get("bits") in (4, 6, 8) else 6,
                    candidates=_candidates(c) if c.get("bits") in (4, 6, 8) else (4, 6, 8),
                    n_pivots=c.get("pivots", 0), fit_iters=c.get("fit_iters", 1))


def _plan(cfg, seed):
    """A plan from statistics of the form calibration gives: lognormal row
    impacts, retentions near one, distortions that fall by 4 per bit."""
    g = np.random.default_rng([seed, 1])
    n = P.stepq_num_units(cfg)
    omega = g.lognormal(0.0, 1.0, (cfg.n_layers, cfg.n_value_heads, D)).astype(np.float32)
    ell = np.log(g.uniform(0.85, 0.999, n))
    scale = g.lognormal(0.0, 1.5, n)
    dist = scale[:, None] * np.array([4.0 ** -b for b in cfg.candidates] + [4.0 ** -11])[None]
    return P.stepq_fit_scales(cfg, omega, ell, dist)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _states(g, n, hv):
    """Dense states with a spread of row and column magnitudes."""
    s = torch.randn((n, hv, D, D), generator=g, device="cuda")
    s *= torch.exp(0.7 * torch.randn((n, hv, D, 1), generator=g, device="cuda"))
    s *= 0.3 * torch.exp(0.5 * torch.randn((n, hv, 1, D), generator=g, device="cuda"))
    return s


def _inputs(g, lead, c):
    """q, k, v, beta, gate with the leading shape `lead`: normal q and v, unit
    keys, sigmoid write strengths; scalar gates in (0.9, 0.999), a quarter of the
    heads long-lived; channel gates in (0.8, 0.999)."""
    hk, hv = c["hk"], c["hv"]
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    uni = lambda *s: torch.rand(s, generator=g, device="cuda")  # noqa: E731
    q, k, v = rnd(*lead, hk, D), rnd(*lead, hk, D), rnd(*lead, hv, D)
    if c["gate"] == "channel":
        k *= torch.exp(rnd(hk, D))
    k /= torch.linalg.vector_norm(k, dim=-1, keepdim=True)
    beta = torch.sigmoid(rnd(*lead, hv))
    if c["gate"] == "channel":
        base = 0.8 + 0.199 * uni(hv, D)
        gate = (base * torch.exp(0.01 * rnd(*lead, hv, D))).clamp_(0.8, 0.999)
    else:
        long_lived = uni(hv) < 0.25
        u = uni(*lead, hv)
        gate = torch.where(long_lived, 0.998 + 0.001 * u, 0.9 + 0.099 * u)
    return [x.contiguous() for x in (q, k, v, beta, gate)]


def _slots(g, batch, slots):
    return torch.randperm(slots, generator=g, device="cuda")[:batch].to(torch.int32)


def prepare(case, seed):
    c, g, cfg = case, _gen(seed), _config(case)
    B, L, hv = c["batch"], c.get("layers", 1), c["hv"]
    st = {"case": c, "cfg": cfg, "t": 0}
    if c["kind"] == "prefill":
        st["states"] = _states(g, B, hv)
        st["in"] = _inputs(g, (B, c["tokens"]), c)
        st["y"] = torch.empty((B, c["tokens"], hv, D), device="cuda")
        return st
    if c["kind"] == "calibrate":
        st["in"] = _inputs(g, (L, c["tokens"], B), c)
        return st
    if c["kind"] == "pages":
        st["plan"] = plan = _plan(cfg, seed)
        st["slots"], st["to"] = _slots(g, B, B), _slots(g, B, B)
        st["pool"], st["packed"] = P.alloc_pool(plan, B), P.alloc_pool(plan, B)
        every = torch.arange(B, dtype=torch.int32, device="cuda")
        for layer in range(L):
            P.stepq_quantize_pool(plan, layer, _states(g, B, hv), every, st["pool"])
        st["dense"] = torch.empty((B, L, hv, D, D), device="cuda")
        st["states"] = torch.stack([_states(g, B, hv) for _ in range(L)], dim=1)
        return st
    S = c["slots"]
    st["slots"] = _slots(g, B, S)
    every = torch.arange(S, dtype=torch.int32, device="cuda")
    if c["kind"] == "state32":
        st["pool"] = torch.stack([_states(g, S, hv) for _ in range(L)], dim=1)
    elif c["kind"] == "intb":
        st["pool"] = torch.zeros(S * P.stepq_intb_slot_bytes(cfg, c["bits"]), dtype=torch.uint8, device="cuda")
        for layer in range(L):
            P.stepq_intb_quantize_pool(cfg, c["bits"], layer, _states(g, S, hv), every, st["pool"])
    else:
        st["plan"] = plan = _plan(cfg, seed)
        st["pool"] = P.alloc_pool(plan, S)
        for layer in range(L):
            P.stepq_quantize_pool(plan, layer, _states(g, S, hv), every, st["pool"])
        if c["kind"] == "split":
            st["delta"] = torch.empty((L, B, hv, D), device="cuda")
    st["in"] = [[_inputs(g, (B,), c) for _ in range(L)] for _ in range(RING)]
    st["y"] = torch.empty((L, B, hv, D), device="cuda")
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    c, cfg = st["case"], st["cfg"]
    if c["kind"] == "prefill":
        P.stepq_prefill_fp32(cfg, st["states"], *st["in"], st["y"])
        return {"y": st["y"], "states": st["states"]}
    if c["kind"] == "calibrate":
        s = P.stepq_calibrate_from_trace(cfg, *st["in"], every=c["every"])
        return {"omega": s.omega, "ell": s.mean_log_ret, "dist": s.dist, "dist1": s.dist_stage1,
                "pivot": s.pivot}
    if c["kind"] == "pages":
        P.stepq_dequantize_pool(st["plan"], -1, st["pool"], st["slots"], st["dense"])
        P.stepq_quantize_pool(st["plan"], -1, st["states"], st["to"], st["packed"])
        return {"dense": st["dense"], "packed": st["packed"]}
    token = st["in"][st["t"] % RING]
    st["t"] += 1
    pool, slots, y = st["pool"], st["slots"], st["y"]
    for layer in range(cfg.n_layers):
        q, k, v, beta, gate = token[layer]
        if c["kind"] == "decode":
            P.stepq_decode_step(st["plan"], layer, pool, slots, q, k, v, beta, gate, y[layer])
        elif c["kind"] == "split":
            P.stepq_decode_readout(st["plan"], layer, pool, slots, q, k, v, beta, gate, y[layer],
                                   st["delta"][layer])
            P.stepq_decode_writeback(st["plan"], layer, pool, slots, k, beta, gate, st["delta"][layer])
        elif c["kind"] == "state32":
            P.stepq_fp32_decode_step(cfg, layer, pool, slots, q, k, v, beta, gate, y[layer])
        else:
            P.stepq_intb_decode_step(cfg, c["bits"], layer, pool, slots, q, k, v, beta, gate, y[layer])
    out = {"y": y, "pool": pool}
    if c["kind"] == "split":
        out["delta"] = st["delta"]
    return out


# ------------------------------------------------------------------ floors
def work(case):
    c = case
    B, L, hv, hk, N = c["batch"], c.get("layers", 1), c["hv"], c["hk"], D * D
    gate = D if c["gate"] == "channel" else 1
    vec = 4 * (2 * hk * D + 2 * hv * D + hv + hv * gate)       # q k, v y, beta, gate of one token
    if c["kind"] == "prefill":
        # the recurrence in chunkwise form: three N-sized products per token and head
        return {"bytes": B * (hv * 2 * 4 * N + c["tokens"] * vec), "flops": B * c["tokens"] * hv * 6.0 * N}
    if c["kind"] == "calibrate":
        passes = 2 if c["gate"] == "channel" and c["pivots"] else 1
        tok = L * c["tokens"] * B
        fits = tok / c["every"] * hv * N * len(_candidates(c))
        return {"bytes": tok * vec, "flops": passes * (tok * hv * 6.0 * N + fits * 16.0)}
    head = {"state32": 4.0 * N, "intb": 256 + N * c["bits"] / 8}.get(c["kind"], 512 + N * c["bits"] / 8)
    piv = c["pivots"] * (D if c["gate"] == "channel" else N)      # an FP16 unit takes 8 bits a value more
    pages = B * (L * hv * head + piv)
    if c["kind"] == "pages":
        return {"bytes": 2 * (B * L * hv * 4 * N + pages), "flops": B * L * hv * 16.0 * N}
    flops = B * L * hv * N * (6.0 if c["kind"] == "state32" else 10.0 if c["kind"] == "intb" else 16.0)
    if c["kind"] == "split":                                      # two calls: the page is read by each
        return {"bytes": 3 * pages + B * L * (vec + 4 * (hk * D + 2 * hv * D + hv + hv * gate)), "flops": flops}
    return {"bytes": 2 * pages + B * L * vec, "flops": flops}


# ------------------------------------------------------------------ 64 bits
def _codes(raw, b):
    """[..., n bytes] of LSB-first b-bit codes -> [..., 8 n / b] signed codes (offset binary)."""
    bits = (raw[..., None] >> torch.arange(8, device=raw.device, dtype=torch.uint8)) & 1
    bits = bits.reshape(*raw.shape[:-1], -1, b).to(torch.float64)
    return bits @ (2.0 ** torch.arange(b, device=raw.device, dtype=torch.float64)) - 2.0 ** (b - 1)


def _f16(raw):
    return raw.contiguous().view(torch.float16).to(torch.float64)


def _unpack_head(seg, b):
    """Head segments [n][bytes] of one head unit of width b -> states [n][128][128]."""
    n, piv = seg.shape[0], b == 16
    # a lane's stream (four chunks of 16 codes): pieces of 16 bytes, interleaved over 32 lanes
    body = seg[:, 0 if piv else 512:].reshape(n, 8, b // 2, 32, 16).permute(0, 1, 3, 2, 4).reshape(n, 8, 32, 8 * b)
    v = _f16(body) if piv else _codes(body.contiguous(), b)
    v = v.reshape(n, 8, 4, 8, 4, 16)                              # warp, column quad, band, column, row
    v = v.permute(0, 3, 5, 1, 2, 4).reshape(n, D, D)
    return v if piv else v * _f16(seg[:, :256])[:, :, None] * _f16(seg[:, 256:512])[:, None, :]


def _unpack_rows(seg, widths):
    """Head segments of row units (128 widths, rows stored by decreasing width) -> states."""
    out = torch.empty((seg.shape[0], D, D), dtype=torch.float64, device=seg.device)
    r, cc = _f16(seg[:, :256]), _f16(seg[:, 256:512])
    at = 512
    for i in sorted(range(D), key=lambda i: -widths[i]):
        b = int(widths[i])
        raw = seg[:, at:at + 16 * b].contiguous()
        out[:, i] = _f16(raw) if b == 16 else _codes(raw, b) * 2.0 ** (8 - b) * r[:, i:i + 1] * cc
        at += 16 * b
    return out


def _head_state(st, layer, h):
    """Dense state [B][128][128] in 64 bits of one head of the batch's slots."""
    c, hv = st["case"], st["case"]["hv"]
    slots = st["slots"].long()
    if c["kind"] == "state32":
        return st["pool"][slots, layer, h].double()
    if c["kind"] == "intb":
        size = 256 + 16 * c["bits"] * D
        pages = st["pool"].view(c["slots"], -1)
        seg = pages[slots, (layer * hv + h) * size:(layer * hv + h + 1) * size]
        return _codes(seg[:, 256:].reshape(-1, D, 16 * c["bits"]), c["bits"]) * _f16(seg[:, :256])[:, :, None]
    plan, at = st["plan"], layer * hv + h
    off, size = int(plan.head_offset[at]), int(plan.head_bytes[at])
    seg = st["pool"].view(-1, plan.slot_stride)[slots, off:off + size].contiguous()
    if c["gate"] == "channel":
        return _unpack_rows(seg, plan.unit_bits[at * D:(at + 1) * D])
    return _unpack_head(seg, int(plan.unit_bits[at]))


def _step(S, q, k, v, beta, gate):
    """One gated Delta step in place: S [n][128][128], gate [n] or [n][128]."""
    S *= gate.reshape(S.shape[0], -1, 1)
    delta = v - torch.einsum("nij,ni->nj", S, k)
    S += (beta[:, None] * k)[:, :, None] * delta[:, None, :]
    return torch.einsum("nij,ni->nj", S, q), delta


def exact(case, seed):
    c = case
    st = prepare(case, seed)
    hv, grp = c["hv"], c["hv"] // c["hk"]
    if c["kind"] == "prefill":
        B, T = c["batch"], c["tokens"]
        q, k, v, beta, gate = [x.double() for x in st["in"]]
        S = st["states"].double().reshape(B * hv, D, D)
        y = torch.empty((B, T, hv, D), dtype=torch.float64, device="cuda")
        for t in range(T):
            args = (q[:, t].repeat_interleave(grp, 1).reshape(-1, D), k[:, t].repeat_interleave(grp, 1).reshape(-1, D),
                    v[:, t].reshape(-1, D), beta[:, t].reshape(-1), gate[:, t].reshape(B * hv, -1))
            y[:, t] = _step(S, *args)[0].reshape(B, hv, D)
        return {"y": y, "states": S.reshape(B, hv, D, D)}
    if c["kind"] == "calibrate":
        q, k, _, beta, gate = [x.double() for x in st["in"]]
        q, k = q.repeat_interleave(grp, 3), k.repeat_interleave(grp, 3)
        d = gate if c["gate"] == "channel" else gate[..., None]
        imp = d * (q - beta[..., None] * k * (k * q).sum(-1, keepdim=True))
        return {"omega": imp.square().mean((1, 2)).cpu().numpy(),
                "ell": torch.log(gate).mean((1, 2)).reshape(-1).cpu().numpy(),
                "dist": None, "dist1": None, "pivot": None}
    if c["kind"] == "pages":
        dense = torch.stack([torch.stack([_head_state(st, layer, h) for h in range(hv)], dim=1)
                             for layer in range(c["layers"])], dim=1)
        return {"dense": dense, "packed": None}
    L, B = c["layers"], c["batch"]
    y = torch.empty((L, B, hv, D), dtype=torch.float64, device="cuda")
    delta = torch.empty_like(y)
    pool = st["pool"].double() if c["kind"] == "state32" else None
    slots = st["slots"].long()
    for layer in range(L):
        q, k, v, beta, gate = [x.double() for x in st["in"][0][layer]]
        for h in range(hv):
            S = _head_state(st, layer, h)
            y[layer, :, h], delta[layer, :, h] = _step(S, q[:, h // grp], k[:, h // grp], v[:, h], beta[:, h], gate[:, h])
            if pool is not None:
                pool[slots, layer, h] = S
    out = {"y": y, "pool": pool}
    if c["kind"] == "split":
        out["delta"] = delta
    return out
