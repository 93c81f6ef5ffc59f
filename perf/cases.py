"""The work that a user of this framework has it do, as cases that can be timed and compared.

A case names a call (``do``) and a layer (``layer``) with its sizes and options:

* ``prefill``  a prompt from the empty state: qstate_init, then qstate_scan over its T tokens;
* ``decode``   a batch of running sequences: qstate_scan over the next T tokens, or, with
               ``call`` = "step", qstate_step for the next token, as a serving loop calls it;
* ``gate``     qstate_quant_decay over a batch's decay rates;
* ``pack`` / ``unpack``  a dense state into the packed form and back (a state taken over from
               another engine, or handed to one);
* ``fp32``     qstate_scan_fp32, the same layer on an unquantised state.

Layers and their distributions are those of the repository's workloads: ``kda`` (decay per key
row, delta rule), ``gdn`` (Gated DeltaNet: decay per head, head unit), ``mamba2`` (decay per head,
no erasure), ``general`` (KDA with a and w given per token).
"""
import math

import torch

import paper_2609_30950_gb300 as qs

# Decode cases keep a ring of tokens: the first WARM of them bring the state to where a running
# sequence has it (widths allocated, statistics settled, ranges of a few tokens' mixture).
WARM = 16

LAYERS = {
    "kda": dict(decay_kind=qs.DECAY_ROW, erase_kind=qs.ERASE_DELTA, unit_kind=qs.UNIT_ROW),
    "general": dict(decay_kind=qs.DECAY_ROW, erase_kind=qs.ERASE_GENERAL, unit_kind=qs.UNIT_ROW),
    "gdn": dict(decay_kind=qs.DECAY_HEAD, erase_kind=qs.ERASE_DELTA, unit_kind=qs.UNIT_HEAD),
    "mamba2": dict(decay_kind=qs.DECAY_HEAD, erase_kind=qs.ERASE_NONE, unit_kind=qs.UNIT_ROW),
}


def listed():
    return [
        # the smallest recurrence: one 64 x 64 head, 256 tokens, two bits, a write-back per token;
        # nothing but latency and launches
        dict(name="tiny_scan", do="prefill", layer="kda", B=1, H=1, dk=64, dv=64, T=256, C=1, bits=2, bmin=1, bmax=16),
        # one sequence being generated: one token of a 32-head KDA layer
        dict(name="kda_step_b1", do="decode", call="step", layer="kda", B=1, H=32, dk=128, dv=128, T=1, C=1, bits=4,
             bmin=0, bmax=8, gate=2),
        # an ordinary, odd-sized serving batch on exact rates, factors refitted every 16th token
        dict(name="kda_step_b37_fit16", do="decode", call="step", layer="kda", B=37, H=16, dk=128, dv=128, T=1, C=1,
             bits=4, bmin=1, bmax=8, fit_every=16),
        # the full KDA decode batch, four tokens in one call
        dict(name="kda_scan_b256", do="decode", layer="kda", B=256, H=32, dk=128, dv=128, T=4, C=1, bits=4, bmin=0,
             bmax=8, gate=2),
        # Gated DeltaNet decode: one width per head, block scales
        dict(name="gdn_scan_b64", do="decode", layer="gdn", B=64, H=16, dk=128, dv=128, T=16, C=1, bits=4, bmin=2,
             bmax=16),
        # Mamba-2 decode: 128 x 64 states, six bits, heads normalised in groups of eight
        dict(name="mamba2_scan_b128", do="decode", layer="mamba2", B=128, H=64, dk=128, dv=64, T=4, C=1, bits=6,
             bmin=1, bmax=16, group=8),
        # prompts of a batch, a write-back every 64 tokens, in chunked form
        dict(name="kda_prefill_b16", do="prefill", layer="kda", B=16, H=32, dk=128, dv=128, T=512, C=64, bits=3,
             bmin=1, bmax=8, chunk=True),
        # one prompt of a length that is no multiple of the write-back period
        dict(name="kda_prefill_b1", do="prefill", layer="kda", B=1, H=32, dk=128, dv=128, T=1000, C=64, bits=3,
             bmin=1, bmax=8, chunk=True),
        # the decay rates of a prefill batch to two-bit codes
        dict(name="gate_b16", do="gate", layer="kda", B=16, H=32, dk=128, dv=128, T=1024, C=64, bits=3, bmin=1,
             bmax=8, gate=2),
        # a batch of dense states into the packed form, and back
        dict(name="pack_b64", do="pack", layer="kda", B=64, H=32, dk=128, dv=128, T=1, C=1, bits=4, bmin=1, bmax=8),
        dict(name="unpack_b64", do="unpack", layer="kda", B=64, H=32, dk=128, dv=128, T=1, C=1, bits=4, bmin=1,
             bmax=8),
        # the layer without quantisation, to compare with
        dict(name="fp32_scan_b16", do="fp32", layer="kda", B=16, H=32, dk=128, dv=128, T=32, C=1, bits=4, bmin=1,
             bmax=8),
    ]


def draw(rng):
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    do = rng.choice(["decode", "decode", "decode", "prefill", "prefill", "gate", "pack", "unpack", "fp32"])
    layer = rng.choice(["kda", "kda", "gdn", "mamba2"] + (["general"] if do in ("decode", "prefill", "fp32") else []))
    H = log_int(1, 64)
    B = min(log_int(1, 256), 8192 // H)
    dk, dv = rng.choice([(128, 128), (128, 128), (128, 128), (128, 64), (64, 64)])
    c = dict(do=do, layer=layer, B=B, H=H, dk=dk, dv=dv, T=1, C=1)
    if layer == "gdn":
        c.update(bits=rng.choice([3, 4, 6]), bmin=2, bmax=rng.choice([8, 16]))
    elif layer == "mamba2":
        c.update(bits=rng.choice([4, 6]), bmin=1, bmax=16)
        c["group"] = rng.choice([g for g in (1, 2, 4, 8) if H % g == 0])
    else:
        c.update(bits=rng.choice([2, 3, 4]), bmin=rng.choice([0, 1]), bmax=8)
    if layer in ("kda", "general") and rng.random() < 0.5:
        c["gate"] = rng.choice([2, 2, 3, 4])
    if do == "decode":
        if rng.random() < 0.5:
            c["call"] = "step"
        else:
            c["T"] = log_int(2, 8)
        if rng.random() < 0.3:
            c["fit_every"] = rng.choice([4, 16])
        if layer == "kda" and rng.random() < 0.15:
            c["current"] = True
    elif do == "prefill":
        c["C"] = rng.choice([16, 64, 64, 64])
        c["B"] = B = min(B, max(1, 512 // H))
        c["T"] = log_int(c["C"] // 2, 512)
        if layer == "kda" and dk == dv == 128 and rng.random() < 0.8:
            c["chunk"] = True
    elif do == "gate":
        c["gate"] = c.get("gate", rng.choice([1, 2, 3]))
        c["T"] = log_int(8, max(8, min(4096, 67_000_000 // (B * H * dk))))
    elif do == "fp32":
        c["B"] = B = min(B, max(1, 1024 // H))
        c["T"] = log_int(2, 64)
        c["C"] = rng.choice([1, 1, 16, 64])
    return c


def config(case):
    return qs.Config(B=case["B"], H=case["H"], dk=case["dk"], dv=case["dv"], group_heads=case.get("group", 1),
                     bbar_num=case["bits"], bbar_den=1, bmin=case["bmin"], bmax=case["bmax"], C=case["C"],
                     fit_every=case.get("fit_every", 1), gate_bits=case.get("gate", 0),
                     alloc_mode=qs.ALLOC_CURRENT if case.get("current") else qs.ALLOC_LAGGED,
                     interval_form=qs.FORM_CHUNK if case.get("chunk") else qs.FORM_TOKEN, **LAYERS[case["layer"]])


def rates(case, T, gen):
    """Decay rates softplus(N(mu, 1)), mu = -2 per key row (KDA) or -3 per head."""
    row = LAYERS[case["layer"]]["decay_kind"] == qs.DECAY_ROW
    shape = (case["B"], T, case["H"]) + ((case["dk"],) if row else ())
    z = torch.randn(shape, device="cuda", generator=gen) + (-2.0 if row else -3.0)
    return torch.nn.functional.softplus(z)


def tokens(case, T, gen):
    """Inputs of T tokens: unit-norm keys and queries (N(0, 1/128) for Mamba-2), v ~ N(0, 1),
    beta = sigmoid(N(0, 1)); general erasure: a near beta k, w = sigmoid(N(0, 1))."""
    B, H, dk, dv, layer = case["B"], case["H"], case["dk"], case["dv"], case["layer"]
    rnd = lambda *s: torch.randn(s, device="cuda", generator=gen)  # noqa: E731

    def keys():
        g = rnd(B, T, H, dk)
        return g / math.sqrt(128.0) if layer == "mamba2" else g / torch.linalg.vector_norm(g, dim=-1, keepdim=True)

    x = qs.Inputs(q=keys(), k=keys(), v=rnd(B, T, H, dv), s=rates(case, T, gen), T=T)
    beta = torch.sigmoid(rnd(B, T, H))
    if layer in ("kda", "gdn"):
        x.beta = beta
    elif layer == "general":
        x.a = beta[..., None] * (x.k + (0.1 / math.sqrt(dk)) * rnd(B, T, H, dk))
        x.w = torch.sigmoid(rnd(B, T, H, dv))
    return x


def code_rates(cfg, x):
    """The rates of x as log-quantised codes and levels, where the layer quantises its gates."""
    row = cfg.decay_kind == qs.DECAY_ROW
    chan, L = cfg.H * (cfg.dk if row else 1), 1 << cfg.gate_bits
    x.s_code = torch.empty(x.s.shape, dtype=torch.uint8, device="cuda")
    x.s_lut = torch.empty(chan * L, device="cuda")
    qs.qstate_quant_decay(cfg, x.s, x.s_code, x.s_lut, torch.empty(chan * (L - 1), device="cuda"))
    x.s = None


def dense_state(case, gen):
    """A dense state whose key rows spread over two decades."""
    shape = (case["B"], case["H"], case["dk"], case["dv"])
    scale = torch.exp(math.log(10.0) * (2.0 * torch.rand(shape[:3] + (1,), device="cuda", generator=gen) - 1.0))
    return torch.randn(shape, device="cuda", generator=gen) * scale


def spread_widths(cfg, st, state, gen):
    """Widths as the layer's own allocation gives them for rows of different decay and range."""
    n = cfg.B * cfg.units
    uni = lambda lo, hi: torch.exp(math.log(lo) + math.log(hi / lo) * torch.rand(n, device="cuda", generator=gen))  # noqa: E731
    st.ema_s.copy_(uni(0.05, 0.6))
    st.ema_r.copy_(uni(1e-4, 0.02))
    st.range.copy_(uni(0.3, 3.0))
    qs.qstate_alloc_bits(cfg, st, state.widths, state.head_off)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 1000003 + 7)
    cfg, do, T = config(case), case["do"], case["T"]
    B, H, dk, dv = cfg.B, cfg.H, cfg.dk, cfg.dv
    if do == "gate":
        s = rates(case, T, gen)
        chan, L = s[0, 0].numel(), 1 << cfg.gate_bits
        return dict(do=do, cfg=cfg, s=s, codes=torch.empty(s.shape, dtype=torch.uint8, device="cuda"),
                    lut=torch.empty(chan * L, device="cuda"), thr=torch.empty(chan * (L - 1), device="cuda"))
    if do in ("pack", "unpack"):
        a, st, S = qs.new_state(cfg), qs.new_stats(cfg), dense_state(case, gen)
        spread_widths(cfg, st, a, gen)
        if do == "unpack":
            qs.qstate_pack(cfg, S, a)
            S = torch.empty_like(S)
        return dict(do=do, cfg=cfg, a=a, S=S, range=st.range if cfg.unit_kind == qs.UNIT_ROW else None)
    if do == "fp32":
        x = tokens(case, T, gen)
        if cfg.gate_bits:
            code_rates(cfg, x)
        return dict(do=do, cfg=cfg, x=x, T=T, S=0.1 * dense_state(case, gen),
                    o=torch.empty((B, T, H, dv), device="cuda"))
    warm = WARM if do == "decode" else 0
    total = warm + (T if do == "prefill" else max(2 * T, 8))   # decode: a ring of tokens after the warm-up
    x = tokens(case, total, gen)
    if cfg.gate_bits:
        code_rates(cfg, x)
    s = dict(do=do, call=case.get("call"), cfg=cfg, x=x, n=T, warm=warm, total=total, t=warm, w=warm,
             a=qs.new_state(cfg), b=qs.new_state(cfg), st=qs.new_stats(cfg),
             o=torch.zeros((B, total, H, dv), device="cuda"))
    if do == "decode":
        qs.qstate_init(cfg, s["a"], s["b"])
        if qs.qstate_scan(cfg, s["a"], s["b"], x, 0, warm, 0, s["o"], s["st"]):
            s["a"], s["b"] = s["b"], s["a"]
    return s


def run(s):
    do, cfg = s["do"], s["cfg"]
    if do == "gate":
        qs.qstate_quant_decay(cfg, s["s"], s["codes"], s["lut"], s["thr"])
        return dict(codes=s["codes"], lut=s["lut"], thr=s["thr"])
    if do == "pack":
        qs.qstate_pack(cfg, s["S"], s["a"], s["range"])
        a = s["a"]
        return dict(payload=a.payload, scales=a.scales, fidx=a.fidx, range=s["range"])
    if do == "unpack":
        qs.qstate_unpack(cfg, s["a"], s["S"])
        return dict(S=s["S"])
    if do == "fp32":
        qs.qstate_scan_fp32(cfg, s["S"], s["x"], 0, s["T"], s["o"])
        return dict(S=s["S"], o=s["o"])
    a, b, n = s["a"], s["b"], s["n"]
    if do == "prefill":
        t, w = 0, 0
        qs.qstate_init(cfg, a, b)
    else:
        t, w = s["t"], s["w"]
        if t + n > s["total"]:
            t = s["warm"]
        s["t"], s["w"] = t + n, w + n
    if s["call"] == "step":
        qs.qstate_step(cfg, a, b, s["x"], t, t + 1, w, s["o"], s["st"])
        a, b = b, a
    elif qs.qstate_scan(cfg, a, b, s["x"], t, t + n, w, s["o"], s["st"]):
        a, b = b, a
    if do == "decode":
        s["a"], s["b"] = a, b
    st = s["st"]
    return dict(o=s["o"][:, t:t + n], payload=a.payload, scales=a.scales, widths=a.widths, head_off=a.head_off,
                fidx=a.fidx, next_widths=b.widths, ema_s=st.ema_s, ema_r=st.ema_r,
                range=st.range if cfg.unit_kind == qs.UNIT_ROW else None)


def work(case):
    """Each input read once and each output written once; a state that stays between tokens of a
    call is read and written once per write-back, as it is stored in between by definition (the
    unquantised state once per call).  Operations: the recurrence (decay, two reductions, one
    rank-one update: 7 per element and token) and, per write-back, the rounding of each element;
    the fit of the range factors is a choice of method and not counted."""
    B, H, dk, dv, T, C = (case[k] for k in ("B", "H", "dk", "dv", "T", "C"))
    row = LAYERS[case["layer"]]["decay_kind"] == qs.DECAY_ROW
    gate, do, heads, elems = case.get("gate", 0), case["do"], B * H, B * H * dk * dv
    if do == "gate":
        n = B * T * H * (dk if row else 1)
        return dict(bytes=5 * n, flops=(1 << gate) * n)
    unit_row = LAYERS[case["layer"]]["unit_kind"] == qs.UNIT_ROW
    units, groups = heads * (dk if unit_row else 1), heads * (dk if unit_row else dk // 32 * dv)
    packed = elems * case["bits"] / 8 + 3 * groups + units + 4 * heads
    if do in ("pack", "unpack"):
        return dict(bytes=4 * elems + packed, flops=3 * elems)
    per_rate = (1 if gate else 4) * (dk if row else 1)
    per_token = 4 * (2 * dk + 2 * dv) + per_rate
    per_token += 4 if case["layer"] in ("kda", "gdn") else 4 * (dk + dv) if case["layer"] == "general" else 0
    if do == "fp32":
        return dict(bytes=8 * elems + heads * T * per_token, flops=7 * elems * T)
    backs = -(-T // C)
    moved = backs * (2 * packed + 20 * units) + heads * T * per_token
    return dict(bytes=moved, flops=elems * (7 * T + 3 * backs))


def tolerance(case):
    """Four times what inputs moved by half a unit in the last place change, over these ranges.
    A rounding that falls the other way moves a code by a whole step, which later write-backs carry
    on, and an allocation that falls the other way by one bit shifts the rows behind it: so the more
    write-backs a pass (and the passes before it on the same state) holds, the further apart two
    correct results are."""
    do = case["do"]
    if do == "gate":      # codes do not differ; levels and thresholds are rounded once from 64 bits
        return {"rel": 2.4e-7, "max": 1e-6}
    if do == "unpack":    # one rounding per element
        return "exact"
    if do == "pack":      # ranges do not differ; two factors may tie within rounding
        return {"rel": 1e-7, "differ": 4e-4}
    if do == "fp32":
        return {"rel": 1e-6, "max": 1e-5}
    if do == "prefill":
        return {"rel": 1.4e-3, "max": 0.99, "differ": 4e-3}
    if case.get("call") == "step":
        return {"rel": 1e-3, "max": 0.3, "differ": 4e-3}
    return {"rel": 2e-2, "max": 0.99, "differ": 1e-2}


def unpacked(cfg, a):
    """The dense state, in 64 bits, of a packed one: row i of a head holds dv codes of its width,
    least significant bit first; two bits and more: (code - n) * step, n = 2^(width-1) - 1; one bit:
    the sign of the mean; no bits: zero."""
    B, H, dk, dv = cfg.B, cfg.H, cfg.dk, cfg.dv
    S = torch.empty((B, H, dk, dv), dtype=torch.float64, device="cuda")
    region = a.payload.numel() // B
    j = torch.arange(dv, device="cuda")
    for b in range(B):
        pay = torch.nn.functional.pad(a.payload[b * region:(b + 1) * region], (0, 4)).long()
        off = a.head_off[b * H:(b + 1) * H].long()
        if cfg.unit_kind == qs.UNIT_ROW:
            w = a.widths[b * H * dk:(b + 1) * H * dk].long().view(H, dk)
            scale = a.scales[b * H * dk:(b + 1) * H * dk].view(torch.float16).double().view(H, dk, 1)
        else:
            w = a.widths[b * H:(b + 1) * H].long().view(H, 1).expand(H, dk)
            g = H * (dk // 32) * dv
            scale = a.scales[b * g:(b + 1) * g].view(torch.float16).double().view(H, dk // 32, 1, dv)
            scale = scale.expand(H, dk // 32, 32, dv).reshape(H, dk, dv)
        start = off[:, None] + (w.cumsum(1) - w) * (dv // 8)
        bit = 8 * start[..., None] + j * w[..., None]
        at = torch.where(w[..., None] > 0, bit >> 3, 0)
        u = (pay[at] | (pay[at + 1] << 8) | (pay[at + 2] << 16)) >> (bit & 7) & ((1 << w[..., None]) - 1)
        n = torch.where(w >= 2, (1 << (w - 1).clamp(min=0)) - 1, 0)[..., None]
        x = torch.where(w[..., None] >= 2, (u - n).double(), 1.0 - 2.0 * u.double())
        S[b] = torch.where(w[..., None] > 0, x * scale, 0.0)
    return S


def recurrence(cfg, x, t0, t1, S):
    """S_t = (I - k a^T) D S + k (w o v)^T and o_t = S_t^T q_t, token by token in 64 bits."""
    o = []
    for t in range(t0, t1):
        q, k, v = (z[:, t].double() for z in (x.q, x.k, x.v))
        S = S * torch.exp(-rate_of(cfg, x, t)).reshape(S.shape[:2] + (-1, 1))
        if cfg.erase_kind == qs.ERASE_NONE:
            u = v
        else:
            general = cfg.erase_kind == qs.ERASE_GENERAL
            a = x.a[:, t].double() if general else x.beta[:, t].double()[..., None] * k
            wv = v * (x.w[:, t].double() if general else x.beta[:, t].double()[..., None])
            u = wv - torch.einsum("bhi,bhij->bhj", a, S)
        S = S + k[..., None] * u[..., None, :]
        o.append(torch.einsum("bhi,bhij->bhj", q, S))
    return torch.stack(o, 1), S


def rate_of(cfg, x, t):
    """Token t's rates, (B, H, dk) or (B, H), in 64 bits."""
    if x.s is not None:
        return x.s[:, t].double()
    L = 1 << cfg.gate_bits
    code = x.s_code[:, t].long()
    chan = torch.arange(code[0].numel(), device="cuda").view(code[0].shape)
    return x.s_lut[chan * L + code].double()


def averages(cfg, x, t0, t1, ms, mr):
    """The running averages of 1 - e^{-2s} and of the erasure term after tokens [t0, t1)."""
    alpha = 2.0 / (cfg.ema_span + 1.0)
    row = cfg.unit_kind == qs.UNIT_ROW
    for t in range(t0, t1):
        r, k = rate_of(cfg, x, t), x.k[:, t].double()
        if cfg.decay_kind == qs.DECAY_HEAD and row:
            r = r[..., None].expand(k.shape)
        xs = -torch.expm1(-2.0 * r)
        if cfg.erase_kind == qs.ERASE_DELTA:
            beta = x.beta[:, t].double()[..., None]
            xr = beta * (2.0 - beta) * k * k
        elif cfg.erase_kind == qs.ERASE_GENERAL:
            a = x.a[:, t].double()
            xr = 2.0 * a * k - a * a * (k * k).sum(-1, keepdim=True)
        else:
            xr = torch.zeros_like(k)
        xr = xr if row else xr.mean(-1)
        ms, mr = (xs, xr) if t == 0 else (ms + alpha * (xs - ms), mr + alpha * (xr - mr))
    return ms.reshape(-1), mr.reshape(-1)


def exact(case, seed):
    """Readouts, states and statistics in 64 bits where the inputs alone give them: over one
    write-back interval, whose readouts and ranges come before the state is rounded again."""
    s = prepare(case, seed)
    cfg, do = s["cfg"], s["do"]
    if do == "gate":
        L = 1 << cfg.gate_bits
        x = s["s"].flatten(0, 1).flatten(1)
        lo, hi = torch.log(x.amin(0).double()), torch.log(x.amax(0).double())
        step = ((hi - lo) / (L - 1))[:, None]
        lut = torch.exp(lo[:, None] + torch.arange(L, device="cuda").double() * step)
        thr = torch.exp(lo[:, None] + (torch.arange(1, L, device="cuda").double() - 0.5) * step)
        return dict(codes=None, lut=lut.reshape(-1), thr=thr.reshape(-1))
    if do == "pack":
        amax = s["S"].abs().amax(-1).double().reshape(-1)
        return dict(payload=None, scales=None, fidx=None, range=None if s["range"] is None else amax)
    if do == "unpack":
        return dict(S=unpacked(cfg, s["a"]))
    if do == "fp32":
        o, S = recurrence(cfg, s["x"], 0, s["T"], s["S"].double())
        return dict(S=S, o=o)
    t, st, row = s["t"], s["st"], cfg.unit_kind == qs.UNIT_ROW
    ms = st.ema_s.double().view((cfg.B, cfg.H) + ((cfg.dk,) if row else ()))
    ms, mr = averages(cfg, s["x"], t, t + s["n"], ms, st.ema_r.double().view(ms.shape))
    o = top = None
    if s["n"] <= cfg.C:
        if do == "prefill":
            S = torch.zeros((cfg.B, cfg.H, cfg.dk, cfg.dv), dtype=torch.float64, device="cuda")
        else:
            S = unpacked(cfg, s["a"])
        o, S = recurrence(cfg, s["x"], t, t + s["n"], S)
        top = S.abs().amax(-1).reshape(-1) if row else None
    return dict(o=o, payload=None, scales=None, widths=None, head_off=None, fidx=None, next_widths=None, ema_s=ms,
                ema_r=mr, range=top)
