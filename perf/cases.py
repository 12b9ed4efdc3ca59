"""The work that the KVM layer is used for, as cases to measure.

One pass of a case goes through the binding's public calls the way a serving or evaluation program does:
an optional prefill (whole, or in calls of `seg` tokens) followed by `steps` single-token decode steps.

  fresh     the pass starts an empty sequence (KVMState.reset); otherwise it goes on with the sequence that
            `prepare` left, `ctx` tokens long.  Those cases have a full fixed-size state, so every pass costs the same.
  host      the inputs and outputs are pinned host buffers (prefill_host, decode_step_host)
  d_model   not 0: the merge gates of the prefill come from the layer input through merge_gate
  qk_ln     LN_q / LN_k inside the layer (fused front end)
  affine    seeded LayerNorm parameters and per-head temperatures instead of 1, 0, 1, 1

Every prefill is followed by at least one decode step: its output depends on all rows of the state the prefill left.
"""
import math

import torch

from paper_2605_09877_b200 import kvm, synth

BASE = dict(B=1, Hq=1, Hkv=1, d=128, C=256, w=2, S=1, r=0, growth="sqrt", slots=0, coeff=16, num=1, den=2, half=0,
            fresh=True, ctx=0, T=0, seg=0, steps=1, kind="normal", host=False, d_model=0, qk_ln=False, affine=False)


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # a small layer with a short prompt and the first tokens of the answer: launches and latency count
        _case("short_prompt_one_head", d=64, C=64, growth="fixed", slots=64, T=1024, steps=8),
        # two sequences of 8192 tokens, fixed 512-row state, partial RoPE
        _case("two_sequences_fixed512", B=2, Hq=16, Hkv=16, C=128, r=32, growth="fixed", slots=512, T=8192, kind="scaled_keys"),
        # one sequence of 32768 tokens whose keys cluster (real keys do), square-root state
        _case("one_sequence_32k", Hq=32, Hkv=32, T=32768, kind="mixture"),
        # long-context retrieval: few heads, 131072 tokens, one in a hundred stands out
        _case("long_context_131k", Hq=8, Hkv=8, r=32, T=131072, kind="needles"),
        # the speed benchmark's shape with the square-root and with the fixed 256-row state
        _case("batch8_32k_sqrt", B=8, Hq=32, Hkv=32, T=32768),
        _case("batch8_32k_fixed256", B=8, Hq=32, Hkv=32, growth="fixed", slots=256, T=32768),
        # bulk prefill of many long sequences, fed in calls of 4096 tokens
        _case("bulk_16x65k", B=16, Hq=32, Hkv=32, T=65536, seg=4096),
        # a whole layer: gates from the layer input, LN_q / LN_k, RoPE, grouped queries, trained parameters;
        # prompts of odd length in odd pieces (chunked prefill), then a few tokens of the answer
        _case("ragged_gqa_front_end", B=3, Hq=32, Hkv=8, r=32, T=5003, seg=1777, steps=21, d_model=2048, qk_ln=True, affine=True),
        # a conversation: each turn brings 300 tokens and takes 64
        _case("chat_turn", Hq=32, Hkv=8, r=32, growth="fixed", slots=256, fresh=False, ctx=3000, T=300, steps=64),
        # generation with one sequence: one block of tokens (with its fold) from a 256-row state
        _case("generate_1x256", Hq=32, Hkv=32, growth="fixed", slots=256, fresh=False, ctx=2048, steps=256),
        # generation with a large batch: one block of tokens from 4096-row states
        _case("generate_64x256", B=64, Hq=32, Hkv=32, growth="fixed", slots=4096, fresh=False, ctx=5120, steps=256),
        # inputs and outputs in (pinned) host memory
        _case("host_buffers_8x4096", B=8, Hq=32, Hkv=32, T=4096, host=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = _weight(listed()[6])
    while True:
        op = rng.choice(["prefill"] * 6 + ["turn"] * 2 + ["generate"] * 3 + ["host"])
        group = rng.choice([1, 1, 1, 2, 4, 8])
        hkv = rng.choice([1, 2, 3, 4, 8, 8, 16, 32, 32])
        C = rng.choice([64, 128, 256, 256, 256, 8 * rng.randint(6, 32)])
        c = _case(B=_log(rng, 1, 64), Hq=hkv * group, Hkv=hkv, d=rng.choice([64, 128, 128]), C=C, w=rng.choice([2, 2, 2, 1, 3]),
                  S=rng.choice([1, 1, 1, 0, 4]), r=rng.choice([0, 0, 32, 64]), affine=rng.random() < 0.3,
                  kind=rng.choice(["normal", "normal", "scaled_keys", "mixture", "needles"]))
        if op in ("prefill", "host"):
            g = rng.choice(["sqrt", "sqrt", "sqrt", "fixed", "fixed", "power", "saturating"])
            c["growth"] = g
            if g == "fixed":
                c["slots"] = _log(rng, 64, 4096)
            elif g == "power":
                num = rng.choice([2, 2, 3])
                c.update(num=num, den=4, coeff=16 if num == 2 else 4)
            elif g == "saturating":
                c.update(slots=_log(rng, 512, 8192), half=_log(rng, 2000, 60000))
            c["T"] = _log(rng, 200, 131072) if op == "prefill" else _log(rng, 200, 16384)
            c["steps"] = rng.choice([1, 1, 4, 17])
            c["host"] = op == "host"
            if op == "prefill" and c["T"] > 1000 and rng.random() < 0.3:
                c["seg"] = rng.choice([1024, 4096, rng.randint(500, 5000)])
            if op == "prefill" and rng.random() < 0.25:
                c["qk_ln"] = True
                c["d_model"] = rng.choice([0, 1024, 2048, 4096])
                if c["d_model"] * c["B"] * c["T"] > 1 << 31:
                    c["d_model"] = 0
        else:
            c.update(growth="fixed", slots=max(C, _log(rng, 64, 4096)), fresh=False)
            c["ctx"] = c["slots"] + (c["w"] + 1) * C + rng.randint(0, C - 1)
            if op == "turn":
                c.update(T=_log(rng, 16, 1500), steps=rng.randint(8, 100))
            else:
                c.update(T=0, steps=C)
        if c["T"] // C > 768 or c["Hq"] > 64:
            continue
        if _weight(c) <= most and _memory(c) <= (30 << 30):
            return c


def _growth(c):
    return kvm.growth(c["growth"], c["slots"], c["coeff"], c["num"], c["den"], c["half"])


def _total(c):
    return c["ctx"] + c["T"] + c["steps"]


def _capacity(c):
    # a fixed state stays at its size however long the sequence gets
    return max(kvm.kvm_plan_capacity(c["C"], c["w"], _growth(c), _total(c)), c["C"], c["slots"] if not c["fresh"] else 0)


def _call_tokens(c):
    return max(min(c["seg"] or c["T"], c["T"]), min(c["ctx"], 1024), 1)


def _memory(c):
    U, d = c["B"] * c["Hkv"], c["d"]
    state = U * _capacity(c) * d * 20 + _call_tokens(c) * d * 2 * c["B"] * (c["Hq"] + 2 * c["Hkv"]) + U * c["C"] * (c["C"] * 8 + d * 24 + 2400)
    return state + c["B"] * (c["T"] + c["steps"]) * d * 2 * (2 * c["Hq"] + 2 * c["Hkv"]) + 2 * c["B"] * c["T"] * c["d_model"] + (2 << 30)


def _plan(c):
    """Per block of the pass: (first token, end, window begin, rows before, rows appended by the fold at its end or -1)."""
    C, w, g = c["C"], c["w"], _growth(c)
    pos, end = (0, c["T"]) if c["fresh"] else (c["ctx"], c["ctx"] + c["T"])
    m = kvm.kvm_plan_capacity(C, w, g, pos)
    out = []
    while pos < end:
        e = (pos // C + 1) * C
        stop = min(e, end)
        na = -1
        if stop == e and e >= w * C:
            m1 = c["slots"] if not c["fresh"] else kvm.kvm_plan_capacity(C, w, g, e)
            na = m1 - m
        out.append((pos, stop, max(0, e - w * C), m, na))
        m += max(na, 0)
        pos = stop
    return out, m


def work(case):
    """Inputs read once, outputs written once, and for a decode step the fp16 rows of state and window it attends over;
    flops of the attention (4 d per query and visible key) and of the routing (2 d per folded token and state row)."""
    c = dict(BASE, **case)
    B, Hq, Hkv, d, C = c["B"], c["Hq"], c["Hkv"], c["d"], c["C"]
    blocks, m = _plan(c)
    att = route = 0
    for p, q, b, rows, na in blocks:
        att += (q - p) * (rows + p - b) + (q - p) * (q - p + 1) // 2
        if na >= 0 and rows > 0:
            route += C * rows + (C - na) * na
    flops = 4 * d * att * B * Hq + 2 * d * route * B * Hkv
    nbytes = B * c["T"] * d * 2 * (2 * Hq + 2 * Hkv) + B * c["T"] * c["d_model"] * 2
    if c["d_model"]:
        flops += 2 * B * c["T"] * c["d_model"] * Hkv
    t0 = c["T"] if c["fresh"] else c["ctx"] + c["T"]
    for t in range(t0, t0 + c["steps"]):
        n = m + t + 1 - max(0, (t // C + 1) * C - c["w"] * C)
        nbytes += B * Hkv * n * d * 4 + B * d * 2 * (2 * Hq + 2 * Hkv)
        flops += 4 * d * n * B * Hq
    return dict(bytes=nbytes, flops=flops)


def _weight(c):
    w = work(c)
    return w["flops"] / 5e14 + w["bytes"] / 3e12


def tolerance(case):
    # measured between the tensor-core and the scalar-core attention (same operand precision, sums in another order,
    # bf16 outputs): 3.5e-4 to 8.5e-4 on the listed cases
    return {"rel": 3.4e-3}


def _rand(shape, gen):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)


def _values(c, n, gen):
    """q, k, v of n tokens: [B, heads, n, d] bf16, distributed like the workloads of synth.make_inputs."""
    B, Hq, Hkv, d = c["B"], c["Hq"], c["Hkv"], c["d"]
    q, k, v = _rand((B, Hq, n, d), gen), _rand((B, Hkv, n, d), gen), _rand((B, Hkv, n, d), gen)
    if c["kind"] == "scaled_keys":
        k.mul_(d ** -0.5)
    elif c["kind"] == "needles":
        pos = torch.randperm(n, generator=gen, device="cuda")[:max(1, int(n * synth.NEEDLE_FRACTION))]
        k[:, :, pos] *= synth.NEEDLE_SCALE
        v[:, :, pos] = torch.nn.functional.one_hot(pos % d, d).to(v.dtype) * synth.NEEDLE_SCALE
    elif c["kind"] == "mixture":
        ck, cv = _rand((synth.N_CENTROIDS, d), gen), _rand((synth.N_CENTROIDS, d), gen)
        for b in range(B):
            zk = torch.randint(0, synth.N_CENTROIDS, (Hkv, n), generator=gen, device="cuda")
            zq = torch.randint(0, synth.N_CENTROIDS, (Hq, n), generator=gen, device="cuda")
            q[b].mul_(synth.MIX_SIGMA).add_(ck[zq])
            k[b].mul_(synth.MIX_SIGMA).add_(ck[zk])
            v[b].mul_(synth.MIX_SIGMA).add_(cv[zk])
    return q, k, v


def _host(t):
    return None if t is None else torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def _params(c, seed):
    """Layer parameters (or None for 1, 0, 1, 1) and the LN_q / LN_k dictionary of a case."""
    par, ln = dict(ln_w=None, ln_b=None, tau_s=None, tau_b=None), None
    if c["affine"]:
        par = synth.make_layer_params(synth.Workload("params", c["B"], c["Hq"], c["Hkv"], c["d"], 1, c["C"], "sqrt", seed=seed), trivial=False)
    if c["qk_ln"]:
        h = torch.Generator().manual_seed(seed + 1)
        ln = dict(eps=1e-5)
        for n, heads in (("q", c["Hq"]), ("k", c["Hkv"])):
            ln[n + "_weight"] = 1.0 + 0.2 * torch.randn((heads, c["d"]), generator=h)
            ln[n + "_bias"] = 0.1 * torch.randn((heads, c["d"]), generator=h)
    return par, ln


def _inputs(c, seed, context):
    """The tensors of a pass, in the order they are drawn; `context(q, k, v)` takes each call of the tokens before it."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    at, s = 0, {"x": None}
    while at < c["ctx"]:
        n = min(_call_tokens(c), c["ctx"] - at)
        context(*_values(c, n, gen))
        at += n
    if c["T"]:
        s["q"], s["k"], s["v"] = _values(c, c["T"], gen)
        if c["d_model"]:
            s["x"] = _rand((c["B"], c["T"], c["d_model"]), gen)
            s["w_gate"] = torch.randn((c["Hkv"], c["d_model"]), generator=gen, device="cuda") / math.sqrt(c["d_model"])
    # one token per step: [step][B, heads, d], every step's tensors contiguous
    s["tq"], s["tk"], s["tv"] = (list(t.permute(2, 0, 1, 3).contiguous()) for t in _values(c, c["steps"], gen))
    return s


def prepare(case, seed):
    c = dict(BASE, **case)
    torch.cuda.empty_cache()   # the layer allocates its state outside torch's pool
    par, ln = _params(c, seed)
    layer = kvm.KVMState(
        kvm.LayerConfig(batch=c["B"], n_q_heads=c["Hq"], n_kv_heads=c["Hkv"], head_dim=c["d"], max_block=c["C"],
                        max_state_slots=_capacity(c), max_call_tokens=_call_tokens(c), n_bswa_chunks=c["w"], sink_len=c["S"]),
        ln_weight=par["ln_w"], ln_bias=par["ln_b"], tau_state=par["tau_s"], tau_bswa=par["tau_b"], qk_ln=ln)
    s = _inputs(c, seed, lambda q, k, v: layer.prefill(q, k, v, c["C"], _growth(c), c["r"]))
    s.update(c=c, layer=layer, growth=_growth(c))
    if c["T"]:
        s["out"] = torch.empty_like(s["q"])
    s["tout"] = torch.empty((c["steps"], c["B"], c["Hq"], c["d"]), dtype=torch.bfloat16, device="cuda")
    if c["host"]:
        for n in ("q", "k", "v", "out", "tout"):
            s[n] = _host(s[n])
        for n in ("tq", "tk", "tv"):
            s[n] = [_host(t) for t in s[n]]
    return s


def run(s):
    c, layer, g = s["c"], s["layer"], s["growth"]
    if c["fresh"]:
        layer.reset()
    res = {}
    if c["T"]:
        q, k, v, out, gate = s["q"], s["k"], s["v"], s["out"], None
        if c["host"]:
            layer.prefill_host(q, k, v, c["C"], g, c["r"], out)
        else:
            if s["x"] is not None:
                gate = res["gate"] = kvm.merge_gate(s["x"], s["w_gate"])
            seg = c["seg"] or c["T"]
            for a in range(0, c["T"], seg):
                z = min(c["T"], a + seg)
                layer.prefill(q[:, :, a:z], k[:, :, a:z], v[:, :, a:z], c["C"], g, c["r"], out=out[:, :, a:z],
                              gate=None if gate is None else gate[:, :, a:z].contiguous())
        res["out"] = out
    step = layer.decode_step_host if c["host"] else layer.decode_step
    for i in range(c["steps"]):
        step(s["tq"][i], s["tk"][i], s["tv"][i], out=s["tout"][i])
    res["tokens"] = s["tout"]
    return res


def _budget(c, e):
    if c["growth"] == "fixed":
        return c["slots"]
    if c["growth"] == "saturating":
        return c["slots"] * e // (e + c["half"])
    num, den = (1, 2) if c["growth"] == "sqrt" else (c["num"], c["den"])
    most = c["coeff"] ** den * e ** num
    n = int(round(most ** (1.0 / den)))
    while n ** den > most:
        n -= 1
    while (n + 1) ** den <= most:
        n += 1
    return n


def _norm(x, w, b, eps):
    """LayerNorm over the channels; w, b [heads, 1, d]."""
    x = x - x.mean(-1, keepdim=True)
    return x / (x.square().mean(-1, keepdim=True) + eps).sqrt() * w + b


def _exact_sequence(c, q, k, v, g, w, b, ts, tb, first, out):
    """One batch element in 64 bits: q [Hkv, G, N, d], k, v [Hkv, N, d], g [Hkv, N] -> out [Hkv, G, N - first, d]."""
    C, L, r, d, N, H = c["C"], c["w"] * c["C"], c["r"], c["d"], k.shape[1], k.shape[0]
    G = q.shape[1]
    half = r // 2
    freq = 10000.0 ** (-torch.arange(half, dtype=torch.float64, device="cuda") / max(half, 1))

    def rope(x, t0):
        if not r:
            return x
        a = torch.arange(t0, t0 + x.shape[-2], dtype=torch.float64, device="cuda")[:, None] * freq
        lo, hi = x[..., :half], x[..., half:r]
        return torch.cat([lo * a.cos() - hi * a.sin(), lo * a.sin() + hi * a.cos(), x[..., r:]], -1)

    K = V = torch.zeros((H, 0, d), dtype=torch.float64, device="cuda")
    rho = torch.zeros((H, 0), dtype=torch.float64, device="cuda")
    m = 0
    for s in range(0, N, C):
        e, z = s + C, min(s + C, N)
        b0 = max(0, e - L)
        kn = _norm(K, w, b, 1e-5)
        if z > first:
            a0 = max(s, first)
            kw, vw = rope(k[:, b0:z].double(), b0), v[:, b0:z].double()
            kr = V * (rho / V.norm(dim=-1).clamp_min(1e-12))[..., None]
            qq = rope(q[:, :, a0:z].double(), a0)
            ls = torch.matmul(qq, kn[:, None].mT) * (ts / math.sqrt(d))
            lw = torch.matmul(qq, kw[:, None].mT) * (tb / math.sqrt(d))
            later = torch.arange(b0, z, device="cuda")[None, :] > torch.arange(a0, z, device="cuda")[:, None]
            lw.masked_fill_(later, -math.inf)
            p = torch.softmax(torch.cat([ls, lw], -1), -1)
            out[:, :, a0 - first:z - first] = torch.matmul(p, torch.cat([kr, vw], 1)[:, None])
        if z < e or e < L:
            continue
        kb, vb, gb = k[:, b0:b0 + C].double().clone(), v[:, b0:b0 + C].double(), g[:, b0:b0 + C]
        kb[..., :r] = 0.0
        kb = _norm(kb, w, b, 1e-5)
        na = C if m == 0 else min(max(m, min(_budget(c, e), m + C)) - m, C)
        if na == C:
            new = torch.arange(C, device="cuda").expand(H, C)
        else:
            sim = torch.matmul(kb, kn.mT)
            new = sim.max(-1).values.sort(dim=-1, stable=True).indices[..., :na].sort(dim=-1).values
        at = new[..., None].expand(-1, -1, d)
        kc, vc = kb.gather(1, at), vb.gather(1, at)
        K, V, rho = torch.cat([K, kc], 1), torch.cat([V, vc], 1), torch.cat([rho, vc.norm(dim=-1)], 1)
        if na < C:
            sim = torch.cat([sim, torch.matmul(kb, _norm(kc, w, b, 1e-5).mT)], -1)
            sim[..., :c["S"]] = -math.inf
            to = sim.argmax(-1)[..., None].expand(-1, -1, d)
            gm = gb.scatter(1, new, 0.0)[..., None]
            K.scatter_add_(1, to, kb * gm)
            V.scatter_add_(1, to, vb * gm)
        m += na


def exact(case, seed):
    """The layer by its definition in 64 bits.  LN_q / LN_k give bf16 tensors (as the stand-alone call does)."""
    c = dict(BASE, **case)
    if work(c)["flops"] > 2e13 or c["B"] * c["Hq"] * _total(c) * c["d"] > 1 << 31:
        return None
    B, Hq, Hkv, d = c["B"], c["Hq"], c["Hkv"], c["d"]
    G = Hq // Hkv
    par, ln = _params(c, seed)
    parts = []
    s = _inputs(c, seed, lambda *t: parts.append(t))
    if c["T"]:
        parts.append((s["q"], s["k"], s["v"]))
    parts.append(tuple(torch.stack(s[n], 2) for n in ("tq", "tk", "tv")))
    first = c["ctx"]

    def dev(a, shape, default):
        return torch.full(shape, default, dtype=torch.float64, device="cuda") if a is None else torch.as_tensor(a).to("cuda").double().reshape(shape)

    w, b = dev(par["ln_w"], (Hkv, 1, d), 1.0), dev(par["ln_b"], (Hkv, 1, d), 0.0)
    ts, tb = dev(par["tau_s"], (Hkv, G, 1, 1), 1.0), dev(par["tau_b"], (Hkv, G, 1, 1), 1.0)
    out = torch.empty((B, Hkv, G, _total(c) - first, d), dtype=torch.float64, device="cuda")
    gates = torch.ones((B, Hkv, _total(c)), dtype=torch.float64, device="cuda")
    if s["x"] is not None:
        for i in range(B):
            z = s["x"][i].double() @ s["w_gate"].double().T
            gates[i, :, first:first + c["T"]] = (1.0 + torch.where(z > 0, z, torch.expm1(z))).T
    for i in range(B):
        q, k, v = (torch.cat([t[n][i] for t in parts], 1) for n in range(3))
        if ln:
            q, k = (_norm(x.double(), ln[n + "_weight"].cuda().double()[:, None], ln[n + "_bias"].cuda().double()[:, None], ln["eps"]).bfloat16()
                    for n, x in (("q", q), ("k", k)))
        _exact_sequence(c, q.reshape(Hkv, G, -1, d), k, v, gates[i], w, b, ts, tb, first, out[i])
    out = out.reshape(B, Hq, -1, d)
    res = {"tokens": out[:, :, c["T"]:].permute(2, 0, 1, 3)}
    if c["T"]:
        res["out"] = out[:, :, :c["T"]]
    if s["x"] is not None:
        res["gate"] = gates[:, :, first:first + c["T"]]
    return res
