"""The calls whose speed matters to a user of the library, as measurable cases.

A program that serves a model with this library prefills prompts, runs
draft-verify-commit steps, trains the drafter every few steps, sometimes
decodes greedily for comparison, and may use the projection on its own.  The
listed cases are those calls at the sizes of the repository's workloads (a
tiny f32 decoder, a 1B-shaped GQA decoder, a 7B-shaped decoder, batch 1 and a
ragged batch of 8, contexts from 32 to 16384 tokens); draw() spreads more of
them over the same ranges, with odd and ragged sizes.

Weights are seeded N(0, 0.02) draws made on the GPU (the upper half's output
projections scaled by 0.3).  As in a trained model, the head is fairly sure of
its next token: each token's head row leans towards the embedding of the token
before it, by about nine standard deviations of the other logits, and the
drafter disagrees with the verifier after three tokens in ten.  Prompts follow
a Zipf(1.1) law over the vocabulary.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2510_05421_gb300 import DVIEngine, DeviceWeights
from paper_2510_05421_gb300.dvi import linear_noalloc

DEV = "cuda"

# d_model, heads, KV heads, head_dim, d_ffn, vocabulary
SHAPES = {
    "tiny": (256, 4, 4, 64, 688, 1024),
    "small": (512, 4, 2, 128, 1408, 4000),
    "mid": (1024, 16, 4, 64, 2816, 32000),
    "1b": (2048, 16, 8, 128, 5632, 32000),
    "7b": (4096, 32, 32, 128, 11008, 32000),
}


def _case(kind, shape, layers, split, **kw):
    c = dict(kind=kind, shape=shape, layers=layers, split=split, dtype="bf16", batch=1, k_spec=5, rank=16,
             update_every=4, prompt_lo=512, prompt_hi=512, gen=32, bonus=0, head_mode=0, objective="dvi")
    c.update(kw)
    return c


def _named(name, c):
    return dict(c, name=name)


def listed():
    return [
        # one projection on its own, the smallest call: a single token row through a square weight
        _named("linear_4096_m1", dict(kind="linear", dtype="bf16", n_out=4096, k_in=4096, rows=1)),
        # the tiny f32 decoder end to end, host prompt to host tokens, KL update every 8 steps: launches and
        # latency count
        _named("tiny_f32_generate", _case("generate", "tiny", 4, 2, dtype="f32", k_spec=4, rank=8, update_every=8,
                                          prompt_lo=32, prompt_hi=32, gen=64, objective="kl")),
        # one chat-sized request on a 1B-shaped GQA decoder: 512-token prompt, 32 tokens out with the drafter
        # training every 4 steps, host to host
        _named("1b_generate", _case("generate", "1b", 16, 8)),
        # the greedy baseline of the same decoder (short prompt, 32 tokens)
        _named("1b_greedy", _case("greedy", "1b", 16, 8, prompt_lo=64, prompt_hi=64)),
        # steady-state serving of a 7B-shaped decoder at batch 1: four decode steps and a drafter update
        _named("7b_round", _case("round", "7b", 32, 2, prompt_lo=1024, prompt_hi=1024)),
        # the same with 8 sequences of ragged length in one batch
        _named("7b_batch8_round", _case("round", "7b", 32, 2, batch=8, prompt_lo=157, prompt_hi=1724)),
        # long context: 16384 cached positions, 8 drafted tokens
        _named("7b_16k_round", _case("round", "7b", 32, 2, k_spec=8, prompt_lo=16384, prompt_hi=16384)),
        # training the whole drafter head W^S instead of LoRA factors
        _named("full_head_round", _case("round", "1b", 8, 4, head_mode=1, prompt_lo=200, prompt_hi=200)),
        # prompts alone (time to first token): ordinary, large model, several short ragged ones, one long one
        _named("prefill_1b_512", _case("prefill", "1b", 16, 8)),
        _named("prefill_7b_1024", _case("prefill", "7b", 32, 2, prompt_lo=1024, prompt_hi=1024)),
        _named("prefill_1b_ragged8", _case("prefill", "1b", 16, 8, batch=8, prompt_lo=23, prompt_hi=301)),
        _named("prefill_16k", _case("prefill", "7b", 2, 1, prompt_lo=16384, prompt_hi=16384)),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    most = max(_seconds(c) for c in listed())
    while True:
        c = _draw(rng)
        if _seconds(c) <= 0.7 * most:
            return c


def _draw(rng):
    kind = rng.choice(["linear", "generate", "greedy", "round", "round", "prefill", "prefill"])
    if kind == "linear":
        if rng.random() < 0.25:   # the f32 projection's fixed scratch takes few rows
            return dict(kind=kind, dtype="f32", n_out=_log_int(rng, 100, 4096), k_in=8 * _log_int(rng, 8, 512),
                        rows=_log_int(rng, 1, 16))
        return dict(kind=kind, dtype="bf16", n_out=_log_int(rng, 100, 32000), k_in=8 * _log_int(rng, 8, 1376),
                    rows=_log_int(rng, 1, 256))
    f32 = rng.random() < 0.15
    shape = rng.choice(["tiny", "small"] if f32 else ["small", "mid", "1b", "1b", "7b", "7b"])
    layers = _log_int(rng, 2, 6 if f32 else (8 if shape == "7b" else 16))
    split = rng.randint(1, max(1, layers // 2))
    batch = rng.choice([1, 1, 1, 2, 3, 5, 8])
    longest = 512 if f32 else (8192 if kind == "prefill" and batch == 1 else 2048)
    hi = _log_int(rng, 16, longest)
    c = _case(kind, shape, layers, split, dtype="f32" if f32 else "bf16", batch=batch,
              k_spec=rng.randint(1, 8), rank=rng.choice([8, 16]), prompt_lo=max(1, int(hi * rng.uniform(0.3, 1.0))),
              prompt_hi=hi, gen=rng.randint(4, 24), bonus=int(rng.random() < 0.2),
              head_mode=int(kind == "round" and rng.random() < 0.15))
    c["update_every"] = rng.randint(1, max(1, min(6, 256 // (batch * c["k_spec"]))))
    return c


# ---------------------------------------------------------------- sizes


def _dims(c):
    d, hq, hkv, hd, f, v = SHAPES[c["shape"]]
    return SimpleNamespace(d=d, hq=hq, hkv=hkv, hd=hd, f=f, v=v, L=c["layers"], k=c["split"], B=c["batch"],
                           K=c["k_spec"], Kv=c["k_spec"] + c["bonus"], r=c["rank"], esz=4 if c["dtype"] == "f32" else 2)


def _lens(c):
    """Prompt lengths of the batch: spread evenly over the range, the longest first."""
    lo, hi, B = c["prompt_lo"], c["prompt_hi"], c["batch"]
    return [hi - (hi - lo) * b // max(1, B - 1) for b in range(B)]


def _room(c):
    """Tokens a context has room for after its prompt."""
    if c["kind"] == "round":
        return 2048
    return c["gen"] * (c["k_spec"] + 1) + c["k_spec"] + 8


def _layer_params(s):
    return s.d * s.hd * (2 * s.hq + 2 * s.hkv) + 3 * s.d * s.f


def _prefill_work(s, lens):
    kv_row = 2 * s.hkv * s.hd * s.esz
    by = fl = 0
    for n in lens:
        by += s.L * _layer_params(s) * s.esz + s.v * s.d * s.esz + s.L * n * kv_row + n * s.d * s.esz
        fl += 2 * s.L * _layer_params(s) * n + s.L * 2 * n * (n + 1) * s.hq * s.hd + 2 * s.v * s.d
    return by, fl


def _steps_work(s, lens, steps):
    """Draft passes (k layers and a head each), then the verify pass: weights once a pass, attended K/V rows once."""
    kv_row = 2 * s.hkv * s.hd * s.esz
    rows = sum(lens)
    head = s.v * s.d * s.esz
    by = s.Kv * s.k * _layer_params(s) * s.esz + s.K * head + (s.L - s.k) * _layer_params(s) * s.esz + head
    by += (s.Kv * s.k + s.L - s.k) * rows * kv_row + 2 * s.B * s.K * s.v * 4
    fl = 2 * s.B * (s.Kv * s.L * _layer_params(s) + (s.K + s.Kv) * s.v * s.d)
    fl += 4 * s.Kv * s.L * rows * s.hq * s.hd
    return steps * by, steps * fl


def _update_work(c, s, updates):
    n = s.B * s.K * c["update_every"]
    if c["head_mode"]:
        vd = s.v * s.d
        by = n * (2 * s.v * 4 + s.d * s.esz) + vd * (24 + (2 if s.esz == 2 else 0) + 2 * s.esz)
        fl = 4 * n * vd
    else:
        by = n * (2 * s.v * 4 + s.d * s.esz) + (s.v + s.d) * s.r * 4 * 7
        fl = 6 * n * s.r * (s.v + s.d) + 20 * n * s.v
    return updates * by, updates * fl


def _add(*pairs):
    return {"bytes": float(sum(p[0] for p in pairs)), "flops": float(sum(p[1] for p in pairs))}


def work(case):
    c = case
    if c["kind"] == "linear":
        n, k, m = c["n_out"], c["k_in"], c["rows"]
        return {"bytes": float(n * k * (2 if c["dtype"] == "bf16" else 4) + 4 * m * (n + k)), "flops": 2.0 * n * k * m}
    s, lens = _dims(c), _lens(c)
    if c["kind"] == "prefill":
        return _add(_prefill_work(s, lens))
    if c["kind"] == "greedy":
        kv = 2 * s.hkv * s.hd * s.esz
        n = c["gen"] - 1
        step = (s.L * _layer_params(s) * s.esz + s.v * s.d * s.esz + s.L * sum(lens) * kv,
                2 * s.B * (s.L * _layer_params(s) + s.v * s.d) + 4 * s.L * sum(lens) * s.hq * s.hd)
        return _add(_prefill_work(s, lens), (n * step[0], n * step[1]))
    if c["kind"] == "round":
        return _add(_steps_work(s, lens, c["update_every"]), _update_work(c, s, 1))
    steps = math.ceil((c["gen"] - 1) / s.Kv)   # the fewest: every draft accepted
    return _add(_prefill_work(s, lens), _steps_work(s, lens, steps), _update_work(c, s, steps // c["update_every"]))


def _seconds(c):
    w = work(c)
    f32 = c["dtype"] == "f32"
    return w["bytes"] / (1.5e12 if f32 else 3e12) + w["flops"] / (5e12 if f32 else 5e14)


# ---------------------------------------------------------------- inputs


def _shape(c):
    s = _dims(c)
    return SimpleNamespace(n_layers=s.L, d_model=s.d, n_heads=s.hq, n_kv_heads=s.hkv, head_dim=s.hd, d_ffn=s.f,
                           vocab=s.v, rms_eps=1e-5, rope_theta=10000.0)


def _hyper(c):
    return SimpleNamespace(objective=c["objective"], lr=1e-3, beta1=0.9, beta2=0.999, adam_eps=1e-8,
                           optimizer="adam", tau=1.0, lambda0=1.0, lambda_kl_min=0.1, lambda_pg_max=1.0, t_warmup=32,
                           t_ramp=32, w_ce=0.0, w_ent=0.0, w_rl_max=0.1, beta0=0.1, beta_min=0.01, t_beta=100.0,
                           baseline_rho=0.9)


def _weights(c, g):
    s = _dims(c)
    td = torch.float32 if c["dtype"] == "f32" else torch.bfloat16

    def mat(rows, cols, std=0.02):
        return torch.empty(rows, cols, dtype=td, device=DEV).normal_(0.0, std, generator=g)

    def gain():
        return 1.0 + 0.05 * torch.randn(s.d, device=DEV, generator=g)

    layers = []
    for l in range(s.L):
        out = 0.02 * (0.3 if l >= s.L // 2 else 1.0)
        layers.append(dict(attn_norm=gain(), wq=mat(s.hq * s.hd, s.d), wk=mat(s.hkv * s.hd, s.d),
                           wv=mat(s.hkv * s.hd, s.d), wo=mat(s.d, s.hq * s.hd, out), ffn_norm=gain(),
                           w_gate=mat(s.f, s.d), w_up=mat(s.f, s.d), w_down=mat(s.d, s.f, out)))
    # the residual stream keeps the embedding in sight: about as large as what the layers add to it
    size = 0.022 * math.sqrt(s.f * s.L)
    embed, lm = mat(s.v, s.d, size), mat(s.v, s.d)
    after = torch.randperm(s.v, device=DEV, generator=g)   # the likely next token of each
    lm[after] += (embed.float() * (0.18 / math.sqrt(s.d) / size)).to(td)
    draft = lm.clone()
    differ = after[torch.randperm(s.v, device=DEV, generator=g)[:3 * s.v // 10]]
    draft[differ] = lm[differ.roll(1)]
    return DeviceWeights(embed=embed, layers=layers, final_norm=gain(), lm_head=lm, draft_head=draft,
                         lora_a=0.01 * torch.randn(s.v, s.r, device=DEV, generator=g),
                         lora_b=0.02 * torch.randn(s.r, s.d, device=DEV, generator=g))


def _prompts(c, g):
    """Zipf(1.1) ids, one int32 tensor per sequence."""
    s = _dims(c)
    cdf = torch.cumsum(torch.arange(1, s.v + 1, dtype=torch.float64, device=DEV) ** -1.1, 0)
    cdf /= cdf[-1].clone()
    out = []
    for n in _lens(c):
        u = torch.rand(n, dtype=torch.float64, device=DEV, generator=g)
        out.append(torch.searchsorted(cdf, u).clamp_(max=s.v - 1).to(torch.int32))
    return out


def _inputs(c, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return _weights(c, g), _prompts(c, g)


def _linear_inputs(c, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    td = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    w = torch.empty(c["n_out"], c["k_in"], dtype=td, device=DEV).normal_(0.0, 0.02, generator=g)
    return w, torch.randn(c["rows"], c["k_in"], device=DEV, generator=g)


def prepare(case, seed):
    c = case
    if c["kind"] == "linear":
        w, x = _linear_inputs(c, seed)
        return SimpleNamespace(kind="linear", w=w, x=x, y=torch.empty(c["rows"], c["n_out"], device=DEV))
    s = _dims(c)
    weights, prompts = _inputs(c, seed)
    eng = DVIEngine(_shape(c), c["dtype"], weights, batch=s.B, k_spec=s.K, split_k=s.k, lora_rank=s.r,
                    max_seq_len=max(_lens(c)) + _room(c), log_steps=c["update_every"], head_mode=c["head_mode"],
                    bonus=bool(c["bonus"]))
    st = SimpleNamespace(kind=c["kind"], eng=eng, weights=weights, prompts=prompts, hyper=_hyper(c),
                         gen=c["gen"], every=c["update_every"], used=0, room=_room(c),
                         need=c["update_every"] * s.Kv + s.Kv + 1)
    cache_t = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    if c["kind"] in ("generate", "greedy"):
        st.host_prompts = [p.cpu().numpy() for p in prompts]
    st.out = {"k": eng.buffer("K_CACHE", cache_t), "v": eng.buffer("V_CACHE", cache_t)}
    if c["kind"] in ("generate", "round"):
        st.out["logits"] = eng.buffer("LOG_LOGITS", torch.float32)
        if c["head_mode"]:
            st.out["w_s"] = weights.draft_head
        else:
            st.out["z"] = eng.buffer("Z", torch.float32)
            st.out["grad_a"] = eng.buffer("GRAD_A", torch.float32)
            st.out["grad_b"] = eng.buffer("GRAD_B", torch.float32)
    if c["kind"] == "round":
        for b, p in enumerate(prompts):
            eng.prefill(b, p)
    return st


def run(state):
    st = state
    if st.kind == "linear":
        linear_noalloc(st.w, st.x, st.y)
        return st.y
    eng = st.eng
    if st.kind == "prefill":
        for b, p in enumerate(st.prompts):
            first = eng.prefill(b, p)
        return {"first": first, **st.out}
    if st.kind == "greedy":
        return {"tokens": eng.generate_ar(st.host_prompts, st.gen), **st.out}
    if st.kind == "generate":
        tokens, _, _, _ = eng.generate(st.host_prompts, st.gen, update_every=st.every, hyper=st.hyper)
        return {"tokens": np.array(tokens, dtype=np.int32), **st.out}
    # a round of steady-state decoding; a request that has filled its context makes room for the next one
    if st.used + st.need > st.room:
        for b, p in enumerate(st.prompts):
            eng.prefill(b, p)
        st.used = 0
    for _ in range(st.every):
        ids, committed, accepted = eng.step()
    st.used += st.every * eng.Kv
    eng.update(st.hyper)
    return {"ids": ids, "committed": committed, "accepted": accepted, **st.out}


# ---------------------------------------------------------------- tolerances


def tolerance(case):
    """About four times what the path is measured to differ from exact() by.

    linear: f32 sums of products of bf16 weights and hi + lo inputs (2.5e-6), or of f32 values (1.4e-7).  bf16 models:
    K/V entries are stored in bf16, and a last-bit difference before that rounding moves an entry by a whole bf16
    step, which the layers above carry on: 1e-4 to 4.5e-4 up to 16 layers, 6.5e-4 at 32; logits and gradients sit
    behind those caches.  f32 models carry f32 sums throughout (7e-7).  Tokens are whole values that only ties could
    change."""
    c = case
    if c["kind"] == "linear":
        return {"rel": 1e-5 if c["dtype"] == "bf16" else 1e-6}
    if c["dtype"] == "f32":
        return {"rel": 1e-5, "differ": 0.01}
    return {"rel": 2e-3 if c["layers"] <= 16 else 3e-3, "differ": 0.01}


# ---------------------------------------------------------------- in 64 bits


class _Ref:
    """The decoder and its drafter in float64, with K/V rows rounded to bf16 where the cache stores bf16."""

    def __init__(self, c, seed):
        self.c, self.s = c, _dims(c)
        self.w, self.prompts = _inputs(c, seed)
        s = self.s
        self.max_len = max(_lens(c)) + _room(c)
        self.bf16 = c["dtype"] != "f32"
        self.kv = [[torch.zeros(2, s.hkv, self.max_len, s.hd, dtype=torch.float64, device=DEV)
                    for _ in range(s.L)] for _ in range(s.B)]
        half = s.hd // 2
        inv = 10000.0 ** (-2.0 * torch.arange(half, dtype=torch.float64, device=DEV) / s.hd)
        ang = torch.arange(self.max_len, dtype=torch.float64, device=DEV)[:, None] * inv[None, :]
        self.cos, self.sin = ang.cos(), ang.sin()
        self.a, self.b = self.w.lora_a.double(), self.w.lora_b.double()

    def norm(self, x, g):
        return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + 1e-5) * g.double()

    def rope(self, x, pos):
        half = self.s.hd // 2
        c, s = self.cos[pos][:, None, :], self.sin[pos][:, None, :]
        a, b = x[..., :half], x[..., half:]
        return torch.cat([a * c - b * s, b * c + a * s], -1)

    def layer(self, l, seq, x, p0):
        s, w = self.s, self.w.layers[l]
        n = x.shape[0]
        pos = torch.arange(p0, p0 + n, device=DEV)
        h = self.norm(x, w["attn_norm"])
        q = self.rope((h @ w["wq"].double().T).view(n, s.hq, s.hd), pos)
        k = self.rope((h @ w["wk"].double().T).view(n, s.hkv, s.hd), pos)
        v = (h @ w["wv"].double().T).view(n, s.hkv, s.hd)
        if self.bf16:
            k, v = k.to(torch.bfloat16).double(), v.to(torch.bfloat16).double()
        kv = self.kv[seq][l]
        kv[0, :, p0:p0 + n] = k.transpose(0, 1)
        kv[1, :, p0:p0 + n] = v.transpose(0, 1)
        grp = s.hq // s.hkv
        o = torch.empty(n, s.hq, s.hd, dtype=torch.float64, device=DEV)
        for r0 in range(0, n, 512):
            r1 = min(n, r0 + 512)
            t = p0 + r1
            qq = q[r0:r1].view(r1 - r0, s.hkv, grp, s.hd).permute(1, 2, 0, 3).reshape(s.hkv, -1, s.hd)
            sc = (qq @ kv[0, :, :t].transpose(1, 2)).view(s.hkv, grp, r1 - r0, t) / math.sqrt(s.hd)
            sc.masked_fill_(torch.arange(t, device=DEV)[None, :] > pos[r0:r1, None], -math.inf)
            oo = torch.softmax(sc, -1).view(s.hkv, -1, t) @ kv[1, :, :t]
            o[r0:r1] = oo.view(s.hkv, grp, r1 - r0, s.hd).permute(2, 0, 1, 3).reshape(r1 - r0, s.hq, s.hd)
        x = x + o.reshape(n, -1) @ w["wo"].double().T
        h = self.norm(x, w["ffn_norm"])
        h = torch.nn.functional.silu(h @ w["w_gate"].double().T) * (h @ w["w_up"].double().T)
        return x + h @ w["w_down"].double().T

    def layers(self, lo, hi, seq, x, p0):
        for l in range(lo, hi):
            x = self.layer(l, seq, x, p0)
        return x

    def embed(self, ids):
        return self.w.embed[torch.as_tensor(ids, device=DEV).long()].double()

    def logits(self, x):
        return self.norm(x, self.w.final_norm) @ self.w.lm_head.double().T

    def prefill(self, seq):
        p = self.prompts[seq]
        x = self.layers(0, self.s.L, seq, self.embed(p), 0)
        return int(self.logits(x[-1:])[0].argmax())

    def step(self, seq, n, pending):
        """One draft-verify-commit step: (committed, accepted, u, z, logits of the drafted positions)."""
        s = self.s
        toks, hk, us, zs = [pending], [], [], []
        for j in range(s.Kv):
            x = self.layers(0, s.k, seq, self.embed([toks[j]]), n + j)
            hk.append(x)
            if j < s.K:
                u = self.norm(x, self.w.final_norm)
                z = u @ self.w.draft_head.double().T + (u @ self.b.T) @ self.a.T
                us.append(u[0])
                zs.append(z[0])
                toks.append(int(z[0].argmax()))
        lg = self.logits(self.layers(s.k, s.L, seq, torch.cat(hk), n))
        best = [int(i) for i in lg.argmax(-1)]
        m = 0
        while m < s.K and toks[m + 1] == best[m]:
            m += 1
        got = toks[1:m + 1] + ([best[m]] if m < s.Kv else [])
        return got, m, us, zs, [lg[i] for i in range(s.K)]

    def decode(self, every, steps, gen):
        """Steps of the whole batch (`steps` of them, or until every sequence has `gen` tokens) with an update of
        the drafter after every `every`; what the caches, the replay buffer and the gradients then hold."""
        s, c = self.s, self.c
        n, count = _lens(c), [1] * self.s.B
        pend = [self.prefill(b) for b in range(s.B)]
        cap = every * s.B * s.K
        lg = torch.zeros(cap, s.v, dtype=torch.float64, device=DEV)
        z = torch.zeros_like(lg)
        u = torch.zeros(cap, s.d, dtype=torch.float64, device=DEV)
        out, logged, t = {}, [], 0
        mom = {}
        i = 0
        while i < steps if steps else min(count) < gen:
            for b in range(s.B):
                got, m, us, zs, ls = self.step(b, n[b], pend[b])
                base = ((i % every) * s.B + b) * s.K
                for j in range(s.K):
                    lg[base + j], z[base + j], u[base + j] = ls[j], zs[j], us[j]
                logged += [base + j for j in range(min(m + 1, s.K))]
                n[b] += len(got)
                count[b] += len(got)
                pend[b] = got[-1]
            i += 1
            if i % every == 0:
                rows = torch.tensor(logged, device=DEV)
                lp, lq = torch.log_softmax(z[rows], -1), torch.log_softmax(lg[rows], -1)
                p = lp.exp()
                G = p * (lp - lq - (p * (lp - lq)).sum(-1, keepdim=True)) / len(logged)
                U = u[rows]
                t += 1
                if c["head_mode"]:
                    if "w" not in mom:
                        mom["w"] = self.w.draft_head.double()
                    mom["w"] = self._adam("w", mom, mom["w"], G.T @ U, t)
                    self.w.draft_head.copy_(mom["w"])
                    out["w_s"] = self.w.draft_head.double()
                else:
                    out["grad_a"] = G.T @ (U @ self.b.T)
                    out["grad_b"] = (G @ self.a).T @ U
                    self.a = self._adam("a", mom, self.a, out["grad_a"], t)
                    self.b = self._adam("b", mom, self.b, out["grad_b"], t)
                logged = []
        if not c["head_mode"]:
            out["z"] = z.reshape(-1)
        return {**out, **self.caches(), "logits": lg.reshape(-1)}

    @staticmethod
    def _adam(name, mom, p, g, t):
        m, v = mom.get(name + ".m", 0.0), mom.get(name + ".v", 0.0)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        mom[name + ".m"], mom[name + ".v"] = m, v
        return p - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)

    def caches(self):
        s = self.s
        return {n: torch.cat([self.kv[b][l][i].reshape(-1) for l in range(s.L) for b in range(s.B)])
                for i, n in enumerate(("k", "v"))}


def exact(case, seed):
    c = case
    if c["kind"] == "linear":
        w, x = _linear_inputs(c, seed)
        return x.double() @ w.double().T
    flops = work(c)["flops"] + (_prefill_work(_dims(c), _lens(c))[1] if c["kind"] == "round" else 0)
    if flops > 1.8e13:   # about 20 seconds at the 64-bit rate
        return None
    r = _Ref(c, seed)
    if c["kind"] == "prefill":
        for b in range(r.s.B):
            r.prefill(b)
        return {"first": None, **r.caches()}
    if c["kind"] == "greedy":
        for b in range(r.s.B):
            tok = r.prefill(b)
            n = r.prompts[b].numel()
            for i in range(c["gen"] - 1):
                x = r.layers(0, r.s.L, b, r.embed([tok]), n + i)
                tok = int(r.logits(x)[0].argmax())
        return {"tokens": None, **r.caches()}
    if c["kind"] == "generate":
        return {"tokens": None, **r.decode(c["update_every"], 0, c["gen"])}
    got = r.decode(c["update_every"], c["update_every"], 0)
    return {"ids": None, "committed": None, "accepted": None, **got}
