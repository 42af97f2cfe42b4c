"""Timed cases of the library: what a program that serves these models asks of it.

Four kinds of work, each through the calls such a program makes (the ctypes binding of libtlf):

- ``attn``      one launch of the paged decode attention on a caller's own cache (``tlf_attn_decode``);
- ``decode``    one decode step for a batch of live sequences (``Context.decode_step``); every pass is the
                next step of the same sequences, so their caches grow by one token a pass;
- ``prefill``   new prompts in, the logits of their last tokens out (``Context.prefill``), then the
                sequences end (``Context.release``, host-side only), so every pass does the same work;
- ``generate``  a whole request: prefill of a batch of prompts, a number of decode steps, release.

Models are the repository's own configurations: ``tiny`` (float32), ``small``, ``mid`` and ``long`` (bf16;
``long`` has grouped-query attention and head_dim 128). Weights stand for a checkpoint that a program keeps
and do not depend on the seed; prompts, decode tokens, past loop counts, queries and caches come from it.

``exact`` restates the model in float64 on the GPU (plain torch).
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2609_15160_gb300 import synth, tlf

PAGE = 64
MODELS = {"tiny": "c1", "small": "c2", "mid": "c3", "long": "c4"}


def listed():
    return [
        # one attention launch of a small batch with short caches: launch and merge latency
        dict(name="attn-8x500", kind="attn", n=8, lo=300, hi=700, hq=8, hkv=8, hd=64, dtype="bf16"),
        # a ragged serving batch, multi-head, short and long caches side by side
        dict(name="attn-32-ragged", kind="attn", n=32, lo=128, hi=8192, hq=16, hkv=16, hd=64, dtype="bf16"),
        # long-context grouped-query attention: HBM streaming
        dict(name="attn-16x32k-gqa", kind="attn", n=16, lo=32000, hi=32768, hq=16, hkv=8, hd=128, dtype="bf16"),
        # one user, one token: latency of the whole step
        dict(name="decode-1x3000", kind="decode", model="mid", n=1, lo=3001, hi=3001, cond=False, rule="argmax", forced=0),
        # ragged serving batch
        dict(name="decode-32-ragged", kind="decode", model="mid", n=32, lo=128, hi=8192, cond=False, rule="argmax",
             forced=0),
        # many short conversations at once
        dict(name="decode-200-short", kind="decode", model="mid", n=200, lo=64, hi=700, cond=False, rule="argmax",
             forced=0),
        # long documents, grouped-query attention
        dict(name="decode-16x32k", kind="decode", model="long", n=16, lo=32000, hi=32700, cond=False, rule="argmax",
             forced=0),
        # a whole request on the float32 model, one sequence
        dict(name="generate-f32", kind="generate", model="tiny", n=1, lo=32, hi=32, steps=16, cond=False, rule="argmax",
             forced=0),
        # a whole request for a batch of eight on the conditioned small model
        dict(name="generate-8x450", kind="generate", model="small", n=8, lo=390, hi=512, steps=32, cond=True,
             rule="argmax", forced=0),
        # time to first token of a short prompt
        dict(name="prefill-1x117", kind="prefill", model="mid", n=1, lo=117, hi=117, cond=False, rule="argmax", forced=0),
        # admission of several ragged prompts
        dict(name="prefill-8-ragged", kind="prefill", model="mid", n=8, lo=128, hi=2048, cond=False, rule="argmax",
             forced=0),
        # a long document, more than one prefill chunk
        dict(name="prefill-1x10k", kind="prefill", model="long", n=1, lo=10007, hi=10007, cond=False, rule="argmax",
             forced=0),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["attn", "decode", "decode", "prefill", "prefill", "generate"])
    if kind == "attn":
        hq, hkv, hd, dtype = rng.choice([(8, 8, 64, "bf16"), (16, 16, 64, "bf16"), (16, 8, 128, "bf16"),
                                         (32, 8, 128, "bf16"), (4, 4, 16, "f32"), (8, 4, 64, "f32")])
        n = _log(rng, 1, 200)
        hi = _log(rng, 64, min(32768, 300000 // n))
        return dict(kind=kind, n=n, lo=rng.randint(1, hi), hi=hi, hq=hq, hkv=hkv, hd=hd, dtype=dtype)
    opt = dict(cond=rng.random() < 0.2, rule="survival" if rng.random() < 0.25 else "argmax",
               forced=1 if rng.random() < 0.15 else 0)
    if kind == "decode":
        model = rng.choice(["small", "mid", "mid", "long"])
        n = _log(rng, 1, 256)
        hi = _log(rng, 64, min(32768, {"small": 400000, "mid": 130000, "long": 200000}[model] // n))
        return dict(kind=kind, model=model, n=n, lo=rng.randint(1, hi), hi=hi, **opt)
    if kind == "prefill":
        model = rng.choice(["small", "mid", "long"])
        n = _log(rng, 1, 16)
        hi = _log(rng, 16, min(8192, 9000 // n))
        return dict(kind=kind, model=model, n=n, lo=rng.randint(1, hi), hi=hi, **opt)
    model = rng.choice(["tiny", "small", "small"])
    n = _log(rng, 1, 4 if model == "tiny" else 16)
    hi = _log(rng, 8, 48 if model == "tiny" else 512)
    return dict(kind=kind, model=model, n=n, lo=rng.randint(1, hi), hi=hi, steps=rng.randint(4, 24), **opt)


# ----------------------------------------------------------------------------
# models and inputs
# ----------------------------------------------------------------------------

def _model(case):
    m = synth.get_config(MODELS[case["model"]]).model
    return dataclasses.replace(m, conditioning=bool(case["cond"]), exit_rule=case["rule"], threshold=0.5)


def _lens(case):
    """n lengths spread over lo..hi (golden-ratio steps): the same for every seed, so the work is known."""
    lo, hi = case["lo"], case["hi"]
    return [lo + int((hi - lo + 0.999) * ((0.31 + 0.6180339887 * b) % 1.0)) for b in range(case["n"])]


_WEIGHTS = {}  # the checkpoint in use (one at a time)


def _weights(m):
    """Weights of the model's shapes: N(0, 0.02), bf16-exact for bf16 models, unit gains, and a router bias that
    gives the configuration's long-tailed loop counts; conditioning weights as the repository makes them."""
    if m in _WEIGHTS:
        return _WEIGHTS[m]
    _WEIGHTS.clear()
    g = torch.Generator(device="cuda").manual_seed(1234)

    def normal(*shape):
        x = torch.randn(shape, generator=g, device="cuda") * m.init_std
        return (x.bfloat16().float() if m.dtype == "bf16" else x).cpu().numpy()

    d, J, ff = m.d_model, m.n_layers, m.ffn_hidden
    w = {"embedding": normal(m.vocab, d), "router_w": normal(m.max_loops, d), "wq": normal(J, m.q_dim, d),
         "wk": normal(J, m.kv_dim, d), "wv": normal(J, m.kv_dim, d), "wo": normal(J, d, m.q_dim),
         "w_gate": normal(J, ff, d), "w_up": normal(J, ff, d), "w_down": normal(J, d, ff)}
    w["router_b"] = (np.zeros(m.max_loops, np.float32) if m.depth_probs is None else synth.calibrate_router_bias(
        w["router_w"], m.depth_probs, m.init_std, m.norm_eps, 0, n_samples=20000))
    w["attn_norm"], w["mlp_norm"] = np.ones((J, d), np.float32), np.ones((J, d), np.float32)
    w["final_norm"] = np.ones(d, np.float32)
    if m.conditioning:
        w.update(synth.make_conditioning_weights(m))
    _WEIGHTS[m] = w
    return w


def _keep(m):
    """P(loop count >= r), r = 1..M."""
    p = np.full(m.max_loops, 1.0 / m.max_loops) if m.depth_probs is None else np.asarray(m.depth_probs)
    return p[::-1].cumsum()[::-1]


def _prompts(case, m, seed):
    rng = np.random.default_rng([seed, 1])
    return [rng.integers(0, m.vocab, size=n).astype(np.int32) for n in _lens(case)]


def _steps(case, m, seed, steps):
    return np.random.default_rng([seed, 2]).integers(0, m.vocab, size=(steps, case["n"])).astype(np.int32)


def _positions(case, m, seed):
    """Past loop counts of every sequence as the positions each loop's cache holds."""
    return [synth.make_cache_positions(m, n, seed * 1000 + b) for b, n in enumerate(_lens(case))]


def _attn_problem(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    lens = _lens(case)
    need = [(n + PAGE - 1) // PAGE for n in lens]
    n_pages, max_pages = sum(need) + 3, max(need)
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    pool = torch.randn((n_pages, 2, 2, case["hkv"], PAGE, case["hd"]), generator=g, device="cuda", dtype=dt)
    q = torch.randn((case["n"], case["hq"], case["hd"]), generator=g, device="cuda")
    order = np.random.default_rng([seed, 3]).permutation(n_pages).astype(np.int32)
    table, o = np.full((case["n"], max_pages), -1, np.int32), 0
    for b, k in enumerate(need):
        table[b, :k] = order[o:o + k]
        o += k
    return dict(lens=torch.tensor(lens, dtype=torch.int32, device="cuda"), table=torch.from_numpy(table).cuda(), pool=pool,
                q=q, n_pages=n_pages, max_pages=max_pages)


def _room(case):
    """Decode steps a state has room for before its sequences end and are restored again."""
    return 4096 if case["n"] <= 16 else 1024


def _forced(case, m, shape):
    return np.full(shape, m.max_loops, np.int32) if case["forced"] else None


def prepare(case, seed):
    if case["kind"] == "attn":
        p = _attn_problem(case, seed)
        out = torch.zeros((case["n"], case["hq"] * case["hd"]), dtype=p["pool"].dtype, device="cuda")
        err = torch.zeros(4, dtype=torch.int32, device="cuda")
        a = tlf.attn_args(case["n"], case["hq"], case["hkv"], case["hd"], 2, 1, case["dtype"], p["max_pages"], p["n_pages"],
                          p["q"], p["pool"], p["table"], p["lens"], out, err)
        nbytes = tlf.tlf_attn_decode_scratch_bytes(a)
        return dict(case=case, p=p, out=out, err=err, args=a, nbytes=nbytes,
                    scratch=torch.empty(nbytes, dtype=torch.uint8, device="cuda"))
    m, n, lens = _model(case), case["n"], _lens(case)
    M = m.max_loops
    grow = {"decode": _room(case), "prefill": 1, "generate": case.get("steps", 0) + 1}[case["kind"]]
    pages = sum(M * ((x + grow + PAGE - 1) // PAGE + 1) for x in lens)
    ctx = tlf.Context(m, _weights(m), max_seqs=n, max_batch=n, max_seq_len=max(lens) + grow, kv_pool_pages=pages)
    s = dict(case=case, ctx=ctx, m=m, ids=np.arange(1, n + 1, dtype=np.uint64))
    if case["kind"] == "decode":
        s.update(tokens=_steps(case, m, seed, grow), step=0, forced=_forced(case, m, n),
                 snapshots=_positions(case, m, seed), logits=torch.empty((n, m.vocab), device="cuda"))
        _restore(s)
        return s
    s["prompts"] = _prompts(case, m, seed)
    f = _forced(case, m, sum(lens))
    s["forced"] = None if f is None else np.split(f, np.cumsum(lens)[:-1])
    s["last"] = torch.empty((n, m.vocab), device="cuda")
    if case["kind"] == "generate":
        s.update(tokens=_steps(case, m, seed, case["steps"]), step_forced=_forced(case, m, n),
                 logits=torch.empty((case["steps"], n, m.vocab), device="cuda"))
    return s


def _restore(s):
    for i, snap in zip(s["ids"], s["snapshots"]):
        s["ctx"].load_cache(int(i), snap)


def run(s):
    kind = s["case"]["kind"]
    if kind == "attn":
        tlf.tlf_attn_decode(s["args"], s["scratch"], s["nbytes"])
        return s["out"]
    ctx, ids = s["ctx"], s["ids"]
    if kind == "decode":
        if s["step"] == len(s["tokens"]):  # the sequences are full: they end and others take their places
            for i in ids:
                ctx.release(int(i))
            _restore(s)
            s["step"] = 0
        logits, loops, margin = ctx.decode_step(ids, s["tokens"][s["step"]], forced=s["forced"], logits=s["logits"])
        s["step"] += 1
        return {"logits": logits, "loops": loops, "margin": margin}
    last, loops = ctx.prefill(ids, s["prompts"], forced=s["forced"], logits_out=s["last"])
    out = {"last": last, "loops": np.concatenate(loops)}
    if kind == "generate":
        out["step_loops"] = np.stack([ctx.decode_step(ids, t, forced=s["step_forced"], logits=s["logits"][k])[1]
                                      for k, t in enumerate(s["tokens"])])
        out["logits"] = s["logits"]
    for i in ids:
        ctx.release(int(i))
    return out


# ----------------------------------------------------------------------------
# work and tolerance
# ----------------------------------------------------------------------------

def work(case):
    lens = np.asarray(_lens(case), float)
    if case["kind"] == "attn":
        eb = 2 if case["dtype"] == "bf16" else 4
        kv = lens.sum() * 2 * case["hkv"] * case["hd"] * eb
        return {"bytes": kv + case["n"] * case["hq"] * case["hd"] * (4 + eb), "flops": 4 * lens.sum() * case["hq"] * case["hd"]}
    m = _model(case)
    eb = 2 if m.dtype == "bf16" else 4
    keep = np.ones(m.max_loops) if case["forced"] else _keep(m)
    depth, J = keep.sum(), m.n_layers
    block, head = J * m.layer_params(), m.vocab * m.d_model
    kv = 2 * m.kv_dim * J * eb  # bytes of one token's cache entries in one loop

    def causal(a, b):  # (query, key) pairs of queries a..b of every loop
        return (keep ** 2).sum() * (b * (b + 1) - a * (a + 1)) / 2

    if case["kind"] == "decode":
        n = case["n"]
        past = _keep(m).sum() * lens.sum()
        b = (block + head) * eb + (past + n * depth) * kv + n * m.vocab * 4
        f = 2.0 * n * (depth * block + head) + 4.0 * (past + n * depth) * m.q_dim * J
        return {"bytes": float(b), "flops": float(f)}
    T, n, steps = lens.sum(), case["n"], case.get("steps", 0)
    b = (block + head) * eb + T * depth * kv + n * m.vocab * 4
    f = 2.0 * (T * depth * block + n * head) + 4.0 * causal(0, lens).sum() * m.q_dim * J
    if steps:
        # each step reads the weights again: a step's tokens are known only after the one before
        b += steps * ((block + head) * eb + n * m.vocab * 4) + (steps * T + n * steps * steps / 2) * depth * kv
        f += 2.0 * steps * n * (depth * block + head) + 4.0 * (causal(lens, lens + steps)).sum() * m.q_dim * J
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    if case["kind"] == "attn":
        return {"rel": 7e-3} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 1e-3}
    if case["model"] == "tiny":
        return {"rel": 1e-5, "max": 1e-3}
    # bf16: activations are rounded between the up to 8 x 4 layers that a token runs. Decode rounds its
    # operands to two terms; prefill to one, and its caches carry that into the steps after it.
    return {"rel": 7e-3} if case["kind"] == "decode" else {"rel": 2.5e-2}


# ----------------------------------------------------------------------------
# the same in float64
# ----------------------------------------------------------------------------

class _Model64:
    def __init__(self, m):
        self.m = m
        self.w = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda().double() for k, v in _weights(m).items()}
        half = m.head_dim // 2
        self.freq = m.rope_base ** (-2.0 * torch.arange(half, device="cuda").double() / m.head_dim)
        self.mods = {}

    def norm(self, x, gain=None):
        y = x / torch.sqrt((x * x).mean(-1, keepdim=True) + self.m.norm_eps)
        return y if gain is None else y * gain

    def loops(self, tokens, forced):
        m = self.m
        if forced:
            return torch.full((len(tokens),), m.max_loops, device="cuda")
        z = self.norm(self.w["embedding"][tokens]) @ self.w["router_w"].T + self.w["router_b"]
        if m.exit_rule == "argmax":
            return z.argmax(-1) + 1
        p = torch.softmax(z, -1).flip(-1).cumsum(-1).flip(-1)
        i = torch.arange(1, m.max_loops + 1, device="cuda")
        return torch.where(p > m.threshold, i, torch.ones_like(i)).amax(-1)

    def modulation(self, j, depth, r):
        """[rows, 4, d]: (alpha_msa, alpha_mlp, gamma_msa, gamma_mlp) of rows of these depths at loop r (0-based)."""
        m, out = self.m, []
        for dep in depth.tolist():
            if (j, dep, r) not in self.mods:
                c = 0.0
                for which, x in (("t", r / dep), ("dt", 1.0 / dep)):
                    wk = torch.exp(-torch.arange(128, device="cuda").double() / 128 * math.log(10000.0))
                    f = torch.stack([torch.cos(x * wk), torch.sin(x * wk)], -1).reshape(-1)
                    h = torch.nn.functional.silu(self.w[f"cond_{which}_w1"] @ f + self.w[f"cond_{which}_b1"])
                    c = c + self.w[f"cond_{which}_w2"] @ h + self.w[f"cond_{which}_b2"]
                v = self.w["mod_w"][j] @ torch.nn.functional.silu(c) + self.w["mod_b"][j]
                self.mods[(j, dep, r)] = v.reshape(4, m.d_model)
            out.append(self.mods[(j, dep, r)])
        return torch.stack(out)

    def rope(self, x, pos):  # x [T, H, hd]
        a = pos.double()[:, None] * self.freq
        c, s = torch.cos(a)[:, None], torch.sin(a)[:, None]
        h = x.shape[-1] // 2
        return torch.cat([x[..., :h] * c - x[..., h:] * s, x[..., :h] * s + x[..., h:] * c], -1)

    def attend(self, q, k, v, past):
        """q [T, Hq, hd] against k, v [past + T, Hkv, hd]; query i sees the first past + i + 1 keys."""
        T, hq, hd = q.shape
        g, out = hq // k.shape[1], torch.empty_like(q)
        for a in range(0, T, 512):
            b = min(T, a + 512)
            n = past + b
            kk, vv = k[:n].transpose(0, 1), v[:n].transpose(0, 1)
            qq = q[a:b].reshape(b - a, -1, g, hd).permute(1, 2, 0, 3).reshape(-1, g * (b - a), hd)
            sc = (qq @ kk.transpose(1, 2)).reshape(-1, g, b - a, n) / math.sqrt(hd)
            seen = torch.arange(n, device="cuda")[None] <= past + torch.arange(a, b, device="cuda")[:, None]
            p = torch.softmax(sc.masked_fill(~seen, -math.inf), -1)
            o = p.reshape(-1, g * (b - a), n) @ vv
            out[a:b] = o.reshape(-1, g, b - a, hd).permute(2, 0, 1, 3).reshape(b - a, hq, hd)
        return out

    def extend(self, cache, tokens, start, forced):
        """Runs new tokens at positions start.. of one sequence; cache(r, j) -> (K, V) or None and cache.put(r, j, K, V)
        keep its caches. Returns (logits after the last token, loop counts)."""
        m, w = self.m, self.w
        tokens = torch.as_tensor(np.asarray(tokens), device="cuda").long()
        loops = self.loops(tokens, forced)
        h = w["embedding"][tokens]
        pos = start + torch.arange(len(tokens), device="cuda")
        for r in range(m.max_loops):
            rows = torch.nonzero(loops > r).reshape(-1)
            if not len(rows):
                break
            x = h[rows]
            for j in range(m.n_layers):
                mod = self.modulation(j, loops[rows], r) if m.conditioning else None
                y = self.norm(x, w["attn_norm"][j])
                y = y if mod is None else y * (1 + mod[:, 2])
                q = self.rope((y @ w["wq"][j].T).reshape(len(rows), -1, m.head_dim), pos[rows])
                k = self.rope((y @ w["wk"][j].T).reshape(len(rows), -1, m.head_dim), pos[rows])
                v = (y @ w["wv"][j].T).reshape(len(rows), -1, m.head_dim)
                old = cache.get(r, j)
                past = 0 if old is None else old[0].shape[0]
                if old is not None:
                    k, v = torch.cat([old[0], k]), torch.cat([old[1], v])
                cache.put(r, j, k, v)
                o = self.attend(q, k, v, past).reshape(len(rows), -1) @ w["wo"][j].T
                x = x + (o if mod is None else o * mod[:, 0])
                y = self.norm(x, w["mlp_norm"][j])
                y = y if mod is None else y * (1 + mod[:, 3])
                u = torch.nn.functional.silu(y @ w["w_gate"][j].T) * (y @ w["w_up"][j].T)
                o = u @ w["w_down"][j].T
                x = x + (o if mod is None else o * mod[:, 1])
            h[rows] = x
        return self.norm(h[-1], w["final_norm"]) @ w["embedding"].T, loops


class _Kept:
    """Caches that are kept from call to call."""

    def __init__(self):
        self.kv = {}

    def get(self, r, j):
        return self.kv.get((r, j))

    def put(self, r, j, k, v):
        self.kv[(r, j)] = (k, v)


class _Restored:
    """The caches of a sequence restored without values: element x of the pool is (fmix32(x) mod 256 - 128) / 64 (the
    documented filling), and a fresh context hands out its pages in order. first[r] is the first page of loop r."""

    def __init__(self, m, lens, first):
        self.m, self.lens, self.first = m, lens, first

    def get(self, r, j):
        m, n = self.m, self.lens[r]
        if n == 0:
            return None
        e = torch.arange(n, device="cuda")
        page_elems = m.n_layers * 2 * m.n_kv_heads * PAGE * m.head_dim
        at = (self.first[r] + e // PAGE) * page_elems + (e % PAGE) * m.head_dim
        head = torch.arange(m.n_kv_heads, device="cuda")[:, None] * PAGE * m.head_dim
        inner = (head + torch.arange(m.head_dim, device="cuda"))[None]
        out = []
        for kv in range(2):
            x = (at[:, None, None] + (j * 2 + kv) * m.n_kv_heads * PAGE * m.head_dim + inner) & 0xFFFFFFFF
            for shift, mul in ((16, 0x85EBCA6B), (13, 0xC2B2AE35), (16, 1)):
                x = ((x ^ (x >> shift)) * mul) & 0xFFFFFFFF
            out.append(((x & 255) - 128).double() / 64)
        return out

    def put(self, r, j, k, v):
        pass


def exact(case, seed):
    if case["kind"] == "attn":
        p, rows = _attn_problem(case, seed), []
        g = case["hq"] // case["hkv"]
        for b, n in enumerate(_lens(case)):
            pages = p["table"][b, :(n + PAGE - 1) // PAGE].long()
            k, v = (p["pool"][pages, 1, i].transpose(1, 2).reshape(-1, case["hkv"], case["hd"])[:n].double() for i in (0, 1))
            q = p["q"][b].double().reshape(case["hkv"], g, case["hd"])
            w = torch.softmax(torch.einsum("hgd,nhd->hgn", q, k) / math.sqrt(case["hd"]), -1)
            rows.append(torch.einsum("hgn,nhd->hgd", w, v).reshape(-1))
        return torch.stack(rows)
    m = _model(case)
    model = _Model64(m)
    if case["kind"] == "decode":
        tokens, logits, loops, page = _steps(case, m, seed, _room(case))[0], [], [], 0
        for b, snap in enumerate(_positions(case, m, seed)):
            lens, first = [len(x) for x in snap["positions"]], []
            for x in lens:
                first.append(page)
                page += (x + PAGE - 1) // PAGE
            lg, lp = model.extend(_Restored(m, lens, first), tokens[b:b + 1], lens[0], case["forced"])
            logits.append(lg)
            loops.append(lp)
        return {"logits": torch.stack(logits), "loops": torch.cat(loops).int().cpu().numpy(), "margin": None}
    last, loops, kept = [], [], []
    for p in _prompts(case, m, seed):
        kept.append(_Kept())
        lg, lp = model.extend(kept[-1], p, 0, case["forced"])
        last.append(lg)
        loops.append(lp)
    out = {"last": torch.stack(last), "loops": torch.cat(loops).int().cpu().numpy()}
    if case["kind"] == "generate":
        lens, logits, step_loops = _lens(case), [], []
        for k, t in enumerate(_steps(case, m, seed, case["steps"])):
            got = [model.extend(kept[b], t[b:b + 1], lens[b] + k, case["forced"]) for b in range(case["n"])]
            logits.append(torch.stack([x for x, _ in got]))
            step_loops.append(torch.cat([x for _, x in got]))
        out["step_loops"] = torch.stack(step_loops).int().cpu().numpy()
        out["logits"] = torch.stack(logits)
    return out
