"""The work that users of the MTP decode path have it do, as measurable cases.

Five kinds of call, each through the package's public entry points:

  viterbi    mtp_viterbi: paths and acceptance of candidate lattices
  heads      mtp_heads_topk: the n heads, log-softmax and top-k of hidden rows
  attention  mtp_attention (decode rows over the paged cache) and
             mtp_attention_tc (prompt rows, "tc": True)
  gemm       mtp_gemm_bf16x2: one of the block's projections over many rows
  request    a whole job: prompts in, prefill, generation, logits of the last step

Sizes are the repository's own configurations (the tiny fp32 model, the
VALL-E-sized bf16 model, the serving ranges and the microbenchmark shapes) and
the ranges around them.  Model weights are fixed, as a service keeps them; the
seed draws everything that changes from call to call.
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2410_13839_gb300 import mtp

V, EOS, HD, N_MAX, K_MAX = 1025, 1024, 64, 8, 32

# layers, d_model, d_ffn, phoneme vocabulary, matrix type
MODELS = {
    "tiny": (2, 256, 1024, 128, "f32"),
    "valle": (12, 1024, 4096, 512, "bf16"),
    "valle_heads": (1, 1024, 1024, 512, "bf16"),  # a program that calls only the heads keeps no block stack
}
PROJECTIONS = {"qkv": (3072, 1024), "wo": (1024, 1024), "w1": (4096, 1024), "w2": (1024, 4096)}


def listed():
    return [
        # one utterance's selection after a step: the smallest call, all latency
        {"name": "viterbi 1", "kind": "viterbi", "batch": 1, "n": 4, "k": 4, "budget": True},
        # offline rescoring of many lattices (the microbenchmark's shape)
        {"name": "viterbi 10000", "kind": "viterbi", "batch": 10000, "n": 8, "k": 16, "budget": False},
        # the heads of one utterance's last hidden row, logits wanted
        {"name": "heads 1", "kind": "heads", "rows": 1, "n": 4, "k": 4, "dtype": "f32", "logits": True},
        # the heads over a batch of hidden rows (the microbenchmark's shape)
        {"name": "heads 256", "kind": "heads", "rows": 256, "n": 8, "k": 16, "dtype": "bf16", "logits": False},
        # one layer's decode attention of a serving batch: ragged contexts, four fed rows a slot
        {"name": "attention decode 32", "kind": "attention", "tc": False, "slots": 32, "per_slot": 4,
         "ctx_lo": 180, "ctx_hi": 2000, "page": 64},
        # one layer's attention of packed prompts, every position of each
        {"name": "attention prompts", "kind": "attention", "tc": True, "slots": 5, "per_slot": 0,
         "ctx_lo": 182, "ctx_hi": 578, "page": 64},
        # the MLP's first projection over the fed rows of 128 slots
        {"name": "projection 512", "kind": "gemm", "proj": "w1", "rows": 512, "splits": 1},
        # the tiny fp32 model: a whole utterance of 150 codes
        {"name": "request tiny", "kind": "request", "model": "tiny", "batch": 1, "ph_lo": 32, "ph_hi": 32,
         "ac_lo": 75, "ac_hi": 75, "tokens": 150, "n": 4, "k": 4, "verify": False},
        # one interactive utterance: a 3 s acoustic prompt, 2.5 s generated
        {"name": "request 1", "kind": "request", "model": "valle", "batch": 1, "ph_lo": 64, "ph_hi": 64,
         "ac_lo": 225, "ac_hi": 225, "tokens": 192, "n": 4, "k": 4, "verify": False},
        # a handful of utterances decoded with verified drafts (output equal to greedy decoding)
        {"name": "request verify 5", "kind": "request", "model": "valle", "batch": 5, "ph_lo": 32, "ph_hi": 128,
         "ac_lo": 150, "ac_hi": 450, "tokens": 24, "n": 4, "k": 4, "verify": True},
        # batched serving: 32 prompts prefilled together, then their first second and a bit
        {"name": "request 32", "kind": "request", "model": "valle", "batch": 32, "ph_lo": 32, "ph_hi": 128,
         "ac_lo": 150, "ac_hi": 450, "tokens": 96, "n": 4, "k": 4, "verify": False},
        # the largest serving batch: admission, prefill and the first packets of 128 utterances
        {"name": "request 128", "kind": "request", "model": "valle", "batch": 128, "ph_lo": 32, "ph_hi": 128,
         "ac_lo": 150, "ac_hi": 450, "tokens": 40, "n": 4, "k": 4, "verify": False},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["viterbi", "heads", "attention", "attention", "gemm", "request", "request", "request"])
    if kind == "viterbi":
        return {"kind": kind, "batch": _log_int(rng, 1, 10000), "n": rng.randint(1, 8), "k": _log_int(rng, 1, 25),
                "budget": rng.random() < 0.5}
    if kind == "heads":
        return {"kind": kind, "rows": _log_int(rng, 1, 500), "n": rng.randint(1, 8), "k": _log_int(rng, 1, 32),
                "dtype": rng.choice(["f32", "bf16"]), "logits": rng.random() < 0.5}
    if kind == "attention":
        tc = rng.random() < 0.5
        lo = _log_int(rng, 33, 1000)
        return {"kind": kind, "tc": tc, "slots": _log_int(rng, 1, 8 if tc else 96),
                "per_slot": 0 if tc else rng.randint(1, 8), "ctx_lo": lo, "ctx_hi": min(2000, lo * rng.randint(1, 3)),
                "page": rng.choice([16, 32, 64, 128])}
    if kind == "gemm":
        proj = rng.choice(sorted(PROJECTIONS))
        splits = rng.choice([1, 2, 4, 8]) if proj in ("wo", "w2") else 1
        return {"kind": kind, "proj": proj, "rows": _log_int(rng, 1, 3000), "splits": splits}
    n = rng.choice([1, 2, 4, 8])
    c = {"kind": kind, "model": "valle" if rng.random() < 0.8 else "tiny", "batch": 1, "n": n,
         "k": rng.choice([1, 4, 8, 25]), "verify": rng.random() < 0.2,
         "ph_lo": 32, "ph_hi": rng.randint(32, 128), "ac_lo": rng.randint(75, 200), "ac_hi": rng.randint(200, 450)}
    if c["model"] == "valle" and rng.random() < 0.6:
        c["batch"] = _log_int(rng, 2, 16 if c["verify"] else 96)
    if c["verify"]:   # about one token a step
        c["tokens"] = rng.randint(8, 24)
    else:
        c["tokens"] = n * rng.randint(4, 24) if c["batch"] < 32 else n * rng.randint(2, 12) - rng.randint(0, n - 1)
    return c


# ---- inputs ----


def _gen(*key):
    seed = 0
    for x in key:
        for b in str(x).encode() + b"/":
            seed = (seed * 1000003 + b + 1) % (1 << 61)
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(gen, *shape, scale=1.0):
    return torch.randn(*shape, device="cuda", generator=gen) * scale


def _transitions(gen):
    """log Q [V][V]: a code is often followed by itself, and its other successors are uneven."""
    g = 2.0 * _normal(gen, V, V).double()
    e = torch.exp(g - g.amax(1, keepdim=True))
    q = 0.7 * e / e.sum(1, keepdim=True) + 0.3 * torch.eye(V, device="cuda", dtype=torch.float64)
    return torch.log(q).float()


def _tensors(name):
    """The model's weights on the GPU in blob order, as (tensor fp32, is a matrix): matrices
    N(0, 0.02) in the matrix type's precision, and head biases that give the codes Zipf-like
    frequencies (the same for every head), as a trained model's are; EOS never wins."""
    layers, d, f, phones, dtype = MODELS[name]
    gen = _gen("weights", name)

    def mat(*shape):
        w = _normal(gen, *shape, scale=0.02)
        return (w.bfloat16().float() if dtype == "bf16" else w, True)

    def vec(*shape, one=0.0):
        return (one + _normal(gen, *shape, scale=0.02), False)

    out = [mat(phones, d), mat(V, d)]
    for _ in range(layers):
        out += [vec(d, one=1.0), vec(d), mat(3 * d, d), vec(3 * d), mat(d, d), vec(d),
                vec(d, one=1.0), vec(d), mat(f, d), vec(f), mat(d, f), vec(d)]
    rank = torch.randperm(V, device="cuda", generator=gen)
    bias = -torch.log(1.0 + rank.float())
    bias[EOS] = -30.0
    out += [vec(d, one=1.0), vec(d), mat(N_MAX, V, d), (vec(N_MAX, V)[0] + bias, False), (_transitions(gen), False)]
    return out


@functools.lru_cache(maxsize=None)
def _blob(name):
    return mtp.pack_weights([(t.cpu().numpy(), m) for t, m in _tensors(name)], MODELS[name][4] == "bf16")


def _context(name, batch, max_ctx, page=64, verify=False):
    layers, d, f, phones, dtype = MODELS[name]
    model = SimpleNamespace(layers=layers, d_model=d, n_attn_heads=d // HD, d_ffn=f, phone_vocab=phones,
                            codec_vocab=V, eos_id=EOS, n_heads_max=N_MAX, top_k_max=K_MAX, weight_dtype=dtype,
                            ln_eps=1e-5)
    config = mtp.make_config(model, batch, max_ctx, page, accept_policy=1 if verify else 0)
    return _Handle(mtp.mtp_create(config, _blob(name), torch.cuda.current_stream()))


class _Handle:
    """An mtp_ctx that is destroyed with its state."""

    def __init__(self, ctx):
        self.ctx = ctx

    def __del__(self):
        if self.ctx:
            mtp.mtp_destroy(self.ctx)
            self.ctx = None


def _lengths(case, seed):
    """Prompt lengths (phonemes, acoustic) of each sequence."""
    rng = np.random.default_rng([seed, 11])
    b = case["batch"]
    return (rng.integers(case["ph_lo"], case["ph_hi"] + 1, b).tolist(),
            rng.integers(case["ac_lo"], case["ac_hi"] + 1, b).tolist())


def _prompts(case, seed):
    gen = _gen("prompts", seed)
    phones = MODELS[case["model"]][3]
    out = []
    for n_ph, n_ac in zip(*_lengths(case, seed)):
        out.append((torch.randint(0, phones, (n_ph,), device="cuda", generator=gen, dtype=torch.int32),
                    torch.randint(0, EOS, (n_ac,), device="cuda", generator=gen, dtype=torch.int32)))
    return out


def _contexts(case):
    """Cached length of each slot (sizes, so part of the case)."""
    rng = np.random.default_rng([case["slots"], case["ctx_lo"], case["ctx_hi"]])
    lens = rng.integers(case["ctx_lo"], case["ctx_hi"] + 1, case["slots"])
    return np.maximum(lens, max(1, case["per_slot"])).astype(np.int64)


def _swizzle(pool):
    """The cache's row layout (its own inverse): 16-byte chunk c of row t at chunk c ^ (t mod 8)."""
    p = pool.shape[-2]
    t = torch.arange(p, device=pool.device)[:, None] & 7
    c = torch.arange(8, device=pool.device)[None, :]
    return pool.view(*pool.shape[:-1], 8, 8)[..., torch.arange(p, device=pool.device)[:, None], c ^ t, :].flatten(-2)


def _attention_inputs(case, seed):
    gen = _gen("attention", seed)
    heads, page, tc = 16, case["page"], case["tc"]
    ctx = _contexts(case)
    per_seq = int((ctx.max() + page - 1) // page) + 1
    n_pages = case["slots"] * per_seq
    pool = _normal(gen, n_pages, 1, 2, heads, page, HD).bfloat16()   # plain layout
    table = torch.randperm(n_pages, device="cuda", generator=gen).to(torch.int32).view(case["slots"], per_seq)
    if tc:  # every position of every prompt, packed
        seq = np.concatenate([np.full(c, s) for s, c in enumerate(ctx)])
        pos = np.concatenate([np.arange(c) for c in ctx])
    else:   # the last rows of every slot
        seq = np.repeat(np.arange(case["slots"]), case["per_slot"])
        pos = np.concatenate([np.arange(c - case["per_slot"], c) for c in ctx])
    q = _normal(gen, len(seq), heads * HD)
    to = lambda x: torch.from_numpy(x.astype(np.int32)).cuda()  # noqa: E731
    return SimpleNamespace(heads=heads, page=page, ctx=ctx, per_seq=per_seq, pool=pool, table=table, seq=to(seq),
                           pos=to(pos), q=q, rows=len(seq))


def _viterbi_inputs(case, seed):
    gen = _gen("viterbi", seed)
    b, n, k = case["batch"], case["n"], case["k"]
    # distinct ids per position, scores descending as a top-k gives them
    ids = torch.topk(torch.rand(b * n, V, device="cuda", generator=gen), k, dim=1).indices
    lp = torch.log(torch.rand(b * n, k, device="cuda", generator=gen).clamp_min(1e-6)).sort(1, descending=True).values
    rem = torch.randint(1, n + 3, (b,), device="cuda", generator=gen, dtype=torch.int32) if case["budget"] else None
    return (ids.to(torch.int32).view(b, n, k).contiguous(), lp.view(b, n, k).contiguous(), rem)


@functools.lru_cache(maxsize=None)
def _log_q():
    return _transitions(_gen("transitions"))


def _hidden(case, seed):
    h = _normal(_gen("hidden", seed), case["rows"], 1024).bfloat16()
    return h if case["dtype"] == "bf16" else h.float()


def _gemm_inputs(case, seed):
    gen = _gen("gemm", seed)
    n_w, k = PROJECTIONS[case["proj"]]
    w = _normal(gen, n_w, k, scale=0.02).bfloat16()
    a = _normal(gen, case["rows"], k)
    hi = a.bfloat16()
    lo = (a - hi.float()).bfloat16()
    return w, hi, lo, (_normal(gen, case["rows"], n_w) if case["splits"] > 1 else None)


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case)
    new = lambda dtype, *shape: torch.zeros(shape, dtype=dtype, device="cuda")  # noqa: E731
    if kind == "viterbi":
        s.ids, s.lp, s.rem = _viterbi_inputs(case, seed)
        s.log_q = _log_q()
        b, n = case["batch"], case["n"]
        s.path, s.score = new(torch.int32, b, n), new(torch.float32, b)
        s.accepted, s.rollback = new(torch.int32, b), new(torch.int32, b)
    elif kind == "heads":
        r, n, k = case["rows"], case["n"], case["k"]
        s.handle = _context("valle_heads", 32, 64)
        s.hidden = _hidden(case, seed)
        s.ids, s.logp, s.lse = new(torch.int32, r, n, k), new(torch.float32, r, n, k), new(torch.float32, r, n)
        s.logits = new(torch.float32, r, n, V) if case["logits"] else None
    elif kind == "attention":
        s.i = i = _attention_inputs(case, seed)
        if case["tc"]:
            i.pool = _swizzle(i.pool).contiguous()
        s.out = new(torch.float32, i.rows, i.heads * HD)
        s.args = mtp.attention_args(rows=i.rows, rows_per_group=case["per_slot"] or 8, n_heads=i.heads,
                                    page_size=i.page, layers=1, layer=0, bt_stride=i.per_seq,
                                    max_keys=int(i.ctx.max()), q=i.q, kv_pool=i.pool, block_table=i.table,
                                    row_seq=i.seq, row_pos=i.pos, out=s.out)
        size = mtp.mtp_attention_tc_workspace_bytes if case["tc"] else mtp.mtp_attention_workspace_bytes
        s.ws_bytes = size(s.args)
        s.ws = new(torch.uint8, max(16, s.ws_bytes))
    elif kind == "gemm":
        s.w, s.hi, s.lo, s.base = _gemm_inputs(case, seed)
        s.out = new(torch.float32, case["rows"], s.w.shape[0])
    else:
        b, n, t = case["batch"], case["n"], case["tokens"]
        s.prompts = _prompts(case, seed)
        longest = max(len(p) + len(a) for p, a in s.prompts)
        s.handle = _context(case["model"], b, longest + t + N_MAX + 8, verify=case["verify"])
        s.tokens, s.lens = new(torch.int32, b, t), new(torch.int32, b)
        s.logits, s.lse = new(torch.float32, b, n, V), new(torch.float32, b, n)
    return s


def run(s):
    case, stream = s.case, torch.cuda.current_stream()
    kind = case["kind"]
    if kind == "viterbi":
        mtp.mtp_viterbi(case["batch"], case["n"], case["k"], V, EOS, s.ids, s.lp, s.log_q, s.rem, s.path, s.score,
                        s.accepted, s.rollback, stream)
        return {"path": s.path, "score": s.score, "accepted": s.accepted, "rollback": s.rollback}
    if kind == "heads":
        mtp.mtp_heads_topk(s.handle.ctx, case["rows"], s.hidden, 1 if case["dtype"] == "bf16" else 0, case["n"],
                           case["k"], s.ids, s.logp, s.logits, s.lse)
        return {"ids": s.ids, "logp": s.logp, "lse": s.lse, "logits": s.logits}
    if kind == "attention":
        call = mtp.mtp_attention_tc if case["tc"] else mtp.mtp_attention
        call(s.args, s.ws, s.ws_bytes, stream)
        return s.out
    if kind == "gemm":
        if s.base is not None:  # added to the residual rows
            s.out.copy_(s.base)
        mtp.mtp_gemm_bf16x2(s.w, s.hi, s.lo, s.out, s.w.shape[0], s.w.shape[1], case["rows"], case["splits"],
                            int(s.base is not None), stream)
        return s.out
    ctx = s.handle.ctx
    if case["batch"] == 1:
        mtp.mtp_prefill(ctx, 0, *s.prompts[0], case["tokens"])
    else:
        for b, (ph, ac) in enumerate(s.prompts):
            mtp.mtp_admit(ctx, b, ph, ac, case["tokens"])
        mtp.mtp_prefill_pending(ctx)
    mtp.mtp_generate(ctx, case["n"], case["k"], s.tokens, case["tokens"], s.lens)
    mtp.mtp_debug_logits(ctx, s.logits, s.lse)
    return {"tokens": s.tokens, "lens": s.lens, "logits": s.logits, "lse": s.lse}


# ---- what a pass cannot do without ----


def work(case):
    kind = case["kind"]
    if kind == "viterbi":
        b, n, k = case["batch"], case["n"], case["k"]
        table = min(V * V, b * (n - 1) * k * k) * 4   # the transition scores that can be looked up
        return {"bytes": b * n * k * 8 + table + b * (4 * n + 16), "flops": 2.0 * b * (n - 1) * k * k}
    if kind == "heads":
        r, n, k = case["rows"], case["n"], case["k"]
        b = n * V * (1024 * 2 + 4) + r * 1024 * (2 if case["dtype"] == "bf16" else 4) + r * n * (8 * k + 4)
        return {"bytes": b + (r * n * V * 4 if case["logits"] else 0), "flops": 2.0 * r * n * V * 1024}
    if kind == "attention":
        mean = (case["ctx_lo"] + case["ctx_hi"]) / 2
        rows = case["slots"] * (mean if case["tc"] else case["per_slot"])
        pairs = case["slots"] * mean * (mean / 2) if case["tc"] else rows * mean
        return {"bytes": case["slots"] * mean * 16 * HD * 2 * 2 + rows * 16 * HD * 4 * 2, "flops": pairs * 16 * HD * 4}
    if kind == "gemm":
        n_w, k = PROJECTIONS[case["proj"]]
        m = case["rows"]
        return {"bytes": n_w * k * 2 + m * k * 4 + m * n_w * 4 * (2 if case["splits"] > 1 else 1),
                "flops": 2.0 * m * n_w * k}
    layers, d, f, phones, dtype = MODELS[case["model"]]
    wb = 2 if dtype == "bf16" else 4
    b, n, t = case["batch"], case["n"], case["tokens"]
    prompt = (case["ph_lo"] + case["ph_hi"] + case["ac_lo"] + case["ac_hi"]) / 2
    block = 4 * d * d + 2 * d * f
    kv = layers * d * 2 * 2                       # bytes of one position's keys and values
    steps = -(-t // n)
    bytes_ = layers * block * wb + b * prompt * kv                           # prefill
    bytes_ += steps * (layers * block * wb + n * V * d * wb + b * (prompt + t / 2) * kv) + b * t * kv
    flops = 2.0 * b * (prompt + t) * layers * block + 2.0 * b * steps * n * V * d
    flops += 4.0 * b * layers * d * (prompt * prompt / 2 + t * (prompt + t / 2))
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "viterbi":
        return "exact"               # one fp32 add at a time, in a stated order
    if kind == "heads":
        return {"rel": 5e-6, "max": 1e-4, "differ": 1e-3}   # fp32 sums of 1024 products; ids: near-ties
    if kind == "attention":
        return {"rel": 1.5e-5, "max": 4e-4}  # fp32 softmax, P and Q as two bf16 parts
    if kind == "gemm":
        return {"rel": 1e-5, "max": 1e-4}    # fp32 sums of exact bf16 products
    # whole models: every layer's activations and cache entries round on their own path
    # (measured 4e-6 from 64 bits, 3e-6 between two runs, whose split sums add in another order)
    return {"rel": 2e-5, "max": 2e-4, "differ": 5e-3}


# ---- the same in 64 bits ----


def _layer_norm(x, g, b):
    mu = x.mean(-1, keepdim=True)
    return (x - mu) / torch.sqrt(((x - mu) ** 2).mean(-1, keepdim=True) + 1e-5) * g + b


class _Reference:
    """The decoder over one sequence in float64; keys and values are kept in bf16, as the cache stores them."""

    def __init__(self, name):
        self.layers, self.d, _, _, _ = MODELS[name]
        ts = [t.double() for t, _ in _tensors(name)]
        self.phone, self.codec = ts[0], ts[1]
        self.block = [ts[2 + 12 * i:14 + 12 * i] for i in range(self.layers)]
        self.lnf, self.heads, self.bias = ts[-5:-3], ts[-3], ts[-2]
        self.log_q = ts[-1].float()

    def start(self):
        self.k, self.v, self.len = [None] * self.layers, [None] * self.layers, 0

    def feed(self, x):
        """Embedded rows [m][d] -> final hidden rows."""
        m, h = x.shape[0], self.d // HD
        pos = torch.arange(self.len, self.len + m, device="cuda", dtype=torch.float64)
        freq = torch.exp(torch.arange(0, self.d, 2, device="cuda", dtype=torch.float64) * (-math.log(10000.0) / self.d))
        ang = pos[:, None] * freq
        x = x + torch.stack([torch.sin(ang), torch.cos(ang)], -1).flatten(1)
        keys = torch.arange(self.len + m, device="cuda")
        hidden = keys[None, :] > pos[:, None]
        for i, (g1, b1, wqkv, bqkv, wo, bo, g2, b2, w1, c1, w2, c2) in enumerate(self.block):
            q, k, v = (_layer_norm(x, g1, b1) @ wqkv.T + bqkv).view(m, 3, h, HD).permute(1, 2, 0, 3)
            k, v = k.float().bfloat16().double(), v.float().bfloat16().double()
            self.k[i] = k if self.k[i] is None else torch.cat([self.k[i], k], 1)
            self.v[i] = v if self.v[i] is None else torch.cat([self.v[i], v], 1)
            a = (q @ self.k[i].transpose(1, 2) / 8.0).masked_fill(hidden, -math.inf)
            o = (torch.softmax(a, -1) @ self.v[i]).transpose(0, 1).reshape(m, self.d)
            x = x + o @ wo.T + bo
            u = _layer_norm(x, g2, b2) @ w1.T + c1
            x = x + (0.5 * u * (1.0 + torch.erf(u / math.sqrt(2.0)))) @ w2.T + c2
        self.len += m
        return x

    def logits(self, h, n):
        z = _layer_norm(h, *self.lnf)
        return torch.einsum("nvd,d->nv", self.heads[:n], z) + self.bias[:n]

    def path(self, logits, k):
        """Viterbi over the heads' top-k candidates."""
        s, ids = torch.sort((logits - torch.logsumexp(logits, -1, keepdim=True)).float(), dim=-1, descending=True,
                            stable=True)
        s, ids = s[:, :k], ids[:, :k]
        delta, back = s[0], []
        for t in range(1, logits.shape[0]):
            best, arg = (delta[:, None] + self.log_q[ids[t - 1]][:, ids[t]]).max(0)
            back.append(arg)
            delta = best + s[t]
        j = int(delta.argmax())
        out = [int(ids[-1, j])]
        for t in range(logits.shape[0] - 1, 0, -1):
            j = int(back[t - 1][j])
            out.append(int(ids[t - 1, j]))
        return out[::-1]


def _exact_request(case, seed):
    if case["batch"] > 40:
        return None
    ref = _Reference(case["model"])
    n, k, t = case["n"], case["k"], case["tokens"]
    all_logits = []
    for ph, ac in _prompts(case, seed):
        ref.start()
        h = ref.feed(torch.cat([ref.phone[ph.long()], ref.codec[ac.long()]]))[-1]
        done = 0
        while True:
            lg = ref.logits(h, n)
            path = ref.path(lg, k)
            done += n
            if done >= t:
                break
            h = ref.feed(ref.codec[torch.tensor(path, device="cuda")])[-1]
        all_logits.append(lg)
    lg = torch.stack(all_logits)
    return {"tokens": None, "lens": None, "logits": lg, "lse": torch.logsumexp(lg, -1)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "viterbi":
        ids, lp, _ = _viterbi_inputs(case, seed)
        ids, lp, q = ids.long(), lp.double(), _log_q().double()
        delta = lp[:, 0]
        for t in range(1, case["n"]):
            delta = (delta[:, :, None] + q[ids[:, t - 1, :, None], ids[:, t, None, :]]).amax(1) + lp[:, t]
        return {"path": None, "score": delta.amax(1), "accepted": None, "rollback": None}
    if kind == "heads":
        ts = [t.double() for t, _ in _tensors("valle_heads")]
        n = case["n"]
        z = _layer_norm(_hidden(case, seed).double(), ts[-5], ts[-4])
        lg = torch.einsum("nvd,bd->bnv", ts[-3][:n], z) + ts[-2][:n]
        lse = torch.logsumexp(lg, -1)
        logp = torch.topk(lg - lse[..., None], case["k"], dim=-1).values
        return {"ids": None, "logp": logp, "lse": lse, "logits": lg if case["logits"] else None}
    if kind == "attention":
        i = _attention_inputs(case, seed)
        out = torch.empty(i.rows, i.heads, HD, dtype=torch.float64, device="cuda")
        for s, c in enumerate(i.ctx):
            rows = (i.seq == s).nonzero().flatten()
            kv = i.pool[i.table[s].long(), 0].double().permute(1, 2, 0, 3, 4).flatten(2, 3)[:, :, :int(c)]
            q = i.q[rows].double().view(len(rows), i.heads, HD).transpose(0, 1)
            a = q @ kv[0].transpose(1, 2) / 8.0
            a = a.masked_fill(torch.arange(int(c), device="cuda")[None, :] > i.pos[rows][:, None], -math.inf)
            out[rows] = (torch.softmax(a, -1) @ kv[1]).transpose(0, 1)
        return out.flatten(1)
    if kind == "gemm":
        w, hi, lo, base = _gemm_inputs(case, seed)
        out = (hi.double() + lo.double()) @ w.double().T
        return out if base is None else out + base.double()
    if case["verify"]:
        return None
    return _exact_request(case, seed)
