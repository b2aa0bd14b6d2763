"""Timed cases of the graded KV-cache path: what a serving program has this library do.

Five kinds of pass, each through the binding's public calls:

  read      one decode step's attention over caches that are in place: `gkv_decode_attn` of every layer
  observe   the same with block masses and the error certificate: `gkv_decode_attn_observe` of every layer
  quest     page selection and the read of the selected pages, every layer
  latent    `read` on 576-wide latent streams (keys and values in one row, 16 heads)
  request   a whole request: a cache is made, the prompt of every layer is ingested, then `steps` decode
            steps append one token per sequence (demoting blocks as they age) and attend, and the cache is
            released.  `steps` = 0 is a prefill: the prompt is ingested and attended once.

A case gives the shape (layers, batch, query and KV heads, context), the ladder (rung widths in tokens,
newest first, or a bit budget for the rate-distortion policy) and the options.  Inputs follow the package's
synthetic workloads: outlier key channels, slow drift, topical clusters for the page scorer, prompt masses.
"""
import math

import numpy as np
import torch

from paper_2608_23599_b200 import binding as B

BLOCK, GROUP = 64, 32
LATENT_SCALE = 1.0 / math.sqrt(192.0)


def _case(name, kind, layers, batch, n_q, n_kv, ctx, *, w16=0, w8=0, w4=0, w2=0, budget=0.0, retire=0, residual=0.0,
          page=0, select=0, reduce_sum=False, drift=0.0, steps=0):
    c = dict(kind=kind, layers=layers, batch=batch, n_q=n_q, n_kv=n_kv, ctx=ctx, w16=w16, w8=w8, w4=w4, w2=w2,
             budget=budget, retire=retire, residual=residual, page=page, select=select, reduce_sum=reduce_sum,
             drift=drift, steps=steps)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a short chat turn on a small model: one layer's call, all latency
        _case("read_tiny", "read", 1, 1, 8, 2, 1000, w16=256, w8=256, w4=256, w2=128),
        # single-user decode of a 3B model: rate-distortion ladder, 1 % exact residual rows, eight query heads a KV head
        _case("read_rd_residual", "read", 8, 1, 16, 2, 16384, budget=5.3437, retire=512, residual=0.01, drift=0.05),
        # batched serving of an 8B model, every rung of the ladder in use, ragged last block
        _case("read_llama_32k", "read", 2, 8, 32, 8, 32757, w16=1024, w8=4096, w4=16384, w2=8192, drift=0.05),
        # decode that watches its attention mass (the steps before a re-allocation), with the certificate
        _case("observe_8k", "observe", 4, 2, 32, 8, 8200, budget=5.0, retire=256, drift=0.02),
        # page selection with small pages: many scores, few tokens read
        _case("quest_16", "quest", 2, 4, 32, 8, 32768 + 40, budget=4.5391, retire=64, page=16, select=2048),
        # page selection as the paper sets it: 64-token pages, 12.5 % of them, a wide graded base
        _case("quest_64", "quest", 4, 4, 32, 8, 32768 + 17, budget=10.2168, retire=64, page=64, select=4096),
        # latent attention, one sequence of a million tokens
        _case("latent_1m", "latent", 1, 1, 16, 1, 1048576, w16=4096, w8=300032, w4=482304),
        # latent attention, a batch of ordinary contexts
        _case("latent_batch", "latent", 4, 8, 16, 1, 8191, w16=512, w8=2048, w4=4096),
        # prefill of a batch under the staircase: every block encoded once
        _case("prefill_llama", "request", 2, 8, 32, 8, 32768, w16=1024, w8=4096, w4=16384, w2=8192, drift=0.05),
        # prefill under the rate-distortion policy with exact residual rows
        _case("prefill_rd", "request", 4, 4, 32, 8, 16384 + 21, budget=5.3437, retire=512, residual=0.01, drift=0.05),
        # a whole request: prompt, then decode steps that fill and demote blocks
        _case("request_2k", "request", 2, 2, 8, 2, 2048 - 30, w16=128, w8=384, w4=768, w2=512, drift=0.05, steps=96),
        # a whole request on latent streams
        _case("request_latent", "request", 2, 2, 16, 1, 16384 - 13, w16=512, w8=4096, w4=8192, steps=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _widths(rng, ctx):
    """Rung widths in whole blocks that leave the oldest tokens to the centroid rung, or not."""
    parts = [rng.uniform(0.03, 0.2), rng.uniform(0.05, 0.4), rng.uniform(0.1, 0.5), rng.uniform(0.0, 0.4)]
    return [max(1, int(p * ctx / BLOCK)) * BLOCK for p in parts]


def draw(rng):
    kind = rng.choice(["read", "read", "observe", "quest", "latent", "request", "request", "request"])
    if kind == "latent" or (kind == "request" and rng.random() < 0.33):
        batch = rng.choice([1, 2, 3, 8])
        prompt = kind == "request"
        ctx = _log_int(rng, 512, (65536 if prompt else 262144) // batch)
        w = _widths(rng, ctx)
        return _case("", kind, rng.choice([1, 2]), batch, 16, 1, ctx, w16=w[0], w8=w[1], w4=w[2],
                     steps=rng.choice([0, 8, 32]) if prompt else 0)
    n_q, n_kv = rng.choice([(8, 2), (16, 2), (32, 8), (12, 4), (14, 2), (8, 8)])
    batch = rng.choice([1, 2, 3, 4])
    layers = rng.choice([1, 2, 3])
    steps = rng.choice([0, 0, 32, 80]) if kind == "request" else 0
    top = 4096 if steps else 32768
    ctx = _log_int(rng, 300, top)
    w = _widths(rng, ctx)
    if kind == "quest":
        page = rng.choice([16, 32, 64])
        ctx = _log_int(rng, 2048, top)
        select = max(page, int(ctx * rng.uniform(0.05, 0.15)) // page * page)
        return _case("", kind, layers, batch, n_q, n_kv, ctx, budget=rng.choice([4.5, 6.0, 10.2]), retire=64,
                     page=page, select=select, reduce_sum=rng.random() < 0.3)
    if kind == "observe" or rng.random() < 0.4:
        return _case("", kind, layers, batch, n_q, n_kv, ctx, budget=rng.uniform(4.0, 8.0), retire=rng.choice([64, 256, 512]),
                     residual=rng.choice([0.0, 0.01, 0.03]), drift=0.02, steps=steps)
    if rng.random() < 0.25:      # a near-centroid base with many exact rows
        return _case("", kind, layers, batch, n_q, n_kv, ctx, w16=256, residual=0.10, drift=0.05, steps=steps)
    return _case("", kind, layers, batch, n_q, n_kv, ctx, w16=w[0], w8=w[1], w4=w[2], w2=w[3], drift=0.05, steps=steps)


# ---- inputs --------------------------------------------------------------------------------------
def _is_latent(c):
    return c["n_kv"] == 1        # one 576-wide row per token serves all 16 heads


def _dims(c):
    return (576, 512) if _is_latent(c) else (128, 128)


def _config(c):
    dk, dv = _dims(c)
    return B.make_config(
        c["layers"], c["batch"], c["n_q"], c["n_kv"], dk, dv, c["ctx"] + max(c["steps"], 64),
        v_aliases_k=1 if _is_latent(c) else 0, page_tokens=c["page"],
        policy=B.POLICY_RD if c["budget"] > 0 else B.POLICY_STAIRCASE, stair_tokens=(c["w16"], c["w8"], c["w4"], c["w2"]),
        retire_after=c["retire"], rd_budget_bpv=c["budget"], residual_fraction=c["residual"],
        quest_reduce=B.REDUCE_SUM if c["reduce_sum"] else B.REDUCE_MAX,
        softmax_scale=LATENT_SCALE if _is_latent(c) else 0.0)


def _inputs(c, seed):
    """Prompt rows, prompt masses, decode rows and queries of every layer, from the seed alone."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    dk, dv = _dims(c)
    b, h, hq, t, n = c["batch"], c["n_kv"], c["n_q"], c["ctx"], c["steps"]
    latent = _is_latent(c)

    def randn(*shape, dtype=torch.float32):
        return torch.randn(shape, generator=g, device=dev, dtype=dtype)

    gain = torch.ones(dk, device=dev)
    layers = []
    for _ in range(c["layers"]):
        perm = torch.randperm(dk, generator=g, device=dev)
        scale = gain.clone()
        scale[perm[: 8 if latent else 4]] = 6.0 if latent else 8.0
        q = randn(max(n, 1), b, hq, dk)
        if c["page"]:
            centres = randn(64, dk)
            n_pages = -(-t // c["page"])
            new_topic = torch.rand((b, n_pages, h), generator=g, device=dev) < 1.0 / 8.0
            topic = torch.cumsum(new_topic.long(), dim=1)
            pick = torch.randint(0, 64, (b, n_pages + 1, h), generator=g, device=dev)
            cluster = torch.gather(pick, 1, topic).repeat_interleave(c["page"], dim=1)[:, :t]
            k = centres[cluster] + 0.3 * randn(b, t, h, dk)
            q = centres[torch.randint(0, 64, (max(n, 1), b, hq), generator=g, device=dev)] + 0.5 * q
        else:
            k = randn(b, t, h, dk)
        k.mul_(scale)
        v = None if latent else randn(b, t, h, dv)
        if c["drift"] > 0:
            k += torch.cumsum(c["drift"] * randn(b, t, h, dk), dim=1)
            v += torch.cumsum(c["drift"] * randn(b, t, h, dv), dim=1)
        mass = None
        if c["budget"] > 0 or c["residual"] > 0:
            # a few tokens hold most of the prompt's attention, the newest ones a little more than the rest
            logits = 1.5 * randn(b, h, t) + 2.0 * torch.linspace(-1, 0, t, device=dev)
            mass = torch.softmax(logits, dim=-1)
        k_step = [(randn(b, 1, h, dk) * scale).bfloat16() for _ in range(n)]
        v_step = [None if latent else randn(b, 1, h, dv).bfloat16() for _ in range(n)]
        layers.append(dict(k=k.bfloat16(), v=None if latent else v.bfloat16(), mass=mass,
                           q=list(q.bfloat16().unbind(0)), k_step=k_step, v_step=v_step))
        del k, v
    return layers


def prepare(case, seed):
    data = _inputs(case, seed)
    cfg = _config(case)
    dk, dv = _dims(case)
    b, h, hq, n = case["batch"], case["n_kv"], case["n_q"], max(case["steps"], 1)
    dev = torch.device("cuda")
    s = dict(case=case, cfg=cfg, data=data)
    s["out"] = [torch.empty((b, hq, dv), dtype=torch.float32, device=dev) for _ in range(case["layers"] * n)]
    s["lse"] = [torch.empty((b, hq), dtype=torch.float32, device=dev) for _ in range(case["layers"] * n)]
    if case["kind"] != "request":
        s["cache"] = B.Cache(cfg)
        for l, d in enumerate(data):
            s["cache"].gkv_append_demote(l, d["k"], d["v"], token_mass=d["mass"])
        s["q"] = [d["q"][0] for d in data]
        del s["data"]              # the prompt's rows are gone once they are ingested
    if case["kind"] == "observe":
        items = -(-case["ctx"] // BLOCK)
        s["mass"] = [torch.empty((b, h, items), dtype=torch.float32, device=dev) for _ in range(case["layers"])]
        s["cert"] = [torch.empty((b, hq), dtype=torch.float32, device=dev) for _ in range(case["layers"])]
    if case["kind"] == "quest":
        k = min(case["select"] // case["page"], case["ctx"] // BLOCK * (BLOCK // case["page"]))
        s["pages"] = [torch.zeros((b, h, k), dtype=torch.int32, device=dev) for _ in range(case["layers"])]
    return s


# ---- one pass ------------------------------------------------------------------------------------
def run(state):
    case, out, lse = state["case"], state["out"], state["lse"]
    kind, layers = case["kind"], case["layers"]
    if kind == "request":
        cache = B.Cache(state["cfg"])
        data = state["data"]
        for l in range(layers):
            cache.gkv_append_demote(l, data[l]["k"], data[l]["v"], token_mass=data[l]["mass"])
            if case["steps"] == 0:
                cache.gkv_decode_attn(l, data[l]["q"][0], out[l], lse[l])
        for i in range(case["steps"]):
            for l in range(layers):
                cache.gkv_append_demote(l, data[l]["k_step"][i], data[l]["v_step"][i])
                cache.gkv_decode_attn(l, data[l]["q"][i], out[i * layers + l], lse[i * layers + l])
        cache.close()
        return {"out": torch.stack(out), "lse": torch.stack(lse)}
    cache, q = state["cache"], state["q"]
    if kind == "observe":
        for l in range(layers):
            cache.gkv_decode_attn_observe(l, q[l], out[l], lse[l], state["mass"][l], state["cert"][l])
        return {"out": out, "lse": lse, "mass": state["mass"], "cert": state["cert"]}
    if kind == "quest":
        pages = state["pages"]
        for l in range(layers):
            n_sel = cache.gkv_quest_select(l, q[l], case["select"], pages[l])
            cache.gkv_decode_attn(l, q[l], out[l], lse[l], page_idx=pages[l], n_sel=n_sel)
        return {"out": out, "lse": lse, "pages": pages}
    for l in range(layers):
        cache.gkv_decode_attn(l, q[l], out[l], lse[l])
    return {"out": out, "lse": lse}


# ---- what a pass cannot do without ----------------------------------------------------------------
def _graded_bytes(c, ctx):
    """Stored bytes of one (layer, sequence, KV head) stream of ctx tokens, residual rows included."""
    dk, dv = _dims(c)
    row = dk if _is_latent(c) else dk + dv
    if c["budget"] > 0:
        graded = min(c["budget"], 16.0) * ctx * row / 8
    else:
        left, graded = ctx, 0.0
        for width, bits in ((c["w16"], 16), (c["w8"], 9), (c["w4"], 5), (c["w2"], 3)):
            n = left if width < 0 else min(left, width)
            graded += n * row * bits / 8
            left -= n
        graded += left * row * 0.25 / 8
    return graded + math.floor(c["residual"] * ctx) * row * 2


def work(case):
    c = case
    dk, dv = _dims(c)
    streams = c["layers"] * c["batch"] * c["n_kv"]
    heads = c["layers"] * c["batch"] * c["n_q"]
    io = heads * (dk * 2 + dv * 4 + 4)
    row = dk if _is_latent(c) else dk + dv

    def read(ctx):
        return streams * _graded_bytes(c, ctx) + io, heads * ctx * 2 * (dk + dv)

    if c["kind"] == "quest":
        pages = c["ctx"] // c["page"]
        per_token = c["budget"] * row / 8
        bytes_ = streams * (pages * dk * 4 + c["select"] * per_token + (c["ctx"] % BLOCK) * row * 2) + io
        return {"bytes": bytes_, "flops": heads * (pages * dk * 2 + c["select"] * 2 * (dk + dv))}
    if c["kind"] != "request":
        bytes_, flops = read(c["ctx"])
        return {"bytes": bytes_, "flops": flops}
    bytes_ = streams * (c["ctx"] * row * 2 + _graded_bytes(c, c["ctx"]))
    flops = 0.0
    for i in range(max(c["steps"], 1)):
        b, f = read(c["ctx"] + (i + 1 if c["steps"] else 0))
        bytes_, flops = bytes_ + b, flops + f
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    # operands are fp16 / bf16 pairs with fp32 sums: four times the error measured against exact()
    return {"rel": 2.5e-4, "max": 1e-2, "differ": 1e-3 if case["kind"] == "quest" else 0.0}


# ---- the same in 64 bits ---------------------------------------------------------------------------
# Codes, scales, centroids, levels, residual rows and page scores are defined by 32-bit arithmetic in a fixed
# order and are made that way here; attention over what they stand for is in 64 bits.
def _quantise(x, bits):
    """x fp32 [..., 32]: what the codes of each group of 32 stand for, fp32."""
    top = float(2 ** bits - 1)
    lo, hi = x.amin(-1, keepdim=True), x.amax(-1, keepdim=True)
    s = ((hi - lo) / top).clamp(-65504.0, 65504.0).half().float()
    z = lo.clamp(-65504.0, 65504.0).half().float()
    inv = torch.where(s > 0, 1.0 / s, torch.zeros_like(s))
    code = torch.round((x - z) * inv).clamp(0.0, top)
    return code * s + z


def _encode(x, level, key):
    """Blocks x fp32 [n][64][d] as stored at `level`, fp32."""
    if level == 16:
        return x
    n, _, d = x.shape
    if level == 1:
        acc = torch.zeros_like(x[:, 0])
        for t in range(BLOCK):
            acc = acc + x[:, t]
        return (acc * (1.0 / BLOCK)).bfloat16().float()[:, None].expand(n, BLOCK, d).contiguous()
    if key:
        g = x.view(n, 2, GROUP, d).transpose(2, 3).contiguous()
        return _quantise(g, level).transpose(2, 3).reshape(n, BLOCK, d)
    return _quantise(x.view(n, BLOCK, d // GROUP, GROUP), level).view(n, BLOCK, d)


def _encode_levels(x, levels, key):
    out = torch.empty_like(x)
    for level in (16, 8, 4, 2, 1):
        at = (levels == level).nonzero()[:, 0]
        if len(at):
            out[at] = _encode(x[at], level, key)
    return out


def _staircase(c, n):
    lv = np.ones(n, dtype=np.int64)
    age = n - 1 - np.arange(n)
    edge = 0
    done = np.zeros(n, dtype=bool)
    for width, level in ((c["w16"], 16), (c["w8"], 8), (c["w4"], 4), (c["w2"], 2)):
        edge += width // BLOCK
        here = ~done & (age < edge)
        lv[here] = level
        done |= here
    return lv


def _allocate(c, mass, rng, n_tail):
    """Rate-distortion levels of one stream: the smallest threshold whose monotone plan fits the budget."""
    n = len(mass)
    y = mass.astype(np.float64) * rng.astype(np.float64)
    pinned = (n - 1 - np.arange(n)) < c["retire"] // BLOCK
    row = 256
    total = math.floor(float(np.float32(c["budget"])) * float((n * BLOCK + n_tail) * row))
    bits = {16: 16 * BLOCK * row, 8: 9 * BLOCK * row, 4: 5 * BLOCK * row, 2: 3 * BLOCK * row, 1: 16 * row}

    def plan(tau):
        lv = np.where(y <= tau, 1, np.where(y <= tau * 3.0, 2, np.where(y <= tau * 15.0, 4, np.where(y <= tau * 255.0, 8, 16))))
        lv[pinned] = 16
        free = np.nonzero(~pinned)[0]
        lv[free] = np.minimum.accumulate(lv[free][::-1])[::-1]      # no level rises toward older blocks
        return lv

    def fits(lv):
        return sum(bits[int(v)] for v in lv) + n_tail * 16 * row <= total

    cand = np.unique(np.concatenate([[0.0], y, y / 3.0, y / 15.0, y / 255.0]))
    lo, hi = 0, len(cand)
    while lo < hi:
        mid = (lo + hi) // 2
        if fits(plan(cand[mid])):
            hi = mid
        else:
            lo = mid + 1
    return plan(cand[min(lo, len(cand) - 1)])


class _Stream:
    """One (layer, sequence, KV head): its blocks as stored, fp32, with levels and exact rows."""

    def __init__(self, c, k, v, mass):
        self.c, self.latent = c, v is None
        n = k.shape[0] // BLOCK
        kf, vf = k.float(), None if v is None else v.float()
        self.tail_k, self.tail_v = kf[n * BLOCK:], None if v is None else vf[n * BLOCK:]
        kb, vb = kf[: n * BLOCK].view(n, BLOCK, -1), None if v is None else vf[: n * BLOCK].view(n, BLOCK, -1)
        if c["budget"] > 0:
            acc = torch.zeros(n, device=k.device)
            for t in range(BLOCK):
                acc = acc + mass[: n * BLOCK].view(n, BLOCK)[:, t]
            rng = (kb.amax(1) - kb.amin(1)).amax(1) if n else acc
            lv = _allocate(c, acc.cpu().numpy(), rng.cpu().numpy(), k.shape[0] - n * BLOCK) if n else np.ones(0, np.int64)
        else:
            lv = _staircase(c, n)
        self.levels = torch.from_numpy(lv).to(k.device)
        self.k = _encode_levels(kb, self.levels, True)
        self.v = None if v is None else _encode_levels(vb, self.levels, False)
        self.lo = self.hi = None
        if c["page"]:
            pages = kb.reshape(n * (BLOCK // c["page"]), c["page"], -1)
            self.lo, self.hi = pages.amin(1), pages.amax(1)
        self.exact = (self.levels == 16)[:, None].expand(n, BLOCK).clone()
        count = math.floor(float(np.float32(c["residual"])) * k.shape[0]) if mass is not None else 0
        if count:
            err = (vb.double() - _encode(vb, 1, False).double()).square().sum(-1)
            score = (mass[: n * BLOCK].view(n, BLOCK).double() * err).float().masked_fill(self.exact, -1.0).view(-1)
            count = min(count, int((~self.exact).sum()))
            at = torch.sort(score, descending=True, stable=True).indices[:count]
            self.k.view(n * BLOCK, -1)[at] = kf[at]
            self.v.view(n * BLOCK, -1)[at] = vf[at]
            self.exact.view(-1)[at] = True
        if c["kind"] == "observe":
            lost = (~self.exact).double()
            self.kappa = self._norm(kb, _encode_levels(kb, self.levels, True))
            self.delta = self._norm(vb, _encode_levels(vb, self.levels, False))
            self.lost = lost
            self.vmax = vf.double().square().sum(-1).sqrt().max()

    @staticmethod
    def _norm(x, y):
        return (x.double() - y.double()).square().sum(-1).sqrt().amax(1)

    def append(self, k, v):
        self.tail_k = torch.cat([self.tail_k, k.float()])
        self.tail_v = None if v is None else torch.cat([self.tail_v, v.float()])
        if len(self.tail_k) < BLOCK:
            return
        self.k = torch.cat([self.k, self.tail_k[None]])
        self.v = None if v is None else torch.cat([self.v, self.tail_v[None]])
        self.levels = torch.cat([self.levels, self.levels.new_full((1,), 16)])
        self.tail_k = self.tail_k[:0]
        self.tail_v = None if v is None else self.tail_v[:0]
        if self.c["budget"] > 0:
            return
        target = torch.from_numpy(_staircase(self.c, len(self.levels))).to(self.levels.device)
        for b in (target < self.levels).nonzero()[:, 0].tolist():
            level = int(target[b])
            self.k[b] = _encode(self.k[b: b + 1], level, True)[0]
            if v is not None:
                self.v[b] = _encode(self.v[b: b + 1], level, False)[0]
            self.levels[b] = level

    def attend(self, q, mask=None):
        """q fp64 [g][dk]: (out [g][dv], lse [g], weights [g][T])."""
        k = torch.cat([self.k.reshape(-1, self.k.shape[-1]), self.tail_k]).double()
        scale = float(np.float32(LATENT_SCALE if self.latent else 1.0 / math.sqrt(q.shape[1])))
        logits = (q @ k.T) * scale
        if mask is not None:
            logits = logits.masked_fill(~mask, -math.inf)
        lse = torch.logsumexp(logits, dim=1)
        w = torch.exp(logits - lse[:, None])
        v = k[:, :512] if self.latent else torch.cat([self.v.reshape(-1, self.v.shape[-1]), self.tail_v]).double()
        return w @ v, lse, w

    def select(self, q):
        """Pages the selection keeps for q fp32 [g][dk], ascending."""
        acc = torch.zeros((q.shape[0], self.lo.shape[0]), device=q.device)
        for d in range(q.shape[1]):
            pick = torch.where(q[:, d: d + 1] >= 0, self.hi[:, d], self.lo[:, d])
            acc = acc + q[:, d: d + 1] * pick
        score = acc[0]
        for j in range(1, q.shape[0]):
            score = score + acc[j] if self.c["reduce_sum"] else torch.maximum(score, acc[j])
        k = min(self.c["select"] // self.c["page"], self.lo.shape[0])
        return torch.sort(torch.sort(score + 0.0, descending=True, stable=True).indices[:k]).values

    def masses(self, w):
        t = w.shape[1]
        pad = torch.zeros((w.shape[0], -t % BLOCK), dtype=w.dtype, device=w.device)
        return torch.cat([w, pad], dim=1).view(w.shape[0], -1, BLOCK).sum(-1).mean(0)

    def certificate(self, w, q):
        n = len(self.levels)
        scale = float(np.float32(1.0 / math.sqrt(q.shape[1])))
        a = (w[:, : n * BLOCK].view(-1, n, BLOCK) * self.lost).sum(-1)
        sure = 1.0 - a.sum(-1)
        eps = scale * q.square().sum(-1).sqrt()[:, None] * self.kappa
        up, down = sure + (a * eps.exp()).sum(-1), sure + (a * (-eps).exp()).sum(-1)
        return (a * self.delta).sum(-1) + (up / down - down / up).clamp(max=2.0) * self.vmax


def exact(case, seed):
    c = case
    data = _inputs(c, seed)
    dk, dv = _dims(c)
    b, h, hq, n = c["batch"], c["n_kv"], c["n_q"], max(c["steps"], 1)
    g = hq // h
    dev = torch.device("cuda")
    out = [torch.empty((b, hq, dv), dtype=torch.float64, device=dev) for _ in range(c["layers"] * n)]
    lse = [torch.empty((b, hq), dtype=torch.float64, device=dev) for _ in range(c["layers"] * n)]
    mass = [torch.empty((b, h, -(-c["ctx"] // BLOCK)), dtype=torch.float64, device=dev) for _ in range(c["layers"])]
    cert = [torch.empty((b, hq), dtype=torch.float64, device=dev) for _ in range(c["layers"])]
    pages = [[[None] * h for _ in range(b)] for _ in range(c["layers"])]
    for l, d in enumerate(data):
        for i in range(b):
            for j in range(h):
                st = _Stream(c, d["k"][i, :, j], None if d["v"] is None else d["v"][i, :, j],
                             None if d["mass"] is None else d["mass"][i, j])
                heads = slice(j * g, (j + 1) * g)
                for s in range(n):
                    at = s * c["layers"] + l
                    if c["steps"]:
                        st.append(d["k_step"][s][i, :, j], None if d["v"] is None else d["v_step"][s][i, :, j])
                    q, mask = d["q"][s][i, heads], None
                    if c["kind"] == "quest":
                        sel = st.select(q.float())
                        pages[l][i][j] = sel.int()
                        mask = torch.zeros(c["ctx"], dtype=torch.bool, device=dev)
                        closed = mask[: c["ctx"] // BLOCK * BLOCK].view(-1, c["page"])
                        closed[sel] = True
                        mask[c["ctx"] // BLOCK * BLOCK:] = True
                    out[at][i, heads], lse[at][i, heads], w = st.attend(q.double(), mask)
                    if c["kind"] == "observe":
                        mass[l][i, j] = st.masses(w)
                        cert[l][i, heads] = st.certificate(w, q.double())
    if c["kind"] == "request":
        return {"out": torch.stack(out), "lse": torch.stack(lse)}
    if c["kind"] == "observe":
        return {"out": out, "lse": lse, "mass": mass, "cert": cert}
    if c["kind"] == "quest":
        return {"out": out, "lse": lse, "pages": [torch.stack([torch.stack(p) for p in x]) for x in pages]}
    return {"out": out, "lse": lse}
