"""What a user of this framework has it do, as cases that can be timed.

A case is one phase of an image generation (its "kind") on a model shape of
synth/configs.py, with the number of sequences, budget ratio, data type and,
where it is not the shape's own, the number of layers and conditioning tokens:

  period    one steady-state period of decoding: the update of every layer,
            then P tokens through every layer (one launch per layer step)
  unfused   the same period through append and attend, as an integration
            does that keeps its own attention call
  dense     one token through every layer of the uncompressed cache, with the
            head types decided in the same pass (the grouping token)
  identify  the head types of every layer as a pass of its own (labels, n_h)
  compress  budgets, arena and repack of every layer, then the first token
            over the compressed cache
  update    the periodic update of every layer, with the cache's counters and
            positions put back before it
  prefill   a new batch: the cache emptied, then the conditioning tokens of
            every layer written
  generate  whole generations through runner.generate, a new engine each

The phases of fixed shape (all but compress, update and generate) are CUDA
graphs captured once, as a serving loop keeps them.

Keys and queries carry the two-dimensional position of their token (queries
with a gain per head), so that heads differ in how far back they look and
both head types occur; values are normal.
"""
from __future__ import annotations

import math
from fractions import Fraction

import torch

from paper_2605_20600_gb300 import hkv as H
from paper_2605_20600_gb300.engine import CacheBuffers, Engine, torch_dtype
from paper_2605_20600_gb300.runner import generate
from synth import configs

GLOBAL_SHARE = 0.45  # of heads; about what the model shapes show at grouping


def listed():
    return [
        # one image with classifier-free guidance: the smallest serving batch
        dict(name="period_janus_b2", kind="period", model="janus_pro_7b", seqs=2, rho="1/8"),
        # the workload bench.py quotes: eight 1024-pixel images, a quarter of the cache
        dict(name="period_lumina1024_b8", kind="period", model="lumina1024", seqs=8, rho="1/4"),
        # many short heads of 64 channels: 64 images with guidance
        dict(name="period_llamagen_b128", kind="period", model="llamagen_xl", seqs=128, rho="1/6"),
        # a full card: 128 images with guidance
        dict(name="period_janus_b256", kind="period", model="janus_pro_7b", seqs=256, rho="1/8"),
        # single precision, an odd batch and an odd prompt length (rows of 512 bytes)
        dict(name="period_lumina768_b3_fp32", kind="period", model="lumina768", seqs=3, rho="1/6",
             dtype="fp32", n_cond=37),
        # append and attention as two calls, two images of 768 pixels with guidance
        dict(name="unfused_lumina768_b4", kind="unfused", model="lumina768", seqs=4, rho="1/4"),
        # the grouping token of the 1024-pixel workload
        dict(name="dense_lumina1024_b8", kind="dense", model="lumina1024", seqs=8, rho="1/4"),
        # head types as their own pass: what the unfused path and the labels study run
        dict(name="identify_lumina1024_b8", kind="identify", model="lumina1024", seqs=8, rho="1/4"),
        # grouping to compressed cache, 32 images with guidance
        dict(name="compress_janus_b64", kind="compress", model="janus_pro_7b", seqs=64, rho="1/8"),
        # the periodic update of the 1024-pixel workload
        dict(name="update_lumina1024_b8", kind="update", model="lumina1024", seqs=8, rho="1/4"),
        # prompts of the 1024-pixel workload
        dict(name="prefill_lumina1024_b8", kind="prefill", model="lumina1024", seqs=8, rho="1/4"),
        # one image with guidance from prompt to last token, launched call by call
        dict(name="generate_llamagen_b2", kind="generate", model="llamagen_xl", seqs=2, rho="1/6"),
    ]


# the most sequences a drawn case has (bf16; half in fp32)
_MOST_SEQS = {"lumina1024": 24, "lumina768": 32, "llamagen_xl": 192, "janus_pro_7b": 192}
_KINDS = ("period", "period", "period", "unfused", "dense", "identify", "compress", "update",
          "prefill", "generate")


def draw(rng):
    most = max(work(c)["bytes"] for c in listed())
    while True:
        kind = rng.choice(_KINDS)
        model = rng.choice(sorted(_MOST_SEQS))
        w = configs.ALL[model]
        dtype = rng.choice(("bf16", "bf16", "bf16", "fp32"))
        top = _MOST_SEQS[model] // (2 if dtype == "fp32" else 1)
        c = dict(kind=kind, model=model, rho=rng.choice(("1/4", "1/6", "1/8")), dtype=dtype,
                 seqs=round(math.exp(rng.uniform(0.0, math.log(top)))),
                 layers=rng.randint(2, w.n_layers),
                 n_cond=round(math.exp(rng.uniform(0.0, math.log(2 * w.n_cond + 8)))))
        if kind == "generate":  # the launches bound it: fewer layers, few sequences
            c["model"] = rng.choice(("llamagen_xl", "janus_pro_7b"))
            c["seqs"] = rng.randint(1, 6)
            c["layers"] = rng.randint(1, 8)
        if work(c)["bytes"] <= most:
            return c


# ---------------------------------------------------------------------------
# shapes
# ---------------------------------------------------------------------------
def _shape(case):
    w = configs.ALL[case["model"]]
    return w.with_(n_seqs=case["seqs"], rho=Fraction(case["rho"]), dtype=case.get("dtype", w.dtype),
                   n_layers=case.get("layers", w.n_layers), n_cond=case.get("n_cond", w.n_cond))


def _config(w):
    return H.make_config(n_layers=w.n_layers, n_seqs=w.n_seqs, n_heads=w.n_heads,
                         head_dim=w.head_dim, dtype=w.dtype, n_cond=w.n_cond, n_image=w.n_image,
                         row_len=w.row_len, recent_w=w.recent_w, local_w=w.w_loc, period=w.period,
                         group_at=w.group_at, rho=w.rho, tau=w.tau, r_s=w.r_s)


def _budget(w):
    return w.n_image * w.rho.numerator // w.rho.denominator


def _tokens_before(w):
    """Image tokens so far at the start of a steady-state period: every
    global head's history is full."""
    first = max(w.group_at, _budget(w)) + w.period
    return min(first + w.period, max(first, w.n_image - w.period))


def work(case):
    w = _shape(case)
    n, row = w.n_head_total, w.head_dim * w.elem_bytes
    out = 4 * w.head_dim
    C, P, E, B, N = w.n_cond, w.period, w.group_at, _budget(w), w.n_image
    kept = C + GLOBAL_SHARE * B + (1 - GLOBAL_SHARE) * w.recent_w  # rows of a head after its update

    def steps(count, rows):  # decode steps of every head over `rows` rows on average
        return (count * n * (2 * rows * row + 3 * row + 2 * row + row + out),
                count * n * 4 * w.head_dim * (rows + 1))

    # scores read every candidate of a global head, the moves about P rows
    upd = (n * (GLOBAL_SHARE * (C + B + P + P) * row + 4 * P * row + 4 * (kept + P)),
           n * GLOBAL_SHARE * 2 * w.head_dim * (B + P))
    kind = case["kind"]
    if kind in ("period", "unfused"):
        s = steps(P, kept + (P - 1) / 2)
        b, f = s[0] + upd[0], s[1] + upd[1]
    elif kind == "dense":
        b, f = steps(1, C + E - 1)
    elif kind == "identify":
        b, f = n * ((C + E + 1) * row + 5), n * 2 * w.head_dim * (C + E)
    elif kind == "compress":
        rows = C + GLOBAL_SHARE * min(B, E) + (1 - GLOBAL_SHARE) * w.recent_w
        trimmed = GLOBAL_SHARE if E > B else 0.0
        s = steps(1, rows)
        b = s[0] + n * (4 * rows * row + 8 * rows + trimmed * (E - B + P) * row)
        f = s[1] + n * trimmed * 2 * w.head_dim * E
    elif kind == "update":
        b, f = upd
    elif kind == "prefill":
        b, f = n * (4 * C * row + 4 * C + 33), 0.0
    else:  # dense steps, then compressed ones
        d = steps(E, C + E / 2)
        s = steps(N - E, C + GLOBAL_SHARE * min(B, N / 2) + (1 - GLOBAL_SHARE) * w.recent_w + P / 2)
        b, f = d[0] + s[0], d[1] + s[1]
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# inputs, from torch alone
# ---------------------------------------------------------------------------
def _generator(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(int(seed))


def _features(w, tokens):
    """[C + tokens, D]: sines and cosines of the token's grid row and column;
    conditioning tokens sit above the grid, one to a cell."""
    D = w.head_dim
    t = torch.arange(tokens, device="cuda")
    c = torch.arange(w.n_cond, device="cuda")
    row = torch.cat([-1 - c // w.row_len, t // w.row_len]).double()
    col = torch.cat([c % w.row_len, t % w.row_len]).double()
    f = 4.0 ** (-torch.arange(D // 4, device="cuda").double() / (D // 16))
    a, b = row[:, None] * f, col[:, None] * f
    return torch.cat([a.cos(), a.sin(), b.cos(), b.sin()], 1).float()


def _gains(w, g):
    """[L, 1, H, 1]: how sharply each head attends (log-uniform, as in the
    shapes' own heads), the same for every sequence."""
    x = torch.rand(w.n_layers, 1, w.n_heads, 1, generator=g, device="cuda")
    return torch.exp(math.log(0.1) + x * math.log(80.0))


def _normal(shape, dtype, g, scale=1.0):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, scale, generator=g)


def _stream_inputs(w, g, tokens, first):
    """q, k, v [tokens, L, S, H, D] of the image tokens from `first` on."""
    dt = torch.float32 if w.dtype == configs.FP32 else torch.bfloat16
    shape = (tokens, w.n_layers, w.n_seqs, w.n_heads, w.head_dim)
    pe = _features(w, first + tokens)[w.n_cond + first:]
    q, k, v = (_normal(shape, dt, g, s) for s in (0.2, 0.3, 1.0))
    gain = _gains(w, g)
    for t in range(tokens):
        k[t] += pe[t].to(dt)
        q[t] = (q[t].float() + gain * pe[t]).to(dt)
    return q, k, v


def _fill_rows(w, buf, pos, g):
    """Keys (the token's position plus noise) and values of every row of an
    arena whose rows are the tokens `pos` ([rows])."""
    buf.k.normal_(0.0, 0.3, generator=g)
    buf.v.normal_(0.0, 1.0, generator=g)
    pe = _features(w, int(pos.max()) + 1 - w.n_cond if pos.numel() else 0)
    step = 1 << 22
    for a in range(0, pos.numel(), step):
        buf.k[a:a + step] += pe[pos[a:a + step].long()].to(buf.k.dtype)


def _labels(w, g):
    """[L*S*H]: a head's type goes with its layer and index, not its sequence;
    every layer has the same number of global heads."""
    x = torch.rand(w.n_layers, 1, w.n_heads, generator=g, device="cuda")
    x = x.argsort(dim=2) < round(GLOBAL_SHARE * w.n_heads)
    return x.expand(-1, w.n_seqs, -1).reshape(-1).to(torch.uint8).contiguous()


def _dense_engine(w, g, tokens):
    """An engine whose uncompressed cache holds the conditioning tokens and
    `tokens` image tokens of every head, and its query ring the newest P."""
    eng = Engine(_config(w))
    seg = w.n_cond + w.group_at
    pos = torch.arange(seg, device="cuda", dtype=torch.int32).repeat(w.n_head_total)
    _fill_rows(w, eng.dense, pos, g)
    eng.dense.pos.copy_(pos)
    eng.dense.len.fill_(w.n_cond + tokens)
    eng.dense.ntok.fill_(tokens)
    _fill_ring(w, eng.dense.qbuf, g, tokens)
    return eng


def _fill_ring(w, qbuf, g, tokens):
    """The ring's queries: image token t in slot t mod P."""
    qbuf.normal_(0.0, 0.2, generator=g)
    pe = _features(w, tokens)[w.n_cond + tokens - w.period:]
    slots = torch.arange(tokens - w.period, tokens, device="cuda") % w.period
    gain = _gains(w, g).expand(w.n_layers, w.n_seqs, w.n_heads, 1).reshape(-1)
    ring = torch.empty_like(pe)
    ring[slots] = pe
    step = max(1, (1 << 28) // ring.numel())
    for a in range(0, qbuf.shape[0], step):
        qbuf[a:a + step] += (gain[a:a + step, None, None] * ring).to(qbuf.dtype)


def _steady_engine(w, g):
    """An engine in mid-generation: a compressed cache whose buffers hold P
    tokens, so that the update is due, and whose global histories are full."""
    cfg = _config(w)
    eng = Engine(cfg)
    eng.release_dense()
    eng.labels.copy_(_labels(w, g))
    n, dev = eng.n, eng.device
    eng.budget = torch.empty(n, dtype=torch.int32, device=dev)
    eng.cap = torch.empty(n, dtype=torch.int32, device=dev)
    eng.off = torch.empty(n, dtype=torch.int64, device=dev)
    eng.total_tokens = H.hkv_allocate_budgets(cfg, eng.labels, eng.budget, eng.cap, eng.off,
                                              eng.stream())
    eng.ragged = eng.cache = CacheBuffers(cfg, eng.total_tokens, dev, qbuf=eng.dense.qbuf,
                                          label=eng.labels, off=eng.off, cap=eng.cap)
    return eng


def _fill_steady(w, eng, g):
    tok = _tokens_before(w)
    C, B, P, rw = w.n_cond, _budget(w), w.period, w.recent_w
    c = eng.ragged
    dev = eng.device
    local = torch.cat([torch.arange(C, device=dev),
                       C + torch.arange(tok - rw - P, tok, device=dev)]).to(torch.int32)
    hist, span = B - rw, tok - rw - P  # a full history out of the older tokens
    at = torch.arange(hist, device=dev)
    lo, hi = at * span // max(hist, 1), (at + 1) * span // max(hist, 1)
    n_global = 16  # different histories, dealt out to the heads
    kinds = []
    for _ in range(n_global):
        pick = lo + (torch.rand(hist, generator=g, device=dev) * (hi - lo)).long()
        kinds.append(torch.cat([torch.arange(C, device=dev), C + pick,
                                C + torch.arange(tok - rw - P, tok, device=dev)]).to(torch.int32))
    table = torch.cat([local] + kinds)
    first = torch.cat([torch.zeros(1, dtype=torch.long, device=dev),
                       local.numel() + torch.arange(n_global, device=dev) * kinds[0].numel()])
    heads = torch.arange(eng.n, device=dev)
    kind = torch.where(eng.labels == 1, 1 + heads % n_global, 0)
    head = torch.repeat_interleave(heads, eng.cap.long())
    pos = table[first[kind][head] + torch.arange(head.numel(), device=dev) - eng.off[head]]
    _fill_rows(w, c, pos, g)
    c.pos.copy_(pos)
    c.len.copy_(eng.cap)
    c.nbuf.fill_(P)
    c.ntok.fill_(tok)
    _fill_ring(w, c.qbuf, g, tok)


def _graph(fn):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        fn()
    return g


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
class _Provider:
    """Hands runner.generate its inputs, as a model's projections would."""

    def __init__(self, kc, vc, q, k, v):
        self.kc, self.vc, self.q, self.k, self.v = kc, vc, q, k, v

    def cond(self, kc, vc, layer, stream):
        kc.copy_(self.kc[layer])
        vc.copy_(self.vc[layer])

    def image(self, q, k, v, l0, nl, t0, nt, stream):
        q.copy_(self.q[t0])
        k.copy_(self.k[t0])
        v.copy_(self.v[t0])


def _cond_inputs(w, g):
    dt = torch.float32 if w.dtype == configs.FP32 else torch.bfloat16
    shape = (w.n_layers, w.n_seqs, w.n_heads, w.n_cond, w.head_dim)
    kc, vc = _normal(shape, dt, g, 0.3), _normal(shape, dt, g)
    kc += _features(w, 0).to(dt)
    return kc, vc


def _make(case, seed):
    """The state before graphs are captured (and all that exact() reads)."""
    w, g = _shape(case), _generator(seed)
    kind = case["kind"]
    st = {"w": w, "kind": kind}
    P, L = w.period, w.n_layers
    out_shape = (w.n_layers, w.n_seqs, w.n_heads, w.head_dim)
    if kind in ("period", "unfused", "update"):
        eng = _steady_engine(w, g)
        if kind != "update":
            st["q"], st["k"], st["v"] = _stream_inputs(w, g, P, _tokens_before(w))
            st["out"] = torch.zeros((P,) + out_shape, device="cuda")
            # the first calls set the kernels up, over empty heads
            eng.evict_all()
            for layer in range(L):
                x = st["q"][0][layer], st["k"][0][layer], st["v"][0][layer]
                if kind == "unfused":
                    eng.append(layer, *x)
                    eng.attend(layer, x[0], st["out"][0][layer])
                else:
                    eng.step(layer, *x, st["out"][0][layer])
        _fill_steady(w, eng, g)
        if kind == "update":
            st["before"] = [t.clone() for t in (eng.ragged.pos, eng.ragged.len, eng.ragged.nbuf)]
    elif kind in ("dense", "identify"):
        eng = _dense_engine(w, g, w.group_at - (1 if kind == "dense" else 0))
        q, k, v = _stream_inputs(w, g, 1, w.group_at - 1)
        st["q"], st["k"], st["v"] = q[0], k[0], v[0]
        st["out"] = torch.zeros(out_shape, device="cuda")
        st["before"] = [eng.dense.len.clone(), eng.dense.ntok.clone()]
    elif kind == "compress":
        eng = _dense_engine(w, g, w.group_at)
        eng.labels.copy_(_labels(w, g))
        q, k, v = _stream_inputs(w, g, 1, w.group_at)
        st["q"], st["k"], st["v"] = q[0], k[0], v[0]
        st["out"] = torch.zeros(out_shape, device="cuda")
    elif kind == "prefill":
        eng = Engine(_config(w))
        for t in (eng.dense.k, eng.dense.v):
            t.zero_()
        st["kc"], st["vc"] = _cond_inputs(w, g)
    else:
        eng = None
        st["cfg"] = _config(w)
        st["provider"] = _Provider(*_cond_inputs(w, g), *_stream_inputs(w, g, w.n_image, 0))
        st["out"] = torch.zeros((w.n_image,) + out_shape, device="cuda")
    st["eng"] = eng
    return st


def _pass(st):
    """The calls of one pass of the kinds that are captured."""
    eng, w, kind = st["eng"], st["w"], st["kind"]
    if kind == "period":
        eng.evict_all()
        for t in range(w.period):
            q, k, v, out = (st[x][t] for x in ("q", "k", "v", "out"))
            for layer in range(w.n_layers):
                eng.step(layer, q[layer], k[layer], v[layer], out[layer])
    elif kind == "unfused":
        for t in range(w.period):
            q, k, v, out = (st[x][t] for x in ("q", "k", "v", "out"))
            for layer in range(w.n_layers):
                eng.append(layer, q[layer], k[layer], v[layer])
                eng.attend(layer, q[layer], out[layer])
    elif kind == "dense":
        eng.dense.len.copy_(st["before"][0])
        eng.dense.ntok.copy_(st["before"][1])
        for layer in range(w.n_layers):
            eng.step_identify(layer, st["q"][layer], st["k"][layer], st["v"][layer],
                              st["out"][layer])
    elif kind == "identify":
        for layer in range(w.n_layers):
            eng.identify(layer, st["q"][layer])
    else:  # prefill
        H.hkv_init_dense(eng.cfg, eng.dense.c, eng.stream())
        for layer in range(w.n_layers):
            eng.prefill(layer, st["kc"][layer], st["vc"][layer])


def prepare(case, seed):
    st = _make(case, seed)
    if st["kind"] in ("dense", "identify", "prefill"):
        _pass(st)  # the first calls set the kernels up; the pass leaves what it found
    if st["kind"] in ("period", "unfused", "dense", "identify", "prefill"):
        st["graph"] = _graph(lambda: _pass(st))
    return st


def run(st):
    eng, kind = st["eng"], st["kind"]
    if kind == "generate":
        eng = Engine(st["cfg"])
        out = st["out"]
        generate(eng, st["provider"], on_step=lambda t, o: out[t].copy_(o))
        return {"out": out, "label": eng.labels, "len": eng.cache.len, "ntok": eng.cache.ntok}
    if kind == "compress":
        eng.compress()
        for layer in range(st["w"].n_layers):
            eng.step(layer, st["q"][layer], st["k"][layer], st["v"][layer], st["out"][layer])
        c = eng.ragged
        return {"out": st["out"], "cap": eng.cap, "off": eng.off, "pos": c.pos, "len": c.len,
                "nbuf": c.nbuf, "ntok": c.ntok}
    if kind == "update":
        c = eng.ragged
        for t, b in zip((c.pos, c.len, c.nbuf), st["before"]):
            t.copy_(b)
        eng.evict_all()
    else:
        st["graph"].replay()
    if kind == "identify":
        return {"label": eng.labels, "n_h": eng.n_h}
    c = eng.cache
    got = {"k": c.k, "v": c.v, "pos": c.pos, "len": c.len, "nbuf": c.nbuf, "ntok": c.ntok}
    if kind == "dense":
        got["label"] = eng.labels
    if "out" in st:
        got["out"] = st["out"]
        got["qbuf"] = c.qbuf
    return got


# ---------------------------------------------------------------------------
# the same in 64 bits, from torch alone
# ---------------------------------------------------------------------------
def _ref_attend(K, V, live, q):
    """softmax(q k^T / sqrt(D)) v over the live rows; [n, rows, D], [n, D]."""
    s = torch.bmm(K, q[:, :, None])[:, :, 0] / math.sqrt(q.shape[1])
    s = s.masked_fill(~live, -math.inf)
    p = torch.softmax(s, 1)
    return torch.bmm(p[:, None], V)[:, 0], p


def _ref_update(w, K, pos, live, label, ring, tok):
    """The live rows the update keeps (Eqs. 2-6). Keys as they are stored;
    ring [n, P, D] with image token t in slot t mod P. Scores are ranked as
    fp32 sums in channel order, which is what the update is specified by."""
    C, P, rw, B = w.n_cond, w.period, w.recent_w, _budget(w)
    hist = live & (pos >= C) & (pos < C + max(tok - rw, 0))
    NH = hist.sum(1)
    M = torch.where(label == 1, (NH - (B - rw)).clamp(min=0), NH)
    evict = hist & (label != 1)[:, None]
    glob = torch.nonzero((label == 1) & (M > 0))[:, 0]
    if glob.numel() == 0:
        return live & ~evict
    big = 1 << 40
    for a in range(0, glob.numel(), 2048):
        g = glob[a:a + 2048]
        h, p, m, nh = hist[g], pos[g].long(), M[g], NH[g]
        qbar = torch.zeros(g.numel(), K.shape[2], device=K.device)
        for j in range(P):
            qbar = qbar + ring[g, (tok - P + j) % P].float()
        Kf = K[g].float()
        s = torch.zeros(h.shape, device=K.device)
        for d in range(K.shape[2]):
            s = s + qbar[:, d, None] * Kf[:, :, d]
        s = (s + 0.0).double()
        order = torch.where(h, p, big).argsort(dim=1)  # by position, others last
        rank = torch.empty_like(order).scatter_(1, order, torch.arange(h.shape[1], device=K.device)
                                                .expand_as(order).contiguous())
        n_long = (nh.double() * w.r_s).floor().long()
        n_near = nh - n_long
        long = h & (rank < n_long[:, None])
        near = h & ~long
        m_long, m_near = m // 2, m - m // 2
        over = (m_long - n_long).clamp(min=0)
        m_long, m_near = m_long - over, m_near + over
        over = (m_near - n_near).clamp(min=0)
        m_long, m_near = m_long + over, m_near - over
        for sub, quota in ((long, m_long), (near, m_near)):
            key = torch.where(sub, s, math.inf).gather(1, order)
            by = order.gather(1, torch.sort(key, dim=1, stable=True)[1])  # by score, then position
            r = torch.empty_like(by).scatter_(1, by, torch.arange(h.shape[1], device=K.device)
                                              .expand_as(by).contiguous())
            evict[g] |= sub & (r < quota[:, None])
    return live & ~evict


def _padded(c, heads, width):
    """[heads, width] arena rows of each head and which of them are live."""
    at = torch.arange(width, device="cuda")
    live = at < c.len[heads].long()[:, None]
    idx = torch.where(live, c.off[heads][:, None] + at, 0)
    return idx, live


def exact(case, seed):
    kind = case["kind"]
    if kind in ("identify", "update"):
        return None  # whole numbers and moved rows
    st = _make(case, seed)
    w, eng = st["w"], st["eng"]
    n, D, P, C = w.heads_per_layer, w.head_dim, w.period, w.n_cond
    if kind == "prefill":
        k, v = (torch.zeros(w.n_head_total, C + w.group_at, D, dtype=x.dtype, device="cuda")
                for x in (st["kc"], st["vc"]))
        k[:, :C] = st["kc"].reshape(-1, C, D)
        v[:, :C] = st["vc"].reshape(-1, C, D)
        return {"k": k.reshape(-1, D), "v": v.reshape(-1, D), "pos": None, "len": None,
                "nbuf": None, "ntok": None}
    out = torch.zeros(st["out"].shape, dtype=torch.float64, device="cuda")
    if kind == "generate":
        _exact_generate(st, out)
        return {"out": out, "label": None, "len": None, "ntok": None}
    c = eng.cache
    for layer in range(w.n_layers):
        heads = torch.arange(layer * n, (layer + 1) * n, device="cuda")
        label = eng.labels[heads]
        width = int(c.len[heads].max())
        idx, live = _padded(c, heads, width)
        pos = c.pos[idx]
        if kind in ("period", "unfused"):
            live = _ref_update(w, c.k[idx], pos, live, label, c.qbuf[heads], _tokens_before(w))
        elif kind == "compress":
            live = _ref_update(w, c.k[idx], pos, live, label, c.qbuf[heads], w.group_at)
        tokens = P if kind in ("period", "unfused") else 1
        K = torch.zeros(n, width + tokens, D, dtype=torch.float64, device="cuda")
        V = torch.zeros_like(K)
        K[:, :width], V[:, :width] = c.k[idx].double(), c.v[idx].double()
        live = torch.cat([live, torch.zeros(n, tokens, dtype=torch.bool, device="cuda")], 1)
        for t in range(tokens):
            q, k, v = (st[x].reshape(tokens, w.n_layers, n, D)[t, layer].double()
                       for x in ("q", "k", "v"))
            K[:, width + t], V[:, width + t] = k, v
            live[:, width + t] = True
            o, _ = _ref_attend(K, V, live, q)
            out.view(tokens, w.n_layers, n, D)[t, layer] = o
    got = {"out": out, "pos": None, "len": None, "nbuf": None, "ntok": None}
    if kind == "compress":
        return {**got, "cap": None, "off": None}
    got |= {"k": None, "v": None, "qbuf": None}
    return {**got, "label": None} if kind == "dense" else got


def _exact_generate(st, out):
    """A whole generation, all heads at once: rows [heads, C + N, D] with the
    tokens in order, those not kept masked out."""
    w, pr = st["w"], st["provider"]
    L, n, D, C, N, E, P = (w.n_layers, w.heads_per_layer, w.head_dim, w.n_cond, w.n_image,
                           w.group_at, w.period)
    heads = L * n
    K = torch.zeros(heads, C + N, D, dtype=torch.float64, device="cuda")
    V = torch.zeros_like(K)
    K[:, :C] = pr.kc.reshape(heads, C, D).double()
    V[:, :C] = pr.vc.reshape(heads, C, D).double()
    pos = torch.arange(C + N, device="cuda").expand(heads, -1)
    live = (pos < C).clone()
    ring = torch.zeros(heads, P, D, device="cuda")
    label = torch.zeros(heads, dtype=torch.long, device="cuda")
    for t in range(N):
        if t > E and (t - E) % P == 0:
            live = _ref_update(w, K, pos, live, label, ring, t)
        q, k, v = (x[t].reshape(heads, D) for x in (pr.q, pr.k, pr.v))
        K[:, C + t], V[:, C + t] = k.double(), v.double()
        live[:, C + t] = True
        ring[:, t % P] = q.float()
        # the rows kept so far, packed, so that a step costs what is kept
        width = int(live.sum(1).max())
        idx = torch.argsort((~live).to(torch.uint8), dim=1, stable=True)[:, :width]
        ok = live.gather(1, idx)
        g = idx[:, :, None].expand(-1, -1, D)
        o, p = _ref_attend(K.gather(1, g), V.gather(1, g), ok, q.double())
        out[t] = o.reshape(out.shape[1:])
        if t == E - 1:  # local iff the newest w_loc - 1 tokens carry tau
            newest = p[:, max(0, C + E - (w.w_loc - 1)):].sum(1)
            label = torch.where(newest >= w.tau, 0, 1)
            live = _ref_update(w, K, pos, live, label, ring, E)
