"""How the one-launch kernel (decode step, attention alone, and the step with
identification) cuts a layer into CTA ranges, at the sizes where the cut
changes: a CTA per head up to 12 grains (16 rows; 8 rows of 512 bytes) a
head, layers around the prologue's table (288 or 352 heads) and around eight
rows of 32 heads a warp, heads of every length around a grain and a tile,
and heads split over many CTAs. Every output against Eq. 1 in fp64, the
appends exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "bf16": 2e-3}


def _lens(kind, n, grain, rng):
    if kind == "aligned":      # every head fits the 12 grains, some exactly
        return np.where(rng.random(n) < 0.3, 12 * grain - 1, rng.integers(0, 12 * grain, n))
    if kind == "just over":    # one grain too many in one head
        x = rng.integers(0, 12 * grain, n)
        x[n // 2] = 12 * grain
        return x
    if kind == "edges":
        e = np.array([0, 1, grain - 2, grain - 1, grain, 2 * grain - 1, 4 * grain - 1, 4 * grain,
                      8 * grain - 1, 8 * grain, 8 * grain + 1])
        return e[rng.integers(0, len(e), n)]
    x = rng.integers(0, 40, n)  # "long": a few heads over many CTAs
    x[[0, n // 3, n - 1]] = [5000, 3001, 1777]
    return x


CASES = [("aligned", 1), ("aligned", 64), ("aligned", 256), ("just over", 64), ("edges", 287),
         ("edges", 288), ("edges", 289), ("edges", 351), ("edges", 352), ("edges", 353),
         ("edges", 2304), ("edges", 2817), ("edges", 3300), ("edges", 6100), ("edges", 9800),
         ("long", 7), ("long", 300), ("long", 900)]


@pytest.mark.parametrize("D,dtype", [(128, "bf16"), (64, "bf16"), (128, "fp32"), (64, "fp32")])
@pytest.mark.parametrize("kind,n", CASES)
def test_split(kind, n, D, dtype):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import CacheBuffers, torch_dtype
    rng = np.random.default_rng(n + D)
    grain = 8 if dtype == "fp32" and D == 128 else 16
    L, layer = 2, 1
    lens = _lens(kind, L * n, grain, rng).astype(np.int64)
    lens[layer * n:] = _lens(kind, n, grain, rng)
    top = int(lens.max()) + 2
    cfg = H.make_config(n_layers=L, n_seqs=1, n_heads=n, head_dim=D, dtype=dtype, n_cond=1,
                        n_image=max(top, 64), row_len=8, recent_w=8, local_w=5, period=8,
                        group_at=max(top - 2, 9), global_budget=16)
    caps = lens + 2
    off = np.concatenate([[0], np.cumsum(caps)[:-1]])
    total = int(caps.sum())
    cb = CacheBuffers(cfg, total, "cuda")
    dt = torch_dtype(cfg)
    g = torch.Generator(device="cuda").manual_seed(n)
    cb.k.normal_(generator=g)
    cb.v.normal_(generator=g)
    live = torch.zeros(total, dtype=torch.bool, device="cuda")
    for o, m in zip(off, lens):
        live[int(o):int(o) + int(m)] = True
    cb.v[~live] = float("nan")          # rows past a head's length must not be read as values
    cb.k[~live] = float("nan")
    cb.off.copy_(torch.from_numpy(off))
    cb.cap.copy_(torch.from_numpy(caps.astype(np.int32)))
    cb.len.copy_(torch.from_numpy(lens.astype(np.int32)))
    cb.ntok.fill_(20)
    q, k, v = (torch.randn(1, n, D, generator=g, device="cuda").to(dt) for _ in range(3))
    sl = slice(layer * n, (layer + 1) * n)
    m, o = lens[sl], off[sl]
    at = torch.from_numpy(o)[:, None] + torch.arange(int(m.max()) + 1)[None]
    ok = torch.arange(int(m.max()) + 1)[None] < torch.from_numpy(m)[:, None]
    at = torch.where(ok, at, 0).cuda()
    ok = ok.cuda()
    K = torch.where(ok[:, :, None], cb.k[at].double(), 0.0)
    V = torch.where(ok[:, :, None], cb.v[at].double(), 0.0)

    def ref(new):
        Kx, Vx, okx = K, V, ok
        if new:
            Kx, Vx = torch.cat([K, k[0].double()[:, None]], 1), torch.cat([V, v[0].double()[:, None]], 1)
            okx = torch.cat([ok, torch.ones(n, 1, dtype=torch.bool, device="cuda")], 1)
        s = torch.einsum("nrd,nd->nr", Kx, q[0].double()) / D ** 0.5
        p = torch.softmax(s.masked_fill(~okx, -torch.inf), 1)
        p = torch.where(okx.any(1)[:, None], p, 0.0)
        return torch.einsum("nr,nrd->nd", p, Vx), p

    ws = torch.zeros(H.hkv_workspace_size(cfg), dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    out = torch.full((1, n, D), float("nan"), device="cuda")
    H.hkv_decode_attention(cfg, cb.c, layer, q, out, ws, ws.numel(), st)
    H.hkv_check(cb.c)
    assert (out[0].double() - ref(False)[0]).abs().max().item() <= TOL[dtype]
    exp, p = ref(True)
    label = torch.full((L * n,), 7, dtype=torch.uint8, device="cuda")
    counters = [t.clone() for t in (cb.len, cb.ntok, cb.nbuf)]
    for identify in (True, False):
        for t, b in zip((cb.len, cb.ntok, cb.nbuf), counters):
            t.copy_(b)
        out.fill_(float("nan"))
        if identify:
            H.hkv_decode_step_identify(cfg, cb.c, layer, q, k, v, out, label, ws, ws.numel(), 0, st)
        else:
            H.hkv_decode_step(cfg, cb.c, layer, q, k, v, out, ws, ws.numel(), 0, st)
        H.hkv_check(cb.c)
        assert (out[0].double() - exp).abs().max().item() <= TOL[dtype]
        assert torch.equal(cb.len[sl], counters[0][sl] + 1)
        assert torch.equal(cb.len[:layer * n], counters[0][:layer * n])
        assert torch.equal(cb.ntok[sl], counters[1][sl] + 1)
        rows = torch.from_numpy(o + m).cuda()
        assert torch.equal(cb.k[rows], k[0]) and torch.equal(cb.v[rows], v[0])
        assert (cb.pos[rows] == 1 + 20).all()
        assert torch.equal(cb.qbuf[sl, 20 % 8], q[0])
    # the newest w_loc - 1 = 4 tokens against tau = 0.9
    width = torch.from_numpy(m).cuda() + 1
    order = torch.arange(p.shape[1] - 1, device="cuda")[None]
    newest = torch.where(order >= (width - 4)[:, None], p[:, :-1], 0.0).sum(1) + p[:, -1]
    sure = (newest - 0.9).abs() > 1e-5
    assert torch.equal(label[sl][sure], torch.where(newest >= 0.9, 0, 1).to(torch.uint8)[sure])


@pytest.mark.parametrize("fault", ["capacity", "state", "bounds", "negative"])
@pytest.mark.parametrize("head", [0, 303, 304, 1700, 3999])
def test_one_bad_head_of_many_short_ones_stops_the_step(fault, head):
    """Layers taken head by head: a bad head anywhere leaves every row, counter
    and query of the layer as it was; repaired, the next call on the same
    workspace takes the step."""
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import CacheBuffers
    n, D, P = 4000, 64, 8   # 255 rows allowed: 16 grains, 17 slots a head
    cfg = H.make_config(n_layers=1, n_seqs=4, n_heads=n // 4, head_dim=D, dtype="bf16", n_cond=1,
                        n_image=300, row_len=8, recent_w=8, local_w=5, period=P, group_at=254,
                        global_budget=40)
    g = torch.Generator(device="cuda").manual_seed(head)
    lens = torch.randint(0, 60, (n,), generator=g, device="cuda", dtype=torch.int32)
    cb = CacheBuffers(cfg, n * 64, "cuda")
    for t in (cb.k, cb.v, cb.qbuf):
        t.normal_(generator=g)
    cb.off.copy_(torch.arange(n, device="cuda") * 64)
    cb.cap.fill_(64)
    cb.len.copy_(lens)
    cb.label.copy_(torch.arange(n, device="cuda") % 2)
    cb.nbuf.fill_(3)
    cb.ntok.fill_(70)
    field, value, code = {"capacity": (cb.cap, lens[head], H.HKV_ERR_CAPACITY),
                          "state": (cb.nbuf, P, H.HKV_ERR_STATE),
                          "bounds": (cb.off, n * 64, H.HKV_ERR_BOUNDS),
                          "negative": (cb.len, -1, H.HKV_ERR_BOUNDS)}[fault]
    good = field[head].clone()
    field[head] = value
    q, k, v = (torch.randn(4, n // 4, D, generator=g, device="cuda").bfloat16() for _ in range(3))
    out = torch.zeros(4, n // 4, D, device="cuda")
    ws = torch.zeros(H.hkv_workspace_size(cfg), dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    names = ("k", "v", "pos", "len", "ntok", "nbuf", "qbuf")
    before = {nm: getattr(cb, nm).clone() for nm in names}
    H.hkv_decode_step(cfg, cb.c, 0, q, k, v, out, ws, ws.numel(), 0, st)
    with pytest.raises(H.HkvError) as e:
        H.hkv_check(cb.c)
    assert e.value.status == code
    for nm in names:
        assert torch.equal(getattr(cb, nm), before[nm]), nm
    field[head] = good
    cb.err.zero_()
    for step in range(2):     # and again: the counters are ready for the next launch
        H.hkv_decode_step(cfg, cb.c, 0, q, k, v, out, ws, ws.numel(), 0, st)
        H.hkv_check(cb.c)
        assert torch.equal(cb.len, lens + 1 + step)
        assert (cb.nbuf == 4 + step).all() and (cb.ntok == 71 + step).all()
    K = cb.k.view(n, 64, D).double()
    V = cb.v.view(n, 64, D).double()
    s = torch.einsum("nrd,nd->nr", K, q.view(n, D).double()) / D ** 0.5
    s = s.masked_fill(torch.arange(64, device="cuda")[None] >= cb.len[:, None], -torch.inf)
    exp = torch.einsum("nr,nrd->nd", torch.softmax(s, 1), V)
    assert (out.view(n, D).double() - exp).abs().max().item() <= TOL["bf16"]


@pytest.mark.parametrize("D,dtype", [(128, "bf16"), (64, "fp32")])
def test_attention_on_streams_that_share_the_gpu(D, dtype):
    """The attention alone, a head over many CTAs, on four streams with a
    workspace each: every call gives the bits of a call on its own."""
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import CacheBuffers, torch_dtype
    n, C = 40, 3000
    cfg = H.make_config(n_layers=1, n_seqs=1, n_heads=n, head_dim=D, dtype=dtype, n_cond=C,
                        n_image=64, row_len=8, recent_w=8, local_w=5, period=8, group_at=9,
                        global_budget=16)
    g = torch.Generator(device="cuda").manual_seed(D)
    cb = CacheBuffers(cfg, n * C, "cuda")
    cb.k.normal_(generator=g)
    cb.v.normal_(generator=g)
    cb.off.copy_(torch.arange(n, device="cuda") * C)
    cb.cap.fill_(C)
    cb.len.copy_(torch.randint(0, C + 1, (n,), generator=g, device="cuda"))
    q = torch.randn(1, n, D, generator=g, device="cuda").to(torch_dtype(cfg))

    def call(out, ws, stream):
        H.hkv_decode_attention(cfg, cb.c, 0, q, out, ws, ws.numel(), stream.cuda_stream)

    nbytes = H.hkv_workspace_size(cfg)
    spaces = [torch.zeros(nbytes, dtype=torch.uint8, device="cuda") for _ in range(4)]
    outs = torch.full((4, 25, 1, n, D), float("nan"), device="cuda")
    alone = torch.empty(1, n, D, device="cuda")
    call(alone, spaces[0], torch.cuda.current_stream())
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(priority=-(i % 2)) for i in range(4)]
    for i in range(25):
        for s, ws, o in zip(streams, spaces, outs):
            call(o[i], ws, s)
    torch.cuda.synchronize()
    H.hkv_check(cb.c)
    assert torch.equal(outs, alone.expand_as(outs))
