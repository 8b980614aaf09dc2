"""Layers of many short heads, which the step takes head by head from a
counter, as they are used: several layers and tokens in one call each, every
launch prefetching behind the one before, eager and in a graph. Outputs
against Eq. 1 in fp64, appends and counters exact, bits as without
prefetching; a bad head stops its own layer only."""
import pytest

pytestmark = pytest.mark.gpu

L, S, N, TOKENS = 3, 4, 1000, 5
NAMES = ("len", "ntok", "nbuf", "k", "v", "pos", "qbuf")
TOL = {"fp32": 1e-5, "bf16": 2e-3}


@pytest.fixture(params=[(128, "bf16"), (64, "bf16"), (128, "fp32"), (64, "fp32")],
                ids=lambda p: f"{p[1]}-{p[0]}")
def case(request):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import CacheBuffers, torch_dtype
    D, dtype = request.param
    grain = 8 if (D, dtype) == (128, "fp32") else 16
    cfg = H.make_config(n_layers=L, n_seqs=S, n_heads=N, head_dim=D, dtype=dtype, n_cond=1,
                        n_image=16 * grain + 44, row_len=8, recent_w=8, local_w=5, period=24,
                        group_at=16 * grain - 2, global_budget=40)
    # 16 grains a head at most, and 160 slots or more for each of the grid's CTAs
    assert S * N * 17 >= 160 * 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert H.hkv_decode_step_launches(cfg) == 1
    n, cap = L * S * N, 6 * grain
    g = torch.Generator(device="cuda").manual_seed(D)
    cb = CacheBuffers(cfg, n * cap, "cuda")
    for t in (cb.k, cb.v, cb.qbuf):
        t.normal_(generator=g)
    cb.off.copy_(torch.arange(n, device="cuda") * cap)
    cb.cap.fill_(cap)
    cb.len.copy_(torch.randint(0, cap - TOKENS + 1, (n,), generator=g, device="cuda"))
    cb.label.copy_(torch.randint(0, 2, (n,), generator=g, device="cuda"))
    cb.nbuf.fill_(3)
    cb.ntok.fill_(70)
    q, k, v = (torch.randn(TOKENS, L, S, N, D, generator=g, device="cuda").to(torch_dtype(cfg))
               for _ in range(3))
    first = {nm: getattr(cb, nm).clone() for nm in NAMES}
    ws = torch.zeros(H.hkv_workspace_size(cfg), dtype=torch.uint8, device="cuda")
    out = torch.empty(TOKENS, L, S, N, D, device="cuda")

    def put():
        for nm in NAMES:
            getattr(cb, nm).copy_(first[nm])
        out.fill_(float("nan"))

    def step(t, flags):
        H.hkv_decode_step_layers(cfg, cb.c, q[t], k[t], v[t], out[t], None, ws, ws.numel(), flags,
                                 torch.cuda.current_stream().cuda_stream)

    return H, cfg, cb, (q, k, v, out), first, put, step, cap, TOL[dtype]


def test_prefetching_layers(case):
    import torch
    H, cfg, cb, (q, k, v, out), first, put, step, cap, tol = case
    n, D = first["len"].numel(), q.shape[-1]
    put()
    for t in range(TOKENS):
        step(t, 0)
        torch.cuda.synchronize()
    H.hkv_check(cb.c)
    # rows and counters
    want = {nm: t.clone() for nm, t in first.items()}
    flat = [x.reshape(TOKENS, n, D) for x in (q, k, v, out)]
    for t in range(TOKENS):
        at = cb.off + want["len"]
        want["k"][at], want["v"][at] = flat[1][t], flat[2][t]
        want["pos"][at] = cfg.n_cond + want["ntok"]
        want["qbuf"][torch.arange(n, device="cuda"), want["ntok"].long() % cfg.period] = flat[0][t]
        for nm in ("len", "ntok", "nbuf"):
            want[nm] += 1
        live = torch.arange(cap, device="cuda")[None] < want["len"][:, None]
        s = torch.einsum("nrd,nd->nr", want["k"].view(n, cap, D).double(), flat[0][t].double())
        p = torch.softmax((s / D ** 0.5).masked_fill(~live, -torch.inf), 1)
        exp = torch.einsum("nr,nrd->nd", p, want["v"].view(n, cap, D).double())
        assert (flat[3][t].double() - exp).abs().max().item() <= tol
    for nm in NAMES:
        assert torch.equal(getattr(cb, nm), want[nm]), nm
    bits = out.clone()

    def same():
        torch.cuda.synchronize()
        H.hkv_check(cb.c)
        assert torch.equal(out, bits)
        for nm in NAMES:
            assert torch.equal(getattr(cb, nm), want[nm]), nm

    for _ in range(3):
        put()
        for t in range(TOKENS):
            step(t, H.HKV_STEP_PREFETCH)
        same()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for t in range(TOKENS):
            step(t, H.HKV_STEP_PREFETCH)
    for _ in range(10):
        put()
        graph.replay()
        same()


@pytest.mark.parametrize("head", [0, 1999, S * N - 1])
def test_a_bad_head_stops_its_layer(case, head):
    import torch
    H, cfg, cb, (q, k, v, out), first, put, step, cap, tol = case
    put()
    n = S * N
    mid = slice(n, 2 * n)
    cb.nbuf[n + head] = cfg.period
    first["nbuf"][n + head] = cfg.period     # (as it has to stay)
    for t in range(2):
        step(t, H.HKV_STEP_PREFETCH)
    with pytest.raises(H.HkvError) as e:
        H.hkv_check(cb.c)
    assert e.value.status == H.HKV_ERR_STATE
    for nm in ("len", "ntok", "nbuf"):
        got, old = getattr(cb, nm), first[nm]
        assert torch.equal(got[mid], old[mid]), nm
        for other in (slice(0, n), slice(2 * n, 3 * n)):
            assert torch.equal(got[other], old[other] + 2), nm
    rows = slice(n * cap, 2 * n * cap)
    for nm in ("k", "v", "pos"):
        assert torch.equal(getattr(cb, nm)[rows], first[nm][rows]), nm
    assert torch.equal(cb.qbuf[mid], first["qbuf"][mid])
    cb.err.zero_()
    cb.nbuf[n + head] = 3
    step(2, H.HKV_STEP_PREFETCH)             # the words are ready for the next launch
    H.hkv_check(cb.c)
    assert torch.equal(cb.len[mid], first["len"][mid] + 1)
