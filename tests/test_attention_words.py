"""The attention alone keeps its own words in the workspace, whatever the
layer and config: between a step and the attention of one layer, launched
back to back, and between the attentions of several configs on one
workspace, nothing is taken for something else. Heads are long, so that every
one is split over CTAs."""
import pytest

pytestmark = pytest.mark.gpu


def _cache(D, dtype, layers, n, rows):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import CacheBuffers, torch_dtype
    cfg = H.make_config(n_layers=layers, n_seqs=1, n_heads=n, head_dim=D, dtype=dtype, n_cond=rows,
                        n_image=64, row_len=8, recent_w=8, local_w=5, period=8, group_at=9,
                        global_budget=16)
    g = torch.Generator(device="cuda").manual_seed(D + layers)
    cap = rows + 8
    cb = CacheBuffers(cfg, layers * n * cap, "cuda")
    cb.k.normal_(generator=g)
    cb.v.normal_(generator=g)
    cb.off.copy_(torch.arange(layers * n, device="cuda") * cap)
    cb.cap.fill_(cap)
    cb.len.fill_(rows)
    q, k, v = (torch.randn(1, n, D, generator=g, device="cuda").to(torch_dtype(cfg))
               for _ in range(3))
    return H, cfg, cb, q, k, v


def test_configs_that_take_turns_on_one_workspace():
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    runs = [_cache(128, "bf16", 2, 10, 3000), _cache(64, "bf16", 3, 40, 2000),
            _cache(128, "fp32", 5, 7, 2500), _cache(128, "bf16", 3, 10, 3000)]
    size = max(H.hkv_workspace_size(cfg) for H, cfg, *_ in runs)

    def attend(run, layer, sign, ws):
        H, cfg, cb, q, _, _ = run
        out = torch.full(q.shape, float("nan"), device="cuda")
        H.hkv_decode_attention(cfg, cb.c, layer, q * sign, out, ws, size, stream)
        H.hkv_check(cb.c)
        return out

    want = {(i, layer, sign): attend(run, layer, sign,
                                     torch.zeros(size, dtype=torch.uint8, device="cuda"))
            for i, run in enumerate(runs) for layer in range(run[1].n_layers) for sign in (1, -1)}
    shared = torch.zeros(size, dtype=torch.uint8, device="cuda")
    for turn in range(6):      # other results at every turn
        for (i, layer, sign), exp in want.items():
            if sign == (1 if turn % 2 == 0 else -1):
                assert torch.equal(attend(runs[i], layer, sign, shared), exp), (turn, i, layer)


@pytest.mark.parametrize("D,dtype", [(128, "bf16"), (64, "bf16"), (128, "fp32")])
def test_attention_and_prefetching_step_of_one_layer(D, dtype):
    import torch
    H, cfg, cb, q, k, v = _cache(D, dtype, 2, 40, 1500)
    size = H.hkv_workspace_size(cfg)
    ws = torch.zeros(size, dtype=torch.uint8, device="cuda")
    outs = torch.empty(4, 1, 40, D, device="cuda")
    names = ("len", "nbuf", "ntok")
    first = {nm: getattr(cb, nm).clone() for nm in names}

    def calls(between):
        s = torch.cuda.current_stream().cuda_stream
        for i in range(4):
            H.hkv_decode_attention(cfg, cb.c, 1, q, outs[i], ws, size, s)
            between()
            H.hkv_decode_step(cfg, cb.c, 1, q, k, v, outs[i], ws, size, H.HKV_STEP_PREFETCH, s)
            between()
            if i % 2 == 0:
                H.hkv_decode_attention(cfg, cb.c, 1, q, outs[i], ws, size, s)
                between()

    calls(torch.cuda.synchronize)
    H.hkv_check(cb.c)
    want = outs.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls(lambda: None)
    for _ in range(20):
        for nm, t in first.items():
            getattr(cb, nm).copy_(t)
        outs.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        H.hkv_check(cb.c)
        assert torch.equal(outs, want)
        assert (cb.len[40:] == 1504).all() and (cb.len[:40] == 1500).all()
