"""A decode step with HKV_STEP_PREFETCH directly behind a call that writes that
step's cache (no kernel in between, one graph): it must find what that call
wrote. On the CPU, the rule that makes it so: such a kernel never lets
the next one start early."""
import os
import re

import pytest

from conftest import ROOT

UPDATE = os.path.join(ROOT, "paper_2605_20600_gb300", "csrc", "hkv_update.cu")


@pytest.mark.parametrize("kernel", ["evict_kernel", "repack_kernel", "init_dense_kernel",
                                    "prefill_kernel"])
def test_kernels_before_a_step_do_not_launch_early(kernel):
    text = re.sub(r"//.*", "", open(UPDATE).read())
    body = text[re.search(r"\b%s\(const CacheArgs" % kernel, text).start():]
    body = body[:body.index("\n}\n")]
    assert "pdl_wait();" in body and "pdl_launch_dependents" not in body


def _copy(c, names):
    return {nm: getattr(c, nm).clone() for nm in names}


def _put(c, saved):
    for nm, t in saved.items():
        getattr(c, nm).copy_(t)


# heads of one launch: all resident at once, so that a successor that may start early does
@pytest.mark.gpu
@pytest.mark.parametrize("D,dtype,C,E,P", [(128, "bf16", 3, 40, 7), (64, "bf16", 29, 100, 24),
                                           (128, "fp32", 128, 500, 65), (64, "fp32", 0, 9, 1)])
def test_step_behind_the_repack_of_every_layer(D, dtype, C, E, P):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import Engine, torch_dtype
    cfg = H.make_config(n_layers=2, n_seqs=2, n_heads=10, head_dim=D, dtype=dtype, n_cond=C,
                        n_image=4 * E, row_len=8, recent_w=8, local_w=8, period=P, group_at=E,
                        global_budget=max(8, E // 2))
    eng = Engine(cfg, "cuda")
    g = torch.Generator(device="cuda").manual_seed(E)
    for t in (eng.dense.k, eng.dense.v, eng.dense.qbuf):
        t.normal_(generator=g)
    eng.dense.pos.copy_(torch.arange(C + E, dtype=torch.int32, device="cuda").repeat(eng.n))
    eng.dense.len.fill_(C + E)
    eng.dense.ntok.fill_(E)
    eng.labels.copy_(torch.randint(0, 2, (eng.n,), generator=g, device="cuda").to(torch.uint8))
    eng.compress()
    q, k, v = (torch.randn(2, 2, 10, D, generator=g, device="cuda").to(torch_dtype(cfg))
               for _ in range(3))
    out = torch.empty(2, 2, 10, D, device="cuda")
    names = ("k", "v", "pos", "len", "nbuf", "ntok", "qbuf")
    c = eng.ragged
    for nm in ("k", "v"):
        getattr(c, nm).zero_()
    for nm in ("pos", "len", "nbuf", "ntok"):
        getattr(c, nm).zero_()
    fresh = _copy(c, names)

    def both(between):
        H.hkv_repack_all(cfg, eng.dense.c, c.c, eng.stream())
        between()
        eng.step_layers(q, k, v, out)

    both(torch.cuda.synchronize)
    eng.check()
    want, want_out = _copy(c, names), out.clone()
    assert int(want["len"].min()) > 1
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        both(lambda: None)
    for _ in range(20):
        _put(c, fresh)
        out.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        eng.check()
        assert torch.equal(out, want_out)
        for nm in names:
            assert torch.equal(getattr(c, nm), want[nm]), nm


@pytest.mark.gpu
def test_step_behind_the_set_up_of_the_uncompressed_cache():
    """Without conditioning tokens the set-up is the kernel before the first step."""
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import Engine
    cfg = H.make_config(n_layers=2, n_seqs=1, n_heads=20, head_dim=64, dtype="bf16", n_cond=0,
                        n_image=64, row_len=8, recent_w=8, local_w=8, period=5, group_at=16,
                        global_budget=16)
    eng = Engine(cfg, "cuda")
    c = eng.dense
    g = torch.Generator(device="cuda").manual_seed(1)
    q, k, v = (torch.randn(2, 1, 20, 64, generator=g, device="cuda").bfloat16() for _ in range(3))
    out = torch.empty(2, 1, 20, 64, device="cuda")
    c.k.normal_(generator=g)
    c.v.normal_(generator=g)

    def both():
        H.hkv_init_dense(cfg, c.c, eng.stream())
        eng.step_layers(q, k, v, out)

    both()     # sets the kernels up
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        both()
    for _ in range(20):
        c.len.fill_(7)      # as an earlier generation leaves them
        c.ntok.fill_(7)
        out.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        eng.check()
        # one token: its own value, times a weight of 1 +- 1 ulp and over it
        assert ((out - v.float()).abs() <= 2.0 ** -22 * v.float().abs()).all()
        assert (c.len == 1).all() and (c.ntok == 1).all() and (c.nbuf == 0).all()
        at = c.off.long()
        assert torch.equal(c.k[at], k.view(-1, 64)) and (c.pos[at] == 0).all()


@pytest.mark.gpu
def test_step_behind_the_prefill_of_its_layer():
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import Engine
    C, n = 40, 20
    cfg = H.make_config(n_layers=2, n_seqs=1, n_heads=n, head_dim=128, dtype="bf16", n_cond=C,
                        n_image=64, row_len=8, recent_w=8, local_w=8, period=5, group_at=16,
                        global_budget=16)
    eng = Engine(cfg, "cuda")
    c = eng.dense
    g = torch.Generator(device="cuda").manual_seed(1)
    q, k, v = (torch.randn(2, 1, n, 128, generator=g, device="cuda").bfloat16() for _ in range(3))
    kc, vc = (torch.randn(2, 1, n, C, 128, generator=g, device="cuda").bfloat16() for _ in range(2))
    out = torch.empty(2, 1, n, 128, device="cuda")

    def both(between):
        for layer in range(2):
            eng.prefill(layer, kc[layer], vc[layer])
            between()
            eng.step(layer, q[layer], k[layer], v[layer], out[layer])

    def empty():
        c.len.zero_()
        c.k.zero_()
        c.v.zero_()
        out.fill_(float("nan"))

    empty()
    both(torch.cuda.synchronize)
    eng.check()
    names = ("k", "v", "pos", "len", "nbuf", "ntok", "qbuf")
    want, want_out = _copy(c, names), out.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        both(lambda: None)
    for _ in range(20):
        empty()
        graph.replay()
        torch.cuda.synchronize()
        eng.check()
        assert torch.equal(out, want_out)
        assert (c.len == C + 1).all()
        for nm in names:
            assert torch.equal(getattr(c, nm), want[nm]), nm
