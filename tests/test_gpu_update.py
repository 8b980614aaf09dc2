"""The periodic update, the repack of every layer and the budgets at the sizes
where their work is cut: segments around the rows a warp stages and the
threads of a block, one to many buffered queries, and head counts around the
budgets' blocks. Against the oracle's ranking (fp32 in the fixed order) and
plain numpy, bit for bit."""
import numpy as np
import pytest

from oracle import headkv as O

pytestmark = pytest.mark.gpu


def _cache(H, cfg, labels, lens, ntok, seed):
    import torch
    from paper_2605_20600_gb300.engine import CacheBuffers
    n = len(lens)
    g = torch.Generator(device="cuda").manual_seed(seed)
    budget, cap, off, total = O.arena_layout(labels, cfg.n_cond, cfg.global_budget, cfg.recent_w,
                                             cfg.period)
    cb = CacheBuffers(cfg, total, "cuda")
    cb.k.normal_(generator=g)
    cb.v.normal_(generator=g)
    cb.qbuf.normal_(generator=g)
    cb.off.copy_(torch.from_numpy(off.astype(np.int64)))
    cb.cap.copy_(torch.from_numpy(cap.astype(np.int32)))
    cb.label.copy_(torch.from_numpy(np.asarray(labels, dtype=np.uint8)))
    cb.len.copy_(torch.from_numpy(np.asarray(lens, dtype=np.int32)))
    cb.ntok.fill_(ntok)
    cb.nbuf.fill_(cfg.period)
    return cb, off, cap


@pytest.mark.parametrize("D,dtype", [(128, "bf16"), (64, "bf16"), (128, "fp32"), (64, "fp32")])
@pytest.mark.parametrize("budget,P,C", [(9, 1, 0), (20, 3, 2), (31, 7, 1), (100, 16, 5),
                                        (127, 33, 3), (500, 65, 17)])
def test_update(budget, P, C, D, dtype):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    rng = np.random.default_rng(budget + D)
    w, n = 8, 40
    ntok = budget + P + 300
    cfg = H.make_config(n_layers=2, n_seqs=2, n_heads=n // 4, head_dim=D, dtype=dtype, n_cond=C,
                        n_image=ntok, row_len=8, recent_w=w, local_w=8, period=P,
                        group_at=max(P, 1), global_budget=budget)
    labels = rng.integers(0, 2, n)
    labels[:2] = 0, 1
    cap = C + np.where(labels == 1, budget, w) + P
    lens = cap.copy()
    short = rng.random(n) < 0.3         # histories that are not full yet
    lens[short] = C + w + P + rng.integers(0, np.maximum(cap - C - w - P, 0) + 1)[short]
    cb, off, cap = _cache(H, cfg, labels, lens, ntok, budget)
    pos0 = {}
    for i in range(n):                  # any order of rows: positions are what counts
        old = np.sort(rng.choice(ntok - w - P, lens[i] - C - w - P, replace=False))
        p = np.concatenate([np.arange(C), C + old, C + np.arange(ntok - w - P, ntok)])
        pos0[i] = rng.permutation(p)
        cb.pos[int(off[i]):int(off[i]) + lens[i]] = torch.from_numpy(pos0[i].astype(np.int32)).cuda()
    k0, v0 = cb.k.float().cpu().numpy(), cb.v.float().cpu().numpy()
    ring = cb.qbuf.float().cpu().numpy()
    H.hkv_evict_all(cfg, cb.c, torch.cuda.current_stream().cuda_stream)
    H.hkv_check(cb.c)
    ln, pos = cb.len.cpu().numpy(), cb.pos.cpu().numpy()
    k1, v1 = cb.k.float().cpu().numpy(), cb.v.float().cpu().numpy()
    assert (cb.nbuf.cpu().numpy() == 0).all()
    for i in range(n):
        o, p = int(off[i]), pos0[i]
        rows = np.flatnonzero((p >= C) & (p < C + ntok - w))
        rows = rows[np.argsort(p[rows])]   # history, oldest first
        gone = np.ones(rows.size, dtype=bool)
        if labels[i] == 1:
            M = max(0, rows.size - (budget - w))
            q = ring[i][(ntok - P + np.arange(P)) % P]
            gone = O.ste_evict(O.ste_scores_fp32(q, k0[o + rows]), p[rows],
                               O.ste_partition(rows.size, cfg.r_s), M) if M else ~gone
        keep = np.ones(p.size, dtype=bool)
        keep[rows[gone]] = False
        new = int(keep.sum())
        src = np.arange(new)               # the i-th hole takes the i-th survivor above
        src[np.flatnonzero(~keep[:new])] = new + np.flatnonzero(keep[new:])
        assert ln[i] == new, i
        assert np.array_equal(pos[o:o + new], p[src]), i
        assert np.array_equal(k1[o:o + new], k0[o + src]), i
        assert np.array_equal(v1[o:o + new], v0[o + src]), i


@pytest.mark.parametrize("C,E,P", [(0, 9, 1), (3, 40, 7), (29, 100, 24), (128, 500, 65)])
def test_repack_of_every_layer_equals_one_per_layer(C, E, P):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import CacheBuffers, Engine
    cfg = H.make_config(n_layers=3, n_seqs=2, n_heads=7, head_dim=128, dtype="bf16", n_cond=C,
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
    one = CacheBuffers(cfg, eng.total_tokens, "cuda", qbuf=eng.dense.qbuf, label=eng.labels,
                       off=eng.off, cap=eng.cap)
    for layer in range(cfg.n_layers):
        H.hkv_repack(cfg, eng.dense.c, one.c, layer, eng.stream())
    eng.check()
    H.hkv_check(one.c)
    for nm in ("len", "nbuf", "ntok", "pos"):
        assert torch.equal(getattr(one, nm), getattr(eng.ragged, nm)), nm
    for o, m in zip(eng.off.tolist(), one.len.tolist()):
        assert torch.equal(one.k[o:o + m], eng.ragged.k[o:o + m])
        assert torch.equal(one.v[o:o + m], eng.ragged.v[o:o + m])
        p = one.pos[o:o + m].long()    # the kept rows are the dense cache's
        assert bool((p[1:] > p[:-1]).all())


@pytest.mark.parametrize("n", [1, 31, 32, 33, 511, 513, 4095, 4096, 4097, 70001, 1048577])
def test_budgets(n):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    cfg = H.make_config(n_layers=1, n_seqs=1, n_heads=n, head_dim=64, dtype="bf16", n_cond=3,
                        n_image=64, row_len=8, recent_w=8, local_w=8, period=5, group_at=8,
                        global_budget=21)
    label = np.random.default_rng(n).integers(0, 2, n).astype(np.uint8)
    dev = torch.from_numpy(label).cuda()
    budget, cap = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    off = torch.zeros(n, dtype=torch.int64, device="cuda")
    total = H.hkv_allocate_budgets(cfg, dev, budget, cap, off, torch.cuda.current_stream().cuda_stream)
    want = np.where(label == 1, 21, 8)
    assert np.array_equal(budget.cpu().numpy(), want)
    assert np.array_equal(cap.cpu().numpy(), want + 8)
    end = np.cumsum(want.astype(np.int64) + 8)
    assert np.array_equal(off.cpu().numpy(), end - want - 8) and total == end[-1]
    for at in (0, n // 2, n - 1):
        bad = dev.clone()
        bad[at] = H.HKV_DENSE
        with pytest.raises(H.HkvError) as e:
            H.hkv_allocate_budgets(cfg, bad, budget, cap, off,
                                   torch.cuda.current_stream().cuda_stream)
        assert e.value.status == H.HKV_ERR_STATE
