"""The update's CTAs have 128, 256 or 512 threads by the heads of a launch and
the longest segment: which, and that an update of one layer (few heads) leaves
the bits of an update of all of them."""
import ctypes

import pytest

from test_abi_host import H  # noqa: F401

SMS = 152


@pytest.mark.parametrize("heads,rows,threads", [
    (1, 512, 512), (4 * SMS, 512, 512), (4 * SMS + 1, 512, 256), (16 * SMS, 5000, 256),
    (16 * SMS + 1, 5000, 128), (1, 511, 256), (2 * SMS, 511, 256), (2 * SMS + 1, 511, 128)])
def test_threads(H, heads, rows, threads):  # noqa: F811
    assert ctypes.CDLL(H.LIB_PATH)._ZN3hkv14update_threadsEiii(heads, rows, SMS) == threads


# heads of one launch: 7 a layer (512 or 256 threads), 700 and 2800 in all
@pytest.mark.gpu
@pytest.mark.parametrize("D,dtype", [(128, "bf16"), (64, "bf16"), (128, "fp32"), (64, "fp32")])
@pytest.mark.parametrize("rows,layers", [(700, 100), (520, 400), (130, 100)])
def test_a_layer_equals_all_layers(H, D, dtype, rows, layers):  # noqa: F811
    import torch
    from paper_2605_20600_gb300.engine import CacheBuffers
    C, P, w, n = 30, 13, 16, 7 * layers
    B = rows - C - P
    cfg = H.make_config(n_layers=layers, n_seqs=1, n_heads=7, head_dim=D, dtype=dtype, n_cond=C,
                        n_image=4 * rows, row_len=8, recent_w=w, local_w=w, period=P, group_at=P,
                        global_budget=B)
    g = torch.Generator(device="cuda").manual_seed(rows)
    cb = CacheBuffers(cfg, n * rows, "cuda")
    for t in (cb.k, cb.v, cb.qbuf):
        t.normal_(generator=g)
    label = torch.arange(n, device="cuda") % 3 > 0
    cap = torch.where(label, rows, C + w + P).to(torch.int32)
    cb.label.copy_(label)
    cb.cap.copy_(cap)
    cb.off.copy_(torch.arange(n, device="cuda") * rows)
    cb.len.copy_(cap)
    cb.nbuf.fill_(P)
    tok = 2 * rows
    cb.ntok.fill_(tok)
    r = torch.arange(rows, device="cuda", dtype=torch.int32)[None]
    cb.pos.copy_(torch.where(r < C, r, C + tok - (cap[:, None] - r)).reshape(-1))
    names = ("k", "v", "pos", "len", "nbuf")
    before = {nm: getattr(cb, nm).clone() for nm in names}
    st = torch.cuda.current_stream().cuda_stream
    H.hkv_evict_all(cfg, cb.c, st)
    H.hkv_check(cb.c)
    assert (cb.len == cap - P).all() and (cb.nbuf == 0).all()
    want = {nm: getattr(cb, nm).clone() for nm in names}
    for nm in names:
        getattr(cb, nm).copy_(before[nm])
    for layer in range(layers):
        H.hkv_evict(cfg, cb.c, layer, st)
    H.hkv_check(cb.c)
    for nm in names:
        assert torch.equal(getattr(cb, nm), want[nm]), nm
