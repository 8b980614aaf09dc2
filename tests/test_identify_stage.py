"""Identification takes its keys through bulk-copied stages where every head
has an SM, or half of one, for itself: which launches do, and that labels and
counts do not depend on it."""
import ctypes

import pytest

from test_abi_host import H  # noqa: F401

SMS = 152


@pytest.mark.parametrize("heads,rows,grid,bytes_,staged", [
    (1, 511, 0, 256, False), (1, 512, 0, 128, True), (2 * SMS, 628, 0, 256, True),
    (2 * SMS + 1, 628, 0, 256, False), (2 * SMS + 1, 628, 0, 512, True),
    (2 * SMS + 1, 1023, 0, 256, False), (5000, 1024, 0, 256, True),
    (2 * SMS + 1, 628, 1, 512, False), (2 * SMS, 6128, 0, 256, True), (1, 33000, 0, 256, True),
    (1, 33300, 0, 256, False), (2 * SMS, 1000, 1, 256, True), (2 * SMS, 1100, 1, 256, False),
    (SMS, 1100, 1, 256, True), (SMS, 8400, 1, 256, False)])
def test_which_launches_are_staged(H, heads, rows, grid, bytes_, staged):  # noqa: F811
    f = ctypes.CDLL(H.LIB_PATH)._ZN3hkv20identify_stage_bytesEiibii
    f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_bool, ctypes.c_int, ctypes.c_int]
    f.restype = ctypes.c_size_t
    assert (f(heads, rows, bool(grid), bytes_, SMS) > 0) == staged


@pytest.mark.gpu
@pytest.mark.parametrize("distance", [0, 1])
@pytest.mark.parametrize("D,dtype", [(128, "bf16"), (64, "bf16"), (128, "fp32"), (64, "fp32")])
def test_many_heads_as_few(H, D, dtype, distance):  # noqa: F811
    import torch
    from paper_2605_20600_gb300.engine import CacheBuffers, torch_dtype
    seg, n = 700, 640            # one layer of 640 heads, or ten of 64
    cfgs = [H.make_config(n_layers=layers, n_seqs=1, n_heads=n // layers, head_dim=D, dtype=dtype,
                          n_cond=20, n_image=1000, row_len=25, recent_w=8, local_w=8, period=8,
                          group_at=seg - 20, global_budget=16, distance_mode=distance)
            for layers in (1, 10)]
    g = torch.Generator(device="cuda").manual_seed(D)
    cb = CacheBuffers(cfgs[0], n * seg, "cuda")
    cb.k.normal_(generator=g)
    cb.off.copy_(torch.arange(n, device="cuda") * seg)
    cb.cap.fill_(seg)
    cb.len.copy_(torch.randint(21, seg + 1, (n,), generator=g, device="cuda"))
    cb.ntok.copy_(cb.len - 20)
    cb.pos.copy_(torch.arange(seg, dtype=torch.int32, device="cuda").repeat(n))
    gain = torch.logspace(-1, 1, n, device="cuda")[:, None]
    q = (torch.randn(n, D, generator=g, device="cuda") * gain).to(torch_dtype(cfgs[0]))
    got = []
    for cfg in cfgs:
        label = torch.full((n,), 9, dtype=torch.uint8, device="cuda")
        n_h = torch.zeros(n, dtype=torch.int32, device="cuda")
        per = n // cfg.n_layers
        for layer in range(cfg.n_layers):
            H.hkv_identify_heads(cfg, cb.c, layer, q[layer * per:(layer + 1) * per], label, n_h,
                                 torch.cuda.current_stream().cuda_stream)
        H.hkv_check(cb.c)
        got.append((label, n_h))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    assert got[0][1].unique().numel() > 20
