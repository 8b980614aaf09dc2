"""Head identification with its keys staged by bulk copies (configs of 512
dense tokens and more) against the kernel for shorter configs on the same
cache: labels and counts are equal bit for bit, at lengths around the rows of
a stage (64 to 256 by row size) and of several stages."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LENS = [1, 2, 31, 63, 64, 65, 127, 128, 129, 191, 192, 193, 255, 256, 257, 383, 384, 385, 449, 500]


@pytest.mark.parametrize("distance", [0, 1])
@pytest.mark.parametrize("D,dtype", [(128, "bf16"), (64, "bf16"), (128, "fp32"), (64, "fp32")])
def test_staged_equals_unstaged(D, dtype, distance):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import CacheBuffers, torch_dtype
    n, seg = len(LENS) * 4, 500
    cfgs = [H.make_config(n_layers=1, n_seqs=1, n_heads=n, head_dim=D, dtype=dtype, n_cond=0,
                          n_image=1000, row_len=25, recent_w=8, local_w=8, period=8, group_at=e,
                          global_budget=16, distance_mode=distance) for e in (seg, 900)]
    g = torch.Generator(device="cuda").manual_seed(D)
    cb = CacheBuffers(cfgs[0], n * seg, "cuda")
    cb.k.normal_(generator=g)
    cb.off.copy_(torch.arange(n, dtype=torch.int64, device="cuda") * seg)
    cb.cap.fill_(seg)
    lens = torch.tensor(LENS * 4, dtype=torch.int32, device="cuda")
    cb.len.copy_(lens)
    cb.ntok.copy_(lens)
    cb.pos.copy_(torch.arange(seg, dtype=torch.int32, device="cuda").repeat(n))
    gain = torch.logspace(-1, 1, n, device="cuda")[:, None]
    q = (torch.randn(1, n, D, generator=g, device="cuda") * gain).to(torch_dtype(cfgs[0]))
    got = []
    for cfg in cfgs:
        label = torch.full((n,), 9, dtype=torch.uint8, device="cuda")
        n_h = torch.zeros(n, dtype=torch.int32, device="cuda")
        H.hkv_identify_heads(cfg, cb.c, 0, q, label, n_h, torch.cuda.current_stream().cuda_stream)
        H.hkv_check(cb.c)
        got.append((label.cpu().numpy(), n_h.cpu().numpy()))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    assert (got[0][1] >= 1).all() and (got[0][1] <= np.array(LENS * 4)).all()
    assert len(set(got[0][1].tolist())) > 20
