"""The longest segment that the update, repack and identification take: the
rule in hkv.h, at the last length it accepts and the first one it refuses."""
import ctypes

import pytest

from test_abi_host import H, tiny_cfg  # noqa: F401

KB227 = 227 * 1024
CASES = [(128, "bf16", 65), (128, "fp32", 49), (64, "bf16", 24), (64, "fp32", 24), (128, "bf16", 700)]


def _longest(D, dtype, P):
    es = 2 if dtype == "bf16" else 4
    return (KB227 - max(P * D * es, 256 * (D * es + 16)) - 4 * D - 2112) // 16


def test_accepted_lengths_with_the_shipped_periods():
    assert [_longest(*c) for c in CASES[:4]] == [10012, 5916, 12076, 10028]


@pytest.mark.parametrize("D,dtype,P", CASES)
def test_rule_of_the_header(H, D, dtype, P):  # noqa: F811
    lib = ctypes.CDLL(H.LIB_PATH)
    limit, used = (getattr(lib, n) for n in ("_ZN3hkv18update_limit_bytesEiiii",
                                             "_ZN3hkv17update_smem_bytesEiiiii"))
    for f in (limit, used):
        f.restype = ctypes.c_size_t
    code = 1 if dtype == "bf16" else 0
    n = _longest(D, dtype, P)
    assert limit(n, D, P, code) <= KB227 < limit(n + 1, D, P, code)
    for threads in (128, 256, 512):
        assert used(threads, n, D, P, code) <= KB227  # what is accepted fits


@pytest.mark.gpu
@pytest.mark.parametrize("D,dtype,P", CASES)
def test_calls_at_the_limit(H, D, dtype, P):  # noqa: F811
    import torch
    from paper_2605_20600_gb300.engine import CacheBuffers
    stream = torch.cuda.current_stream().cuda_stream
    q = torch.zeros(1, 1, D, dtype=torch.bfloat16 if dtype == "bf16" else torch.float32, device="cuda")
    for over in (0, 1):
        E = _longest(D, dtype, P) - 8 + over      # C + E tokens
        cfg = tiny_cfg(H, n_layers=1, n_seqs=1, n_heads=1, head_dim=D, dtype=dtype, n_cond=8,
                       n_image=E, period=P, group_at=E)
        cb = CacheBuffers(cfg, 8 + E, "cuda")
        cb.cap.fill_(8 + E)
        calls = [lambda: H.hkv_evict(cfg, cb.c, 0, stream), lambda: H.hkv_evict_all(cfg, cb.c, stream),
                 lambda: H.hkv_append_evict(cfg, cb.c, 0, q, q, q, stream)]
        for call in calls:
            if over:
                with pytest.raises(H.HkvError) as e:
                    call()
                assert e.value.status == H.HKV_ERR_CAPACITY
            else:
                call()
        H.hkv_check(cb.c)
        assert int(cb.len[0]) == 1 - over
