"""The grouping token's step when its CTAs are not all resident at once, as
when launches on other streams hold part of the GPU: no CTA may wait for one
with a higher number. A test build launches three times the CTAs that fit;
then several streams run the step at once."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

# a layer whose heads are checked by every CTA, and one too long for that
SHAPES = [(40, 9000), (700, 500)]
TYPES = [(128, "bf16"), (64, "bf16"), (128, "fp32"), (64, "fp32")]
TOL = {"fp32": 1e-5, "bf16": 2e-3}


def _cache(n, rows, D, dtype, layers):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    from paper_2605_20600_gb300.engine import CacheBuffers, torch_dtype
    cfg = H.make_config(n_layers=layers, n_seqs=1, n_heads=n, head_dim=D, dtype=dtype, n_cond=rows,
                        n_image=64, row_len=8, recent_w=8, local_w=40, period=8, group_at=16,
                        global_budget=16)
    g = torch.Generator(device="cuda").manual_seed(n + D)
    cap = rows + 16
    cb = CacheBuffers(cfg, layers * n * cap, "cuda")
    cb.k.normal_(generator=g)
    cb.v.normal_(generator=g)
    cb.off.copy_(torch.arange(layers * n, device="cuda") * cap)
    cb.cap.fill_(cap)
    cb.len.copy_(torch.randint(rows // 2, rows, (layers * n,), generator=g, device="cuda"))
    q, k, v = (torch.randn(layers, 1, n, D, generator=g, device="cuda").to(torch_dtype(cfg))
               for _ in range(3))
    # half of the heads look at their newest tokens only
    at = cb.off[::2, None] + cb.len[::2, None].long() - 1 - torch.arange(20, device="cuda")
    cb.k[at] += 3 * q.reshape(-1, D)[::2, None]
    return cfg, cb, q, k, v


NAMES = ("len", "ntok", "nbuf", "k", "v", "pos", "qbuf")


def _waves_main(lib_path):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    H.LIB_PATH = lib_path
    fit = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    for n, rows in SHAPES:
        for D, dtype in TYPES:
            cfg, cb, q, k, v = _cache(n, rows, D, dtype, 2)
            grain, tile = (8, 32) if (D, dtype) == (128, "fp32") else (16, 64 if D == 128 or dtype == "fp32" else 128)
            slots = int(((cb.len[:n].long() + grain) // grain + 1).sum())
            assert slots // (3 * tile // grain) > 2 * fit      # of ranges at their smallest
            ws = torch.zeros(H.hkv_workspace_size(cfg), dtype=torch.uint8, device="cuda")
            first = {nm: getattr(cb, nm).clone() for nm in NAMES}
            got = []
            for two in (True, False):
                os.environ.pop("HKV_STEP_TWO_KERNELS", None)
                if two:
                    os.environ["HKV_STEP_TWO_KERNELS"] = "1"
                for rep in range(1 if two else 5):
                    for nm in NAMES:
                        getattr(cb, nm).copy_(first[nm])
                    out = torch.full((3, 2, 1, n, D), float("nan"), device="cuda")
                    label = torch.full((2 * n,), 7, dtype=torch.uint8, device="cuda")
                    labels = []
                    for t in range(3):
                        for layer in range(2):
                            H.hkv_decode_step_identify(
                                cfg, cb.c, layer, q[layer], k[layer], v[layer], out[t, layer], label,
                                ws, ws.numel(), H.HKV_STEP_PREFETCH if rep % 2 else 0,
                                torch.cuda.current_stream().cuda_stream)
                        labels.append(label.clone())
                    H.hkv_check(cb.c)
                    got.append((out, torch.stack(labels), {nm: getattr(cb, nm).clone() for nm in NAMES}))
            want = got[0]
            assert set(want[1].unique().tolist()) == {0, 1}
            assert torch.equal(want[2]["len"], first["len"] + 3)
            for out, label, state in got[1:]:
                assert (out - want[0]).abs().max().item() <= 2 * TOL[dtype]
                assert torch.equal(out, got[1][0])
                assert torch.equal(label, want[1])
                for nm in NAMES:
                    assert torch.equal(state[nm], want[2][nm]), nm
            # a bad head stops the step, whichever CTA finds it, and only that one
            for head in (0, n // 2, n - 1):
                for nm in NAMES:
                    getattr(cb, nm).copy_(first[nm])
                cb.cap[n + head] = cb.len[n + head]
                for layer in (0, 1, 0):
                    H.hkv_decode_step_identify(cfg, cb.c, layer, q[layer], k[layer], v[layer],
                                               out[0, layer], label[0], ws, ws.numel(), 0,
                                               torch.cuda.current_stream().cuda_stream)
                with pytest.raises(H.HkvError) as e:
                    H.hkv_check(cb.c)
                assert e.value.status == H.HKV_ERR_CAPACITY
                assert torch.equal(cb.len[:n], first["len"][:n] + 2)
                assert torch.equal(cb.len[n:], first["len"][n:])
                rows1 = slice(n * (rows + 16), None)
                assert torch.equal(cb.k[rows1], first["k"][rows1])
                assert torch.equal(cb.qbuf[n:], first["qbuf"][n:])
                cb.cap[n + head] = rows + 16
                cb.err.zero_()
    print("waves ok")


def test_three_times_the_resident_ctas(tmp_path):
    sys.path.insert(0, ROOT)
    from paper_2605_20600_gb300 import build as B
    lib = str(tmp_path / "libheadkv_waves.so")
    B.build(force=True, extra_flags=["-DHKV_STEP_TEST_WAVES=3", "-DHKV_WAIT_TIMEOUT_NS=300000000ull"],
            lib_path=lib, build_dir=str(tmp_path / "obj"))
    code = (f"import sys; sys.path.insert(0, {ROOT!r}); sys.path.insert(0, {HERE!r}); "
            f"import test_identify_waves as t; t._waves_main({lib!r})")
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "waves ok" in r.stdout


@pytest.mark.parametrize("n,rows", SHAPES)
def test_streams_that_share_the_gpu(n, rows):
    import torch
    from paper_2605_20600_gb300 import hkv as H
    D, dtype, steps = 128, "bf16", 12
    runs = [_cache(n, rows, D, dtype, 1) for _ in range(4)]
    cfg = runs[0][0]
    spaces = [torch.zeros(H.hkv_workspace_size(cfg), dtype=torch.uint8, device="cuda") for _ in runs]
    outs = torch.full((4, steps, 1, n, D), float("nan"), device="cuda")
    labels = torch.full((4, steps, n), 7, dtype=torch.uint8, device="cuda")

    def call(i, t, stream):
        _, cb, q, k, v = runs[i]
        H.hkv_decode_step_identify(cfg, cb.c, 0, q[0], k[0], v[0], outs[i, t], labels[i, t],
                                   spaces[i], spaces[i].numel(), 0, stream.cuda_stream)

    for t in range(steps):                       # one run on its own
        call(0, t, torch.cuda.current_stream())
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(priority=-(i % 2)) for i in range(4)]
    for t in range(steps):
        for i in range(1, 4):
            call(i, t, streams[i])
    torch.cuda.synchronize()
    for i in range(4):
        H.hkv_check(runs[i][1].c)
        assert torch.equal(outs[i], outs[0]) and torch.equal(labels[i], labels[0])
        for nm in NAMES:
            assert torch.equal(getattr(runs[i][1], nm), getattr(runs[0][1], nm)), nm
