"""hkv_decode_attention_noalloc keeps nothing between calls: whatever its
scratch array holds when a call starts (what overlapping calls left behind,
other results, any bytes), the call gives what hkv_decode_attention gives. A
test build of the library gains two functions that write the array."""
import ctypes
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

SOURCE = r"""
#include "hkv_noalloc.cu"
extern "C" int test_fill(int byte) {
  void *p;
  if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess) return 1;
  return cudaMemset(p, byte, sizeof(g_scratch)) != cudaSuccess;
}
extern "C" int test_arrivals(unsigned n) {  // as calls that overlapped may leave them
  void *p;
  if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess) return 1;
  return cudaMemcpy(static_cast<char *>(p) + kBarAt, &n, 4, cudaMemcpyHostToDevice) != cudaSuccess;
}
"""


def _main(lib_path):
    import torch
    import test_zz_no_alloc as Z
    from paper_2605_20600_gb300 import hkv as H
    H.LIB_PATH = lib_path
    f = Z._noalloc(H)
    lib = ctypes.CDLL(lib_path)
    for D, dtype in ((128, "bf16"), (64, "bf16"), (128, "fp32")):
        lens = [2000, 1, 0, 3000, 1777, 65, 900] * 5     # long heads are split over CTAs
        cfg, cb, q, _, _ = Z._ragged_cache(H, lens, D, dtype, seed=D)
        st = torch.cuda.current_stream().cuda_stream
        ws = torch.zeros(H.hkv_workspace_size(cfg), dtype=torch.uint8, device="cuda")

        def both(q):
            want = torch.zeros(len(lens), D, device="cuda")
            H.hkv_decode_attention(cfg, cb.c, 0, q, want, ws, ws.numel(), st)
            out = torch.full_like(want, float("nan"))
            assert f(ctypes.byref(cfg), ctypes.byref(cb.c), 0, q.data_ptr(), out.data_ptr(), st) == 0
            H.hkv_check(cb.c)
            assert torch.equal(out, want)

        both(q)
        for byte in (0xFF, 0x01, 0xA5, 0x00):
            assert lib.test_fill(byte) == 0
            both(q)
            both(-q)
        assert lib.test_arrivals(5) == 0
        for i in range(6):
            both(q * (i + 1))
        graph = torch.cuda.CUDAGraph()       # and under capture
        out = torch.zeros(len(lens), D, device="cuda")
        with torch.cuda.graph(graph):
            assert f(ctypes.byref(cfg), ctypes.byref(cb.c), 0, q.data_ptr(), out.data_ptr(),
                     torch.cuda.current_stream().cuda_stream) == 0
        want = torch.zeros_like(out)
        H.hkv_decode_attention(cfg, cb.c, 0, q, want, ws, ws.numel(), st)
        for byte in (0xFF, 0x00):
            assert lib.test_fill(byte) == 0
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, want)
    print("scratch ok")


def test_whatever_the_scratch_holds(tmp_path):
    sys.path.insert(0, ROOT)
    from paper_2605_20600_gb300 import build as B
    B.build()
    src, obj, lib = (str(tmp_path / n) for n in ("scratch.cu", "scratch.o", "libheadkv_scratch.so"))
    open(src, "w").write(SOURCE)
    cc = B.nvcc()
    subprocess.check_call([cc, *B.ARCH, *B.FLAGS, "-c", src, "-o", obj])
    others = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.SOURCES
              if s != "hkv_noalloc.cu"]
    subprocess.check_call([cc, *B.ARCH, "-shared", *others, obj, "-o", lib])
    code = (f"import sys; sys.path.insert(0, {ROOT!r}); sys.path.insert(0, {HERE!r}); "
            f"import test_noalloc_scratch as t; t._main({lib!r})")
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "scratch ok" in r.stdout
