"""The calls over every layer (include/hkv_layers.h): exported, validated on
the host like the calls per layer, and bit for bit what those give."""
import ctypes
import os
import re

import pytest

from conftest import ROOT

from test_abi_host import H, fake_cache, tiny_cfg  # noqa: F401


def test_declared_symbols_are_exported(H):  # noqa: F811
    text = re.sub(r"/\*.*?\*/", "", open(os.path.join(ROOT, "include", "hkv_layers.h")).read(),
                  flags=re.S)
    names = sorted(set(re.findall(r"\b(hkv_[a-z_]+)\s*\(", text)))
    assert names == ["hkv_decode_step_layers", "hkv_repack_all"]
    for n in names:
        assert hasattr(H.lib(), n)


def test_host_checks(H, monkeypatch):  # noqa: F811
    lib, cfg = H.lib(), tiny_cfg(H)
    c, other = fake_cache(H), fake_cache(H)
    other.qbuf = c.qbuf + 16

    def step(q=16, out=16, ws=16, size=1 << 40, flags=0, cfg=cfg, label=None):
        return lib.hkv_decode_step_layers(ctypes.byref(cfg), ctypes.byref(c), q, 16, 16, out, label,
                                          ws, size, flags, None)

    assert step(q=None) == H.HKV_ERR_INVALID_ARG
    assert step(ws=None) == H.HKV_ERR_INVALID_ARG
    assert step(out=24) == H.HKV_ERR_ALIGN
    assert step(size=H.hkv_workspace_size(cfg) - 1) == H.HKV_ERR_CAPACITY
    assert step(flags=2) == H.HKV_ERR_INVALID_ARG
    assert step(cfg=tiny_cfg(H, distance_mode=1), label=16) == H.HKV_ERR_INVALID_ARG
    assert step(cfg=tiny_cfg(H, head_dim=96)) == H.HKV_ERR_SHAPE
    assert lib.hkv_repack_all(ctypes.byref(cfg), ctypes.byref(c), ctypes.byref(other), None) == \
        H.HKV_ERR_INVALID_ARG
    for name, call, code in (("decode_step_layers", step, 7), ("decode_step", step, 4),
                             ("decode_step_identify", lambda: step(label=16), 4),
                             ("repack_all", lambda: lib.hkv_repack_all(
                                 ctypes.byref(cfg), ctypes.byref(c), ctypes.byref(c), None), 3)):
        monkeypatch.setenv("HKV_FAULT_INJECT", f"{name}:{code}")
        assert call() == code, name


@pytest.mark.gpu
@pytest.mark.parametrize("name,layers,seqs", [("tiny", 1, 1), ("llamagen_xl", 3, 2),
                                              ("janus_pro_7b", 2, 5)])
def test_generation_equals_one_call_per_layer(name, layers, seqs):
    import torch
    from _gpu_util import cfg_of
    from paper_2605_20600_gb300 import hkv
    from paper_2605_20600_gb300.engine import Engine
    from paper_2605_20600_gb300.runner import generate
    from synth import configs
    from synth.gpu import DeviceSynth
    w = configs.ALL[name].with_(n_layers=layers, n_seqs=seqs)

    class PerLayer(Engine):
        def step_layers(self, q, k, v, out, identify=False):
            for i in range(self.cfg.n_layers):
                if identify:
                    self.step_identify(i, q[i], k[i], v[i], out[i])
                else:
                    self.step(i, q[i], k[i], v[i], out[i])

    runs = []
    for cls in (Engine, PerLayer):
        eng, outs = cls(cfg_of(hkv, w), "cuda"), []
        generate(eng, DeviceSynth(w, "cuda"), last_step=w.group_at + 2 * w.period + 1,
                 on_step=lambda t, o: outs.append(o.clone()))
        eng.check()
        runs.append((eng, torch.stack(outs)))
    (a, x), (b, y) = runs
    assert torch.equal(x, y) and torch.equal(a.labels, b.labels)
    for nm in ("len", "nbuf", "ntok", "qbuf"):
        assert torch.equal(getattr(a.cache, nm), getattr(b.cache, nm)), nm
    for o, m in zip(a.off.tolist(), a.cache.len.tolist()):
        assert torch.equal(a.cache.pos[o:o + m], b.cache.pos[o:o + m])
        assert torch.equal(a.cache.k[o:o + m], b.cache.k[o:o + m])
