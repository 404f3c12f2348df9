"""The autotuner's cache key follows the library's sources: a choice cached for other kernels is measured again (CPU)."""
import types

import numpy as np
import torch

from paper_2512_06102_gb300 import autotune, build, jwf


def test_key_changes_with_the_kernels(tmp_path, monkeypatch):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda d: "gpu")
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    src = [tmp_path / "k_a.cu", tmp_path / "k_b.cu"]
    for f in src:
        f.write_text("old")
    monkeypatch.setattr(build, "_deps", lambda: [str(f) for f in src])
    sim = types.SimpleNamespace(H=np.array([64, 64, 40]), W=np.array([64, 64, 50]))
    key = autotune.signature(sim, jwf.KERNEL_FUSED, 16)
    assert autotune.signature(sim, jwf.KERNEL_FUSED, 16) == key
    src[1].write_text("new")
    assert autotune.signature(sim, jwf.KERNEL_FUSED, 16) != key
    src[1].write_text("old")
    assert autotune.signature(sim, jwf.KERNEL_FUSED, 16) == key
