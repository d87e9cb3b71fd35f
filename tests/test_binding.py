"""Argument checks of the ctypes binding that no kernel is needed for: tensors that claim to live on a device, and a library
that records its calls."""
import contextlib

import pytest
import torch

from paper_2605_26636_b200 import jetvit as jv


class OnDevice(torch.Tensor):
    """A CPU tensor that passes for a CUDA one."""
    is_cuda = property(lambda self: True)

    def get_device(self):
        return 0


class Library:
    def __init__(self):
        self.calls = []

    def __getattr__(self, name):
        def call(*args):
            self.calls.append(name)
            return jv.JV_OK
        return call


@pytest.fixture
def lib(monkeypatch):
    recorder = Library()
    monkeypatch.setattr(jv, "lib", lambda: recorder)
    monkeypatch.setattr(jv, "_current_device", lambda device: contextlib.nullcontext())
    monkeypatch.setattr(jv, "_stream", lambda stream: 0)
    return recorder


def _dev(*shape):
    return torch.zeros(shape, dtype=torch.bfloat16).as_subclass(OnDevice)


B, H, Hg, Wg = 2, 3, 4, 5
N, C = Hg * Wg, 64 * H
LAYOUTS = {   # of the three outputs; the kernel writes [B, H, N, 64] arrays
    "contiguous": lambda: _dev(B, H, N, 64),
    "every other channel": lambda: _dev(B, H, N, 128)[..., ::2],
    "half of wider rows": lambda: _dev(B, H, N, 128)[..., :64],
    "one head for all": lambda: _dev(B, 1, N, 64).expand(B, H, N, 64),
    "token-major": lambda: _dev(B, N, H, 64).permute(0, 2, 1, 3),
    "transposed": lambda: _dev(B, H, 64, N).transpose(2, 3),
}


@pytest.mark.parametrize("layout", LAYOUTS)
def test_qkv_proj_writes_contiguous_outputs_only(lib, layout):
    out = tuple(LAYOUTS[layout]() for _ in range(3))
    call = lambda: jv.qkv_proj(_dev(B, N, C), _dev(3 * C, C), None, H, Hg, Wg, out=out)
    if layout == "contiguous":
        assert call() == out and lib.calls == ["jv_qkv_proj"]
    else:
        with pytest.raises(ValueError):
            call()
        assert lib.calls == []


@pytest.mark.parametrize("layout", LAYOUTS)
def test_mixers_refuse_inputs_that_are_neither_layout(lib, layout):
    q, k, v = (LAYOUTS[layout]() for _ in range(3))
    out = _dev(B, H, N, 64)
    if layout in ("contiguous", "token-major"):
        jv.window_attn(q, k, v, Hg, Wg, 2, 2, out=out)
        assert lib.calls == ["jv_window_attn"]
    else:
        with pytest.raises(ValueError):
            jv.window_attn(q, k, v, Hg, Wg, 2, 2, out=out)
        assert lib.calls == []
