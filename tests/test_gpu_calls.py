"""Layer's native marshalling and the general path behind it: the same results for buffers that are not tensors, the same
errors for what neither takes, and the allocation rules (slabs once per row count, outputs per call)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2510_02822_b200 import binding as fx
from paper_2510_02822_b200 import inputs

pytestmark = pytest.mark.gpu


class Buffer:
    """A device buffer that is no tensor: an address and what Layer asks of it."""

    def __init__(self, t):
        self.t, self.dtype = t, t.dtype

    def data_ptr(self):
        return self.t.data_ptr()

    def numel(self):
        return self.t.numel()


def make(conv=None):
    dev = torch.device("cuda:0")
    shape = (48, 3, 3, 64) if conv else (64, 48)
    W = torch.from_numpy((inputs.uniform(41, 0, int(np.prod(shape))) * 255).astype(np.int64) - 127).to(torch.int8).reshape(shape).to(dev)
    return fx.Layer(W, torch.full((48,), 0.01, device=dev), None, np.arange(4, dtype=np.int32)[::-1].copy(), np.array([1, 0, 2, 1], np.uint8), 16, conv=conv)


def test_tensors_and_other_buffers_give_the_same():
    L, C = make(), make(conv=(1, 1))
    for layer in (L, C):
        layer.set_lowbit_ratio(0.5)
    X = torch.from_numpy(inputs.normal(42, 0, 36 * 64).reshape(36, 64).astype(np.float32)).cuda()
    for dynamic in (False, True):
        x4, x8, pos = L.quantize_lower(X, 0.02, dynamic=dynamic)
        a = x4[:36 * 64].clone()
        y = L.mixed_gemm(x4, x8, 36, 0.02, 0.5, fx.OUT_DEQUANT_F16, x_shift=pos)
        b4, b8, bpos = L.quantize_lower(Buffer(X), 0.02, dynamic=dynamic)
        assert b4 is x4 and b8 is x8 and torch.equal(a, b4[:36 * 64])          # slabs are kept per row count
        assert (pos is None and bpos is None) if not dynamic else torch.equal(pos, bpos)
        z = L.mixed_gemm(Buffer(b4), Buffer(b8), 36, 0.02, 0.5, fx.OUT_DEQUANT_F16, x_shift=pos)
        assert torch.equal(y, z) and y.data_ptr() != z.data_ptr() and y.shape == (36, 48) and y.dtype == torch.float16
    c4, c8, _ = C.quantize_lower(X, 0.02)
    y = C.mixed_conv(c4, c8, 1, 6, 6, 0.02, 0.5, fx.OUT_REQUANT_I8)
    assert y.shape == (1, 6, 6, 48) and torch.equal(y, C.mixed_conv(Buffer(c4), Buffer(c8), 1, 6, 6, 0.02, 0.5, fx.OUT_REQUANT_I8))
    own = torch.empty_like(y)
    assert C.mixed_conv(c4, c8, 1, 6, 6, 0.02, 0.5, fx.OUT_REQUANT_I8, Y=own) is own and torch.equal(own, y)


def test_the_same_errors():
    L = make()
    X = torch.zeros(8, 64, device="cuda")
    L.quantize_lower(X, np.float32(1.0))
    x4, x8, _ = L.quantize_lower(X, 1)                                          # whole numbers are numbers
    with pytest.raises(ctypes.ArgumentError):
        L.quantize_lower(X, "1.0")
    with pytest.raises(KeyError):
        L.quantize_lower(X.double(), 1.0)
    with pytest.raises(KeyError):
        L.mixed_gemm(x4, x8, 8, 1.0, 1.0, 3)
    for call in (lambda: L.quantize_lower(X, -1.0), lambda: L.mixed_gemm(x4, x8, 8, 1.0, 0.0, fx.OUT_REQUANT_I8), lambda: L.set_lowbit_ratio(1.5),
                 lambda: L.mixed_conv_to_slab(x4, x8, 1, 2, 4, 1.0, L, 1.0) if L.conv else L.mixed_gemm_to_slab(x4, x8, 8, 1.0, make(), 1.0)):
        with pytest.raises(fx.FlexiqError) as e:
            call()
        assert e.value.code == fx.ERR_INVALID_ARG and str(e.value).startswith("flexiq error -1: ")
    L.close()
    with pytest.raises(fx.FlexiqError):
        L.quantize_lower(X, 1.0)
