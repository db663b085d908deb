"""The Python side of a layer without its native marshalling: objects that only look like a layer keep working."""
import numpy as np
import pytest

from paper_2510_02822_b200 import binding as fx
from paper_2510_02822_b200 import build


class Bare(fx.Layer):
    """A subclass that sets itself up and never runs Layer.__init__."""

    def __init__(self):
        self.h, self.K, self.N, self.G, self.conv, self.R, self.S = "handle", 64, 64, 16, (1, 1), 3, 3


class Next:
    h = "next"

    def alloc_slabs(self, M):
        return f"slab of {M}", None


@pytest.fixture(scope="module")
def lib_built():
    build.build_library()


@pytest.fixture
def calls(monkeypatch):
    seen = []
    for name in ("flexiq_mixed_gemm_to_slab", "flexiq_mixed_conv_to_slab", "flexiq_set_lowbit_ratio", "flexiq_layer_destroy"):
        monkeypatch.setattr(fx, name, lambda *a, name=name: seen.append((name, *a)))
    return seen


def test_without_the_native_module(monkeypatch, lib_built):
    monkeypatch.setattr(fx, "_calls_module", None)
    monkeypatch.setitem(__import__("sys").modules, "paper_2510_02822_b200._calls", None)      # import raises ImportError
    monkeypatch.delattr(__import__("paper_2510_02822_b200"), "_calls", raising=False)
    with pytest.warns(RuntimeWarning, match="native marshalling"):
        assert fx._native_calls() is None
    assert fx._native_calls() is None                                                         # and says so once


def test_build_is_stale_for_another_torch_and_finds_nvcc_by_name(monkeypatch, lib_built, tmp_path):
    assert not build._calls_stale()
    monkeypatch.setattr(build, "_calls_for", lambda: "python 0.0, torch 0.0")
    assert build._calls_stale() and build._stale()
    tool = tmp_path / "bin" / "nvcc"
    tool.parent.mkdir()
    tool.write_text("#!/bin/sh\n")
    tool.chmod(0o755)
    monkeypatch.setenv("PATH", str(tool.parent))
    monkeypatch.setenv("NVCC", "nvcc")
    assert build._nvcc() == str(tool)


def test_next_layer_of_another_type(calls):
    L = Bare()
    assert L.mixed_gemm_to_slab("x4", None, 5, 0.5, Next(), 0.25) == "slab of 5"
    assert L.mixed_conv_to_slab("x4", None, 2, 4, 4, 0.5, Next(), 0.25, relu=True) == "slab of 32"
    L.set_lowbit_ratio(0.5)
    assert [c[0] for c in calls] == ["flexiq_mixed_gemm_to_slab", "flexiq_mixed_conv_to_slab", "flexiq_set_lowbit_ratio"]
    assert calls[0][1] == "handle" and calls[0][7] == "next" and calls[1][9] == "next"


def test_native_layer_with_a_next_layer_of_another_type(calls):
    class Native:
        def __getattr__(self, name):
            raise AssertionError(f"{name} was called with an object the native side does not know")
    L = Bare()
    L._calls = Native()
    assert L.mixed_gemm_to_slab("x4", None, 5, 0.5, Next(), 0.25) == "slab of 5"
    assert L.mixed_conv_to_slab("x4", None, 1, 4, 4, 0.5, Next(), 0.25) == "slab of 16"


def test_selections_without_the_native_module(monkeypatch, lib_built):
    """Checked and enqueued in one call, with the ratios set before it and put back where it is refused."""
    seen, low = [], {"a": 16, "b": 48}
    monkeypatch.setattr(fx, "_native_calls", lambda: None)
    monkeypatch.setattr(fx, "flexiq_get_max_4bit_ch", lambda h: low[h])

    def set_ratio(h, ratio):
        low[h] = int(np.ceil(ratio * 4 - 1e-4)) * 16
    monkeypatch.setattr(fx, "flexiq_set_lowbit_ratio", set_ratio)

    def lay_out(*args):
        seen.append((args, dict(low)))
        if args[0][-1] == "a":
            raise fx.FlexiqError(fx.ERR_INVALID_ARG, "refused")
    monkeypatch.setattr(fx, "flexiq_layers_set_group_perm", lay_out)
    A, B = Bare(), Bare()
    A.h, B.h = "a", "b"
    flags = np.array([0, 1, 0, 1], np.uint8), [1, 0, 0, 0]
    fx.select_groups([(A, "Wa", flags[0], None), (B, "Wb", flags[1], [0, 1, 2, 3])])
    ((handles, weights, perms, shifts), then), = seen
    assert handles == ["a", "b"] and weights == ["Wa", "Wb"] and then == low == {"a": 32, "b": 16}
    assert [p.tolist() for p in perms] == [[1, 3, 0, 2], [0, 1, 2, 3]] and all(p.dtype == np.int32 for p in perms)
    assert shifts[0] is None and shifts[1].dtype == np.uint8 and shifts[1].tolist() == [0, 1, 2, 3]
    with pytest.raises(fx.FlexiqError):
        fx.select_groups([(B, "Wb", flags[0], None), (A, "Wa", [1, 1, 1, 1], None)])
    assert seen[1][1] == {"a": 64, "b": 32} and low == {"a": 32, "b": 16}
    B.select_groups("Wb", [0, 0, 0, 0], None)
    assert seen[2][0][0] == ["b"] and low == {"a": 32, "b": 0}
    A.h = B.h = None
