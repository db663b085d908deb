"""CPU-only checks of the boundary and the host logic: the C-ABI library loads, exports
every symbol the header declares, and rejects bad arguments before touching a device."""
import ctypes as C
import os
import re
import subprocess

import numpy as np
import pytest
import torch

import oracle
from paper_2510_02822_b200 import binding as fx
from paper_2510_02822_b200 import build as fxbuild
from paper_2510_02822_b200 import calib, inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    fxbuild.build_library()
    return fx.lib()


def test_library_exports_every_declared_symbol(lib):
    header = open(os.path.join(ROOT, "include", "flexiq.h")).read()
    declared = set(re.findall(r"\b(flexiq_[a-z0-9_]+)\s*\(", header))
    assert declared, "no declarations found"
    assert declared == set(fx.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), name


def test_create_rejects_bad_arguments_without_a_device(lib):
    h = C.c_void_p()
    perm = np.arange(8, dtype=np.int32)
    dummy = C.c_void_p(16)  # never dereferenced: validation fails first
    pp = perm.ctypes.data_as(C.c_void_p)
    cases = [
        (dict(K=100, N=16, G=16), "multiple of group_size"),
        (dict(K=128, N=16, G=8), "group_size"),
        (dict(K=128, N=20, G=16), "multiple of 16"),
        (dict(K=0, N=16, G=16), "positive"),
    ]
    for kw, msg in cases:
        rc = lib.flexiq_layer_create_linear(C.byref(h), kw["K"], kw["N"], kw["G"], dummy, dummy, None, pp, None, None)
        assert rc == fx.ERR_INVALID_ARG and msg in fx.last_error(), (kw, fx.last_error())
    rc = lib.flexiq_layer_create_linear(C.byref(h), 128, 16, 16, None, dummy, None, pp, None, None)
    assert rc == fx.ERR_INVALID_ARG
    bad = np.array([0, 1, 2, 3, 4, 5, 6, 6], np.int32)
    rc = lib.flexiq_layer_create_linear(C.byref(h), 128, 16, 16, dummy, dummy, None, bad.ctypes.data_as(C.c_void_p), None, None)
    assert rc == fx.ERR_INVALID_ARG and "permutation" in fx.last_error()
    shifts = np.array([0, 1, 2, 3, 4, 5, 0, 0], np.uint8)
    rc = lib.flexiq_layer_create_linear(C.byref(h), 128, 16, 16, dummy, dummy, None, pp, shifts.ctypes.data_as(C.c_void_p), None)
    assert rc == fx.ERR_INVALID_ARG and "exceeds 4" in fx.last_error()
    assert lib.flexiq_layer_create_linear(None, 128, 16, 16, dummy, dummy, None, pp, None, None) == fx.ERR_INVALID_ARG


def test_calls_reject_dead_handles(lib):
    assert lib.flexiq_set_lowbit_ratio(None, 0.5) == fx.ERR_INVALID_ARG
    assert lib.flexiq_layer_destroy(None) == fx.ERR_INVALID_ARG
    assert lib.flexiq_mixed_gemm(None, None, None, None, 1, 1.0, 1.0, 0, None, None) == fx.ERR_INVALID_ARG
    assert lib.flexiq_mixed_conv(None, None, None, None, 1, 1, 1, 1.0, 1.0, 0, None, None) == fx.ERR_INVALID_ARG
    assert lib.flexiq_quantize_lower(None, None, 0, 1, 1.0, 0, None, None, None, None, None) == fx.ERR_INVALID_ARG
    assert "handle" in fx.last_error()


def test_missing_library_fails_loudly(monkeypatch):
    monkeypatch.setattr(fx, "_lib", None)
    monkeypatch.setattr(fx, "LIB_PATH", "/nonexistent/libflexiq.so")
    with pytest.raises(FileNotFoundError, match="no CPU fallback"):
        fx.lib()


def test_host_calibration_matches_oracle():
    for case in (inputs.config1(), inputs.ranged_linear("g", 64, 256, 32, 32, seed=9, group_structured=True)):
        qcal = oracle.quantize(case.Xcal, case.x_scale)
        q2 = calib.quantize_reference(torch.from_numpy(case.Xcal), case.x_scale).numpy()
        assert np.array_equal(qcal, q2)
        lo, hi = oracle.channel_ranges(qcal)
        sx = oracle.static_positions(lo, hi, case.G)
        perm, _ = oracle.greedy_order(lo, hi, oracle.weight_absmax_linear(case.Wq), case.G)
        p2, s2 = calib.static_preparation(torch.from_numpy(q2), torch.from_numpy(case.Wq), case.G)
        assert np.array_equal(perm, p2) and np.array_equal(sx, s2)
    c = inputs.resnet_conv("c", 2, 6, 64, 16, 3, seed=3)
    qcal = oracle.quantize(c.Xcal, c.x_scale).reshape(-1, c.C)
    lo, hi = oracle.channel_ranges(qcal)
    perm, _ = oracle.greedy_order(lo, hi, oracle.weight_absmax_conv(c.Wq), c.G)
    p2, s2 = calib.static_preparation(torch.from_numpy(qcal), torch.from_numpy(c.Wq), c.G, conv=True)
    assert np.array_equal(perm, p2) and np.array_equal(oracle.static_positions(lo, hi, c.G), s2)


def test_inputs_are_seeded_and_shaped():
    a, b = inputs.config1(), inputs.config1()
    assert np.array_equal(a.X, b.X) and np.array_equal(a.Wq, b.Wq) and a.y_scale == b.y_scale
    assert a.X.shape == (256, 384) and a.Wq.shape == (384, 384) and a.Wq.dtype == np.int8
    u = inputs.uniform(1, 2, 1000)
    assert 0 <= u.min() and u.max() < 1 and abs(u.mean() - 0.5) < 0.05
    z = inputs.normal(1, 2, 20000)
    assert abs(z.mean()) < 0.05 and abs(z.std() - 1) < 0.05
    v = inputs.vit_linear("v", 32, 768, 64, seed=5)
    assert 20 <= v.meta["outlier_channels"] <= 60  # about 5 % of 768


def test_tile_choice_host_logic(lib):
    """The automatic tile shape (host-only hook): what the benchmark's four ViT-B layers get on 148 SMs, and
    properties that hold for every shape."""
    M = 64 * 197
    assert fx.flexiq_choose_tile(M, 2304, 6) == (2, 256)      # QKV: CTA pairs, 256 x 256
    assert fx.flexiq_choose_tile(M, 3072, 6) == (2, 256)      # fc1
    assert fx.flexiq_choose_tile(M, 768, 24) == (2, 192)      # fc2: 200 pair tiles fill three waves better than 150
    assert fx.flexiq_choose_tile(M, 768, 6) == (1, 192)       # proj
    rng = np.random.default_rng(5)
    for _ in range(300):
        m, n = int(rng.integers(1, 40000)), 16 * int(rng.integers(1, 300))
        kb, bk, sms = int(rng.integers(1, 40)), int(rng.choice([64, 128])), int(rng.choice([74, 132, 148]))
        cg, bn = fx.flexiq_choose_tile(m, n, kb, bk, sms)
        assert cg in (1, 2) and bn in (64, 128, 192, 256)
        assert not (cg == 2 and bn < 128)
        assert (cg, bn) == fx.flexiq_choose_tile(m, n, kb, bk, sms)      # a pure function of its arguments
    for bad in [(0, 64, 1, 128, 148), (5, 0, 1, 128, 148), (5, 64, 0, 128, 148), (5, 64, 1, 96, 148), (5, 64, 1, 128, 0)]:
        with pytest.raises(fx.FlexiqError):
            fx.flexiq_choose_tile(*bad)


# Nb, H, W, Cin, Cout, R, S: us as streamed patches and as im2col copies (prologue + convolution), and which of them runs
@pytest.mark.parametrize("shape, streamed, im2col", [
    ((32, 14, 14, 256, 256, 3, 3), 10.7, 12.9), ((32, 28, 28, 256, 256, 3, 3), 19.7, 20.9), ((8, 16, 16, 512, 512, 3, 3), 13.1, 16.4),
    ((32, 28, 28, 144, 144, 3, 3), 18.0, 21.7), ((1, 64, 64, 256, 256, 3, 3), 10.4, 12.5), ((8, 28, 28, 128, 512, 3, 3), 10.0, 10.7),
    ((32, 16, 16, 512, 512, 3, 3), 29.1, 20.7), ((32, 32, 32, 256, 256, 3, 3), 28.6, 22.3), ((8, 64, 64, 64, 256, 3, 3), 17.6, 12.5),
    ((4, 120, 64, 160, 160, 3, 3), 25.6, 20.1), ((32, 56, 56, 64, 256, 3, 3), 27.4, 23.6), ((5, 77, 77, 672, 352, 2, 2), 57.0, 38.7),
    ((12, 16, 16, 736, 208, 3, 1), 13.7, 12.1), ((32, 56, 56, 64, 192, 1, 3), 24.8, 17.4)])
def test_conv_kind_is_the_faster_one(lib, shape, streamed, im2col):
    assert fx.flexiq_choose_conv_kind(*shape, 1, shape[6] // 2) == (3 if streamed < im2col else 1)


def test_conv_kind_host_logic(lib):
    assert fx.flexiq_choose_conv_kind(32, 56, 56, 256, 64, 1, 1, 1, 0) == 0
    assert fx.flexiq_choose_conv_kind(32, 56, 56, 64, 64, 3, 3, 1, 1) == 2       # channels in a K block, outputs in a tile
    assert fx.flexiq_choose_conv_kind(32, 28, 28, 256, 256, 3, 3, 2, 1) == 1     # stride 2
    assert fx.flexiq_choose_conv_kind(8, 128, 128, 256, 256, 3, 3, 1, 1) == 1    # rows wider than a tile
    for bad in [(0, 8, 8, 64, 64, 3, 3, 1, 1), (1, 1, 8, 64, 64, 3, 3, 1, 0), (1, 8, 8, 64, 64, 3, 3, 0, 1), (1, 8, 8, 64, 64, 3, 3, 1, -1)]:
        with pytest.raises(fx.FlexiqError):
            fx.flexiq_choose_conv_kind(*bad)


def test_even_share_of_any_grid(tmp_path):
    """The shared memory that spreads a grid over the SMs: with it a share of the blocks and no more fits an SM, whatever the grid."""
    src = tmp_path / "share.cpp"
    src.write_text("""
#include "flexiq_internal.h"
#include <stdio.h>
int main()
{
    for (long long sms : {1ll, 74ll, 148ll})
        for (long long blocks = 1; blocks <= 1000000; blocks += 1 + blocks / 5000) {
            const long long smem = (long long)flexiq::even_share_smem(blocks, sms), share = (blocks + sms - 1) / sms;
            if (smem < 0 || smem > 113 * 1024 || (smem && (smem + 1024) * share > 228 * 1024) || (share < 200 && (smem + 1024) * (share + 2) < 228 * 1024)) {
                printf("%lld blocks on %lld SMs: %lld bytes\\n", blocks, sms, smem);
                return 1;
            }
        }
    return 0;
}
""")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(fxbuild._nvcc())))
    exe = str(tmp_path / "share")
    subprocess.run(["g++", "-std=c++17", *(f"-I{d}" for d in (fxbuild.CSRC, os.path.join(ROOT, "include"), os.path.join(cuda, "include"))), str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_kernels_that_overlap_their_predecessor_read_with_coherent_loads():
    """A non-coherent load is defined for memory that nobody writes while its kernel is resident; a kernel with a dependency wait is
    resident while the launches before it still write its inputs, its layer's tables (a layout) and its positions (a prologue)."""
    waiting = 0
    for name in sorted(os.listdir(fxbuild.CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        text = open(os.path.join(fxbuild.CSRC, name)).read()
        code = re.sub(r"//[^\n]*", "", text)
        for line in code.splitlines():
            assert ("__ldg(" not in line or "fsrc" in line) and "ld.global.nc" not in line, (name, line)
        for kernel in re.split(r"\b__global__\b", code)[1:]:
            head, body = kernel.split("{", 1)
            body = body.split("\n}\n", 1)[0]
            if "pdl_wait" in body:
                waiting += 1
                assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", head), (name, head)
    assert waiting >= 12
