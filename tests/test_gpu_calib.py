"""GPU parity of the device calibration kernels against the oracle: channel ranges of the
Eq. 1-quantized calibration batch, weight ranges, static positions, error scores, greedy order,
unused-bit histogram (integers: bit-exact) and the moving-average activation range (fp32: exact)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_02822_b200 import binding as fx
from paper_2510_02822_b200 import calib, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return torch.device("cuda:0")


def _check(case, dev, conv, batches, dtype=torch.float32):
    Xc = torch.from_numpy(case.Xcal).to(dev).to(dtype)
    perm, xs, info = calib.static_preparation_device(Xc, case.x_scale, torch.from_numpy(case.Wq).to(dev), case.G, conv=conv, batches=batches)
    C = case.Xcal.shape[-1]
    q = oracle.quantize(Xc.float().cpu().numpy().reshape(-1, C), case.x_scale)
    lo, hi = oracle.channel_ranges(q)
    assert np.array_equal(info["lo"].cpu().numpy(), lo) and np.array_equal(info["hi"].cpu().numpy(), hi)
    wmax = oracle.weight_absmax_conv(case.Wq) if conv else oracle.weight_absmax_linear(case.Wq)
    assert np.array_equal(info["wmax"].cpu().numpy(), wmax)
    assert np.array_equal(xs, oracle.static_positions(lo, hi, case.G))
    perm_e, score_e = oracle.greedy_order(lo, hi, wmax, case.G)
    assert np.array_equal(info["score"].cpu().numpy(), score_e)
    assert np.array_equal(perm, perm_e)
    assert np.array_equal(info["unused_hist"].cpu().numpy(), oracle.unused_bits_histogram(lo, hi))
    # and the host front end used elsewhere agrees with both
    perm_h, xs_h = calib.static_preparation(calib.quantize_reference(torch.from_numpy(case.Xcal).to(dtype), case.x_scale), torch.from_numpy(case.Wq), case.G, conv=conv)
    assert np.array_equal(perm_h, perm) and np.array_equal(xs_h, xs)


@pytest.mark.parametrize("K,N,G,batches", [(384, 384, 16, 1), (768, 2304, 16, 3), (3072, 768, 32, 2), (64, 16, 64, 1), (192, 80, 16, 5)])
def test_linear_calibration(dev, K, N, G, batches):
    _check(inputs.ranged_linear("c", 64, K, N, G, seed=K + N, group_structured=True), dev, False, batches)


def test_vit_outlier_channels_and_half_precision(dev):
    _check(inputs.vit_linear("v", 64, 768, 768, 16, seed=11), dev, False, 2)
    _check(inputs.ranged_linear("h", 64, 256, 64, 16, seed=12), dev, False, 1, dtype=torch.float16)
    _check(inputs.ranged_linear("b", 64, 256, 64, 16, seed=13), dev, False, 1, dtype=torch.bfloat16)


@pytest.mark.parametrize("H,C,Cout,R", [(14, 128, 64, 3), (28, 64, 256, 1), (7, 512, 512, 3)])
def test_conv_calibration(dev, H, C, Cout, R):
    _check(inputs.resnet_conv("c", 2, H, C, Cout, R, seed=H + C), dev, True, 2)


def test_wide_layer_and_ragged_window(dev):
    rng = np.random.default_rng(3)
    K = 8192 + 48  # 32 full channel windows and a partial one
    X = torch.from_numpy(rng.normal(0, 1, (40, K)).astype(np.float32)).to(dev)
    lo = torch.empty(K, dtype=torch.int32, device=dev)
    hi = torch.empty(K, dtype=torch.int32, device=dev)
    fx.flexiq_calib_channel_ranges(X, fx.DTYPE_F32, 40, K, 0.05, False, lo, hi)
    elo, ehi = oracle.channel_ranges(oracle.quantize(X.cpu().numpy(), 0.05))
    assert np.array_equal(lo.cpu().numpy(), elo) and np.array_equal(hi.cpu().numpy(), ehi)


@pytest.mark.parametrize("M,K,dt", [(700, 96, torch.float32), (3000, 768, torch.float16), (129, 1040, torch.int8)])
def test_histogram_and_coverage_ranges(dev, M, K, dt):
    rng = np.random.default_rng(M + K)
    xs = 0.05
    x = (rng.normal(0, 1, (M, K)) * rng.uniform(0.2, 6, (1, K))).astype(np.float32)
    if dt == torch.int8:
        X = torch.from_numpy(oracle.quantize(x, xs)).to(dev)
        q = X.cpu().numpy()
    else:
        X = torch.from_numpy(x).to(dt).to(dev)
        q = oracle.quantize(X.float().cpu().numpy(), xs)
    hist = torch.empty((K, 256), dtype=torch.int32, device=dev)
    half = M // 2
    fx.flexiq_calib_channel_histogram(X[:half], fx._dtype_code(X), half, K, xs, False, hist)
    fx.flexiq_calib_channel_histogram(X[half:], fx._dtype_code(X), M - half, K, xs, True, hist)
    eh = oracle.channel_histogram(q)
    assert np.array_equal(hist.cpu().numpy().view(np.uint32), eh)
    lo = torch.empty(K, dtype=torch.int32, device=dev)
    hi = torch.empty(K, dtype=torch.int32, device=dev)
    for tail in (0, int(M * 0.01 / 2), M):
        fx.flexiq_calib_ranges_from_histogram(hist, K, tail, lo, hi)
        elo, ehi = oracle.ranges_from_histogram(eh, tail)
        assert np.array_equal(lo.cpu().numpy(), elo) and np.array_equal(hi.cpu().numpy(), ehi)


def test_absmax_ema(dev):
    rng = np.random.default_rng(5)
    x = (rng.normal(0, 1, (7, 4096)) * rng.uniform(0.5, 4, (7, 1))).astype(np.float32)
    for dt in (torch.float32, torch.float16):
        xb = torch.from_numpy(x).to(dt).to(dev)
        state = torch.zeros(4, dtype=torch.float32, device=dev)
        for b in range(7):
            fx.flexiq_calib_absmax_ema(xb[b], fx._dtype_code(xb), xb[b].numel(), 0.99, state)
        s = state.cpu().numpy()
        assert s[1] == 7.0
        assert s[0] == np.float32(oracle.absmax_ema(xb.float().cpu().numpy(), 0.99))


def test_argument_errors(dev):
    z = torch.zeros(64, dtype=torch.int32, device=dev)
    x = torch.zeros((4, 64), dtype=torch.float32, device=dev)
    with pytest.raises(fx.FlexiqError):
        fx.flexiq_calib_channel_ranges(x, fx.DTYPE_F32, 4, 60, 0.1, False, z, z)       # K not a multiple of 16
    with pytest.raises(fx.FlexiqError):
        fx.flexiq_calib_channel_ranges(x, fx.DTYPE_F32, 4, 64, 0.0, False, z, z)       # scale must be positive
    with pytest.raises(fx.FlexiqError):
        fx.flexiq_calib_prepare(z, z, z, 64, 24, z, z, z, z)                           # group size
    with pytest.raises(fx.FlexiqError):
        fx.flexiq_calib_absmax_ema(x, fx.DTYPE_I8, 256, 0.99, x)                       # integer input has no range to track


def test_front_end_with_coverage(dev):
    case = inputs.vit_linear("v", 64, 768, 768, 16, seed=17)
    Xc = torch.from_numpy(case.Xcal).to(dev)
    perm, xs, info = calib.static_preparation_device(Xc, case.x_scale, torch.from_numpy(case.Wq).to(dev), case.G, batches=3, coverage=0.99)
    q = oracle.quantize(case.Xcal, case.x_scale)
    lo, hi = oracle.ranges_from_histogram(oracle.channel_histogram(q), int(q.shape[0] * (1.0 - 0.99) / 2.0))
    assert np.array_equal(info["lo"].cpu().numpy(), lo) and np.array_equal(info["hi"].cpu().numpy(), hi)
    assert np.array_equal(xs, oracle.static_positions(lo, hi, case.G))
    perm_e, _ = oracle.greedy_order(lo, hi, oracle.weight_absmax_linear(case.Wq), case.G)
    assert np.array_equal(perm, perm_e)


@pytest.mark.parametrize("K, N, taps, offset", [(16, 1, 0, 0), (48, 17, 0, 0), (33, 512, 0, 0), (70, 528, 0, 1), (768, 3072, 0, 0),
                                                (16, 1, 9, 0), (272, 48, 9, 0), (260, 32, 1, 0), (512, 130, 9, 4), (4096, 3, 1, 0)])
def test_weight_ranges_wide_and_byte_loads(dev, K, N, taps, offset):
    """Rows that allow 16-byte loads and rows that do not (odd lengths, odd addresses), -128 among the weights."""
    shape = (N, taps, K) if taps else (K, N)
    w = ((inputs.uniform(77, K, int(np.prod(shape))) * 256).astype(np.int64) - 128).astype(np.int8)
    w = (w >> (np.arange(w.size) % 5)).astype(np.int8)
    w[-1] = -128
    raw = torch.empty(w.size + 16, dtype=torch.int8, device=dev)
    W = raw[offset:offset + w.size]
    W.copy_(torch.from_numpy(w))
    wmax = torch.full((K,), -1, dtype=torch.int32, device=dev)
    fx.flexiq_calib_weight_absmax(W, bool(taps), K, N, max(taps, 1), wmax)
    ref = np.abs(w.astype(np.int32).reshape(shape)).max(axis=(0, 1) if taps else 1)
    assert np.array_equal(wmax.cpu().numpy(), ref)


@pytest.mark.parametrize("K, G", [(16, 16), (2048 * 16, 16), (2049 * 16, 16), (4096, 64)])
def test_prepare_few_and_many_groups(dev, K, G):
    """Group scores and order where they meet in shared memory and where they do not, ties included."""
    lo = -(inputs.uniform(78, 0, K) * 129).astype(np.int32)
    hi = (inputs.uniform(78, 1, K) * 128).astype(np.int32)
    wm = (inputs.uniform(78, 2, K) * 3).astype(np.int32)
    t = [torch.from_numpy(a).to(dev) for a in (lo, hi, wm)]
    n_g = K // G
    perm, xs = torch.empty(n_g, dtype=torch.int32, device=dev), torch.empty(n_g, dtype=torch.uint8, device=dev)
    score, hist = torch.empty(n_g, dtype=torch.int64, device=dev), torch.empty(5, dtype=torch.int32, device=dev)
    fx.flexiq_calib_prepare(*t, K, G, perm, xs, score, hist)
    ref = (np.maximum(hi, -lo).astype(np.int64) * wm).reshape(n_g, G).max(1)
    assert np.array_equal(score.cpu().numpy(), ref)
    assert np.array_equal(perm.cpu().numpy(), np.argsort(ref, kind="stable"))
    assert np.array_equal(xs.cpu().numpy(), oracle.static_positions(lo, hi, G))
    assert np.array_equal(hist.cpu().numpy(), oracle.unused_bits_histogram(lo, hi))


def test_coverage_that_is_no_number():
    X, W = torch.randn((64, 32), device="cuda"), torch.ones((32, 16), dtype=torch.int8, device="cuda")
    for coverage, error in ((float("nan"), ValueError), (float("-inf"), OverflowError)):
        with pytest.raises(error):
            calib.static_preparation_device(X, 0.1, W, 16, coverage=coverage)
    perm, x_shift, _ = calib.static_preparation_device(X, 0.1, W, 16, coverage=0.99)
    assert sorted(perm.tolist()) == [0, 1]


@pytest.mark.parametrize("K,N,G,rows,shape,dtype,coverage,offset", [
    (128, 128, 16, 256, "linear", torch.float32, None, 0), (272, 48, 16, 257, "linear", torch.float16, None, 0), (4096, 64, 64, 1000, "linear", torch.bfloat16, None, 0),
    (512 * 16, 16, 16, 33, "linear", torch.int8, None, 0), (513 * 16, 16, 16, 33, "linear", torch.float32, None, 0),   # the most groups in one launch, and one more
    (768, 80, 16, 300, "linear", torch.float32, None, 1), (256, 48, 32, 999, "conv", torch.float16, None, 0), (48, 16, 16, 5, "conv", torch.float32, None, 3),
    (720, 1104, 16, 2000, "linear", torch.float32, 0.99, 0), (160, 32, 32, 500, "conv", torch.bfloat16, 0.9, 0)])
def test_one_launch_equals_the_calls_it_stands_for(dev, K, N, G, rows, shape, dtype, coverage, offset):
    g = torch.Generator(device=dev).manual_seed(K + rows)
    X = torch.randn((rows, K), generator=g, device=dev) * torch.exp(torch.randn(K, generator=g, device=dev))
    X = torch.clamp(X * 30, -128, 127).to(dtype) if dtype == torch.int8 else X.to(dtype)
    size = (N, 3, 3, K) if shape == "conv" else (K, N)
    raw = torch.randint(-128, 128, (int(np.prod(size)) + 16,), generator=g, device=dev, dtype=torch.int8)
    W = raw[offset:offset + int(np.prod(size))].view(size)
    perm, xs, info = calib.static_preparation_device(X, 0.05, W, G, conv=shape == "conv", coverage=coverage)
    lo, hi, wmax = (torch.empty(K, dtype=torch.int32, device=dev) for _ in range(3))
    if coverage is None:
        fx.flexiq_calib_channel_ranges(X, fx._dtype_code(X), rows, K, 0.05, False, lo, hi)
    else:
        hist = torch.empty((K, 256), dtype=torch.int32, device=dev)
        fx.flexiq_calib_channel_histogram(X, fx._dtype_code(X), rows, K, 0.05, False, hist)
        fx.flexiq_calib_ranges_from_histogram(hist, K, int(rows * (1.0 - coverage) / 2.0), lo, hi)
    fx.flexiq_calib_weight_absmax(W, shape == "conv", K, N, 9 if shape == "conv" else 1, wmax)
    perm_e, xs_e = torch.empty(K // G, dtype=torch.int32, device=dev), torch.empty(K // G, dtype=torch.uint8, device=dev)
    score, unused = torch.empty(K // G, dtype=torch.int64, device=dev), torch.empty(5, dtype=torch.int32, device=dev)
    fx.flexiq_calib_prepare(lo, hi, wmax, K, G, perm_e, xs_e, score, unused)
    assert np.array_equal(perm, perm_e.cpu().numpy()) and np.array_equal(xs, xs_e.cpu().numpy())
    for name, want in (("lo", lo), ("hi", hi), ("wmax", wmax), ("score", score), ("unused_hist", unused)):
        assert torch.equal(info[name], want), name


def test_interpreter_out_of_memory_is_reported(dev):
    """An allocation of Python's that fails behind the launch is a MemoryError: not swallowed, not answered with "take the general path"."""
    testcapi = pytest.importorskip("_testcapi")
    native = fx._native_calls()
    if native is None:
        pytest.skip("built without the native module")
    X, W = torch.randn((64, 64), device=dev), torch.randint(-128, 128, (64, 48), device=dev, dtype=torch.int8)
    args = (X, 0.1, W, 16, False, 1, None)
    call, arm, disarm = native.static_preparation, testcapi.set_nomemory, testcapi.remove_mem_hooks
    want = call(*args)
    failed = 0
    for k in range(40):
        got = None
        arm(k, k + 1)
        try:
            got = call(*args)
        except MemoryError:
            failed += 1
        finally:
            disarm()
        assert got is not NotImplemented, k
        if got is not None:
            assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert failed
