"""Layout post-processing of a handle: the slab-order weights, their 4-bit form and the positions of every
(group, output channel) against the oracle and a plain gather, at the edges of the kernels' tiles (64 output
channels x 128 input channels; whole convolution rows), for every group size, for weights at odd addresses and
for more groups than a launch's parameters carry."""
import contextlib

import numpy as np
import pytest
import torch

import oracle
from paper_2510_02822_b200 import binding as fx
from paper_2510_02822_b200 import inputs

pytestmark = pytest.mark.gpu


def draw(seed, shape):
    w = (inputs.uniform(seed, 0, int(np.prod(shape))) * 256).astype(np.int64) - 128
    narrow = np.repeat((inputs.uniform(seed, 1, -(-w.size // 32)) * 6).astype(np.int64), 32)[:w.size]   # every position occurs
    return (w >> narrow).astype(np.int8).reshape(shape)


@pytest.mark.parametrize("shape, G, offset", [
    ((16, 16), 16, 0), ((128, 64), 16, 0), ((144, 80), 16, 0), ((112, 48), 16, 1), ((192, 208), 64, 0), ((320, 64), 32, 2),
    ((1025 * 16, 16), 16, 0),                                                  # linear [K, N]
    ((16, 1, 1, 16), 16, 0), ((48, 3, 3, 80), 16, 0), ((64, 3, 3, 64), 64, 4), ((160, 1, 1, 544), 32, 0), ((16, 5, 3, 272), 16, 0),
    ((32, 1, 1, 1025 * 16), 16, 0), ((16, 1, 1, 2049 * 16), 16, 0)])           # convolution [N, R, S, C]
def test_layout_matches_oracle(shape, G, offset):
    dev = torch.device("cuda:0")
    conv = len(shape) == 4
    W = draw(500 + G + shape[0], shape)
    C, N = (shape[3], shape[0]) if conv else shape
    T, n_g = W.size // (C * N), C // G
    raw = torch.empty(W.size + 16, dtype=torch.int8, device=dev)
    Wd = raw[offset:offset + W.size].view(shape)
    Wd.copy_(torch.from_numpy(W))
    ones = torch.ones(N, device=dev)
    L = fx.Layer(Wd, ones, None, np.arange(n_g, dtype=np.int32), None, G, conv=(1, 0) if conv else None)
    sx = (np.arange(n_g) % 5).astype(np.uint8)
    for perm in (np.arange(n_g, dtype=np.int32)[::-1].copy(), np.argsort(inputs.uniform(7, 2, n_g), kind="stable").astype(np.int32)):
        L.set_group_perm(Wd, perm, sx)
        cols = (perm[:, None].astype(np.int64) * G + np.arange(G)).reshape(-1)
        slab = (W[..., cols] if conv else W[cols].T).reshape(N, T, C)
        sw = oracle.weight_positions_conv(W, G, perm) if conv else oracle.weight_positions_linear(W, G, perm)
        s = np.repeat(sw.reshape(n_g, N).T.astype(np.int64), G, axis=1)[:, None, :]
        nib = ((slab.astype(np.int64) >> s) & 15).astype(np.uint8).reshape(N, T * C)
        sw_g, w8, w4 = np.empty((n_g, N), np.uint8), np.empty((N, T * C), np.int8), np.empty((N, T * C // 2), np.uint8)
        fx.flexiq_layer_export(L.h, sw_g, w8, w4)
        assert np.array_equal(sw_g, sw.reshape(n_g, N))
        assert np.array_equal(w8, slab.reshape(N, T * C))
        assert np.array_equal(w4, nib[:, 0::2] | (nib[:, 1::2] << 4))
        # the masked weights, the order and the activation positions through the mixed kernel itself (one tap of input)
        if not conv:
            X = draw(900, (5, C))
            for ratio in (1.0, 0.5):
                L.set_lowbit_ratio(ratio)
                x4, x8, _ = L.quantize_lower(torch.from_numpy(X).to(dev), 1.0)
                acc = L.mixed_gemm(x4, x8, 5, 1.0, 1.0, fx.OUT_ACC_I32)
                assert np.array_equal(acc.cpu().numpy(), oracle.mixed_gemm_acc(X, W, G, perm, sx[perm].copy(), sw, oracle.n_low(ratio, n_g)))
        else:
            R, S = shape[1], shape[2]
            X = draw(901, (1, R, S, C))
            for ratio in (1.0, 0.5):
                L.set_lowbit_ratio(ratio)
                x4, x8, _ = L.quantize_lower(torch.from_numpy(X).to(dev), 1.0)
                acc = L.mixed_conv(x4, x8, 1, R, S, 1.0, 1.0, fx.OUT_ACC_I32)
                ref = oracle.mixed_conv_acc(X, W, 1, 0, G, perm, sx[perm].copy(), sw, oracle.n_low(ratio, n_g))
                assert np.array_equal(acc.cpu().numpy().reshape(-1), ref.reshape(-1))
    fx.flexiq_check_status()
    L.close()


@pytest.mark.parametrize("K, N, G", [(112, 48, 16), (144, 80, 16), (400, 64, 16), (192, 208, 64), (128, 16, 16)])
def test_layout_cuts_the_block_of_the_ratio_in_force(K, N, G):
    """A layout made at a ratio inside a K block: the weight block that holds both kinds of channels is the new order's, and a GEMM
    that follows without another prologue reads it."""
    dev = torch.device("cuda:0")
    n_g = K // G
    W, X = draw(700 + K, (K, N)), draw(701 + K, (70, K))
    Wd, Xd, ones = torch.from_numpy(W).to(dev), torch.from_numpy(X).to(dev), torch.ones(N, device=dev)
    sx = (np.arange(n_g) % 5).astype(np.uint8)
    L = fx.Layer(Wd, ones, None, np.arange(n_g, dtype=np.int32), sx, G)
    for low in range(n_g + 1):
        perm = np.argsort(inputs.uniform(70 + low, 2, n_g), kind="stable").astype(np.int32)
        flags = np.zeros(n_g, np.uint8)
        flags[perm[:low]] = 1
        L.select_groups(Wd, flags, sx)
        order = np.concatenate([np.flatnonzero(flags), np.flatnonzero(flags == 0)]).astype(np.int32)
        sw = oracle.weight_positions_linear(W, G, order)
        x4, x8, _ = L.quantize_lower(Xd, 1.0)
        acc = L.mixed_gemm(x4, x8, 70, 1.0, 1.0, fx.OUT_ACC_I32)
        assert np.array_equal(acc.cpu().numpy(), oracle.mixed_gemm_acc(X, W, G, order, sx[order].copy(), sw, low)), low
        # other weights in the same order, so that the slab stays what it is: the GEMM finds the block cut and launches nothing for it
        W2 = draw(702 + low, (K, N))
        L.select_groups(torch.from_numpy(W2).to(dev), flags, sx)
        watched = low in (1, n_g // 2, n_g - 1)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) if watched else contextlib.nullcontext() as seen:
            acc = L.mixed_gemm(x4, x8, 70, 1.0, 1.0, fx.OUT_ACC_I32)
            torch.cuda.synchronize()
        if watched:
            launched = [e.key for e in seen.key_averages() if "flexiq::" in e.key]
            assert len(launched) == 1 and "mixed_gemm_kernel" in launched[0], launched
        sw = oracle.weight_positions_linear(W2, G, order)
        assert np.array_equal(acc.cpu().numpy(), oracle.mixed_gemm_acc(X, W2, G, order, sx[order].copy(), sw, low)), low
    fx.flexiq_check_status()
    L.close()


@pytest.mark.parametrize("shapes", [
    [(144, 80, 16), (112, 48, 16)], [(192, 208, 64), (128, 16, 16), (400, 64, 16), (64, 64, 16), (768, 96, 16)],      # two in a launch; four and one
    [(600 * 16, 16, 16), (500 * 16, 16, 16), (32, 16, 16)], [(1025 * 16, 16, 16), (64, 32, 32)]])   # more groups than a launch carries, together and alone
def test_several_layers_laid_out_at_once(shapes):
    dev = torch.device("cuda:0")
    made = []
    for i, (K, N, G) in enumerate(shapes):
        W, n_g = draw(800 + i, (K, N)), K // G
        sx = (np.arange(n_g) % 5).astype(np.uint8)
        Wd = torch.from_numpy(W).to(dev)
        made.append((W, Wd, G, n_g, sx, fx.Layer(Wd, torch.ones(N, device=dev), None, np.arange(n_g, dtype=np.int32), sx, G)))
    for turn in range(2):
        flags = [(inputs.uniform(80 + turn, i, m[3]) < 0.4).astype(np.uint8) for i, m in enumerate(made)]
        fx.select_groups([(m[5], m[1], f, m[4]) for m, f in zip(made, flags)])
        for (W, Wd, G, n_g, sx, L), f in zip(made, flags):
            order, low = np.concatenate([np.flatnonzero(f), np.flatnonzero(f == 0)]).astype(np.int32), int(f.sum())
            assert L.K_lo == low * G
            X = draw(850, (5, W.shape[0]))
            sw = oracle.weight_positions_linear(W, G, order)
            x4, x8, _ = L.quantize_lower(torch.from_numpy(X).to(dev), 1.0)
            acc = L.mixed_gemm(x4, x8, 5, 1.0, 1.0, fx.OUT_ACC_I32)
            assert np.array_equal(acc.cpu().numpy(), oracle.mixed_gemm_acc(X, W, G, order, sx[order].copy(), sw, low))
            sw_g, w8, w4 = np.empty((n_g, W.shape[1]), np.uint8), np.empty((W.shape[1], W.shape[0]), np.int8), np.empty((W.shape[1], W.shape[0] // 2), np.uint8)
            fx.flexiq_layer_export(L.h, sw_g, w8, w4)
            assert np.array_equal(sw_g, sw.reshape(n_g, -1))
    # one handle twice, or a position that is none: refused, and nothing has changed
    m, before = made[0], made[0][5].K_lo
    bad = m[4].copy()
    bad[0] = 5
    for args in ([(m[5], m[1], np.ones(m[3], np.uint8), m[4])] * 2, [(m[5], m[1], np.ones(m[3], np.uint8), bad)]):
        with pytest.raises(fx.FlexiqError):
            fx.select_groups(args)
        assert m[5].K_lo == before
    fx.flexiq_check_status()
    for m in made:
        m[5].close()


@pytest.mark.parametrize("widths", [(67264,), (34304, 34304)])   # 33,632 and 2 x 17,152 blocks of one launch: more than 227 an SM
def test_layout_of_very_large_layers(widths):
    """Each alone when it is created, and together in one launch; a few output columns against the oracle."""
    dev, K, G = torch.device("cuda:0"), 4096, 64
    n_g = K // G
    gen = torch.Generator(device=dev).manual_seed(widths[0])
    sx = (np.arange(n_g) % 5).astype(np.uint8)
    X = draw(860, (5, K))
    made = []
    for N in widths:
        W = torch.randint(-128, 128, (K, N), generator=gen, device=dev, dtype=torch.int8)
        W >>= torch.randint(0, 6, (n_g, N), generator=gen, device=dev, dtype=torch.int8).repeat_interleave(G, 0)
        made.append((W, fx.Layer(W, torch.ones(N, device=dev), None, np.arange(n_g, dtype=np.int32), sx, G)))

    def check(L, W, order, low):
        cols = np.unique(np.concatenate([np.arange(16), np.linspace(0, L.N - 1, 97).astype(np.int64), np.arange(L.N - 16, L.N)]))
        Wc = np.ascontiguousarray(W[:, torch.from_numpy(cols).to(dev)].cpu().numpy())
        x4, x8, _ = L.quantize_lower(torch.from_numpy(X).to(dev), 1.0)
        acc = L.mixed_gemm(x4, x8, 5, 1.0, 1.0, fx.OUT_ACC_I32).cpu().numpy()
        sw = oracle.weight_positions_linear(Wc, G, order)
        assert np.array_equal(acc[:, cols], oracle.mixed_gemm_acc(X, Wc, G, order, sx[order].copy(), sw, low))

    for W, L in made:
        L.set_lowbit_ratio(0.5)
        check(L, W, np.arange(n_g, dtype=np.int32), n_g // 2)
    flags = [(inputs.uniform(90, i, n_g) < 0.4).astype(np.uint8) for i in range(len(made))]
    fx.select_groups([(L, W, f, sx) for (W, L), f in zip(made, flags)])
    for (W, L), f in zip(made, flags):
        check(L, W, np.concatenate([np.flatnonzero(f), np.flatnonzero(f == 0)]).astype(np.int32), int(f.sum()))
    fx.flexiq_check_status()
    for _, L in made:
        L.close()


def test_selections_in_python_as_in_native_code():
    """Without the native module: the same layouts in the same call, and a refused one changes nothing."""
    dev = torch.device("cuda:0")
    pairs = []
    for i, (K, N, G) in enumerate([(144, 80, 16), (192, 208, 64), (112, 48, 16)]):
        Wd, n_g = torch.from_numpy(draw(870 + i, (K, N))).to(dev), K // G
        sx = (np.arange(n_g) % 5).astype(np.uint8)
        pair = [fx.Layer(Wd, torch.ones(N, device=dev), None, np.arange(n_g, dtype=np.int32), sx, G) for _ in range(2)]
        pair[1]._calls = None
        pairs.append((pair, Wd, (inputs.uniform(95, i, n_g) < 0.4).astype(np.uint8), sx))

    def same():
        for (a, b), Wd, _, _ in pairs:
            assert a.K_lo == b.K_lo
            X = torch.from_numpy(draw(880, (7, a.K))).to(dev)
            ya, yb = (L.mixed_gemm(*L.quantize_lower(X, 1.0)[:2], 7, 1.0, 1.0, fx.OUT_ACC_I32) for L in (a, b))
            assert torch.equal(ya, yb)
    for k in (0, 1):
        fx.select_groups([(pair[k], Wd, f, sx) for pair, Wd, f, sx in pairs])
    same()
    first, last = pairs[0], pairs[-1]
    bad = last[3].copy()
    bad[-1] = 5
    ones = [np.ones_like(p[2]) for p in pairs]
    for args in ([(p[0][1], p[1], o, p[3]) for p, o in zip(pairs[:-1], ones)] + [(last[0][1], last[1], ones[-1], bad)],
                 [(first[0][1], first[1], ones[0], first[3])] * 2):
        with pytest.raises(fx.FlexiqError):
            fx.select_groups(args)
        same()
    fx.flexiq_check_status()
    for pair, *_ in pairs:
        for L in pair:
            L.close()
