"""The activation prologue at the edges of its kernel: the one- and two-operation forms of Eq. 1's division against
IEEE division over whole input types and next to every rounding boundary, and the tiling's edges (few and many rows,
ragged last tiles, narrow and wide rows), every group size, static and dynamic positions."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_02822_b200 import binding as fx
from paper_2510_02822_b200 import inputs

pytestmark = pytest.mark.gpu
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16, "i8": torch.int8}


def make_layer(K, G, perm=None, sx=None, N=16):
    dev = torch.device("cuda:0")
    W = torch.from_numpy((inputs.uniform(3, K, K * N) * 255).astype(np.int64) - 127).to(torch.int8).reshape(K, N).to(dev)
    perm = np.arange(K // G, dtype=np.int32) if perm is None else perm
    return fx.Layer(W, torch.ones(N, device=dev), None, perm, sx, G)


def slab(L, X, scale, **kw):
    x4, _, pos = L.quantize_lower(X, scale, **kw)
    M = X.numel() // L.K
    return x4[:M * L.K].view(torch.int8).view(M, L.K).cpu().numpy(), pos


def ieee(x, S):
    with np.errstate(over="ignore"):
        return np.clip(np.rint(x.astype(np.float32) / np.float32(S)), -128, 127).astype(np.int8)


def scales(kind):
    """Ordinary scales, powers of two and their neighbours, few-bit significands, and scales that put an input of the
    type next to a half-integer (where the short forms of the division are refused or just hold)."""
    f = np.float32
    out = [f(0.0317), f(1.0), f(2.0 ** -14), f(3.0) * f(2.0 ** -9), f(1e-3), f(0.75)]
    out += [f(2.0 ** -5) * (f(1.0) + f(d) * f(2.0 ** -23)) for d in (1, 3, 8, 9, 64)]
    step = {"f16": 2.0 ** -10, "bf16": 2.0 ** -7, "f32": 2.0 ** -23}[kind]
    for i, k in enumerate((0, 1, 2, 7, 30, 63, 64, 100, 126, 127)):
        s = f((1.0 + (37 * i + 5) % 97 * step) / (k + 0.5))
        out += [s, np.nextafter(s, f(0)), np.nextafter(s, f(1e9))]
    return out


@pytest.mark.parametrize("kind", ["f16", "bf16"])
def test_every_16_bit_input(kind):
    bits = np.arange(65536, dtype=np.uint16)
    t = torch.from_numpy(bits.view(np.int16)).view(DTYPES[kind])
    t = t[~torch.isnan(t.float())]
    t = torch.cat([t, t[:(-t.numel()) % 64]])
    X = t.cuda().view(-1, 64)
    L = make_layer(64, 16)
    for S in scales(kind):
        got, _ = slab(L, X, float(S))
        assert np.array_equal(got.reshape(-1), ieee(t.float().numpy(), S)), float(S)
    L.close()


def test_fp32_next_to_every_boundary():
    L = make_layer(64, 16)
    near = np.arange(-6, 7, dtype=np.int32)
    for S in scales("f32"):
        at = ((np.arange(-129, 129) + 0.5) * np.float64(S)).astype(np.float32)
        x = (at.view(np.int32)[:, None] + near).view(np.float32).reshape(-1)
        x = np.concatenate([x, np.array([np.inf, -np.inf, 0.0, -0.0, 1e-45, -1e-45, 3e38, -3e38], np.float32)])
        x = np.concatenate([x, np.zeros((-x.size) % 64, np.float32)])
        got, _ = slab(L, torch.from_numpy(x).cuda().view(-1, 64), float(S))
        assert np.array_equal(got.reshape(-1), ieee(x, S)), float(S)
    L.close()


def test_scales_and_types_in_turn_on_one_layer():
    """The plan of the division belongs to a scale and a type: changing either between calls, scales far outside the inputs' range."""
    rng = np.random.RandomState(4)
    L = make_layer(64, 16)
    tiny = [np.float32(1.0901 * 2.0 ** e) for e in (-71, -49, -24, 20, 60)]
    for i, S in enumerate((tiny + scales("f16") + scales("bf16") + tiny) * 2):
        kind = ("f16", "bf16", "f32", "i8")[(i * 7 + i // 4) % 4]
        x = rng.randn(64, 64).astype(np.float32) * np.float32(min(max(float(S) * 90, 1e-6), 2e4))
        t = torch.from_numpy(x).to(DTYPES[kind]) if kind != "i8" else torch.from_numpy(rng.randint(-128, 128, (64, 64)).astype(np.int8))
        got, _ = slab(L, t.cuda(), float(S))
        assert np.array_equal(got, ieee(t.float().numpy(), S) if kind != "i8" else t.numpy()), (kind, float(S))
    L.close()


@pytest.mark.parametrize("kind", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("M", [5, 40000])                # the one-launch dynamic kernel, and the two phases
def test_infinities_and_nan(kind, M):
    perm, sx = np.array([3, 0, 2, 1], np.int32), np.array([0, 1, 2, 4], np.uint8)
    X = torch.zeros((M, 64))
    X[0, ::16], X[1, ::16], X[2, ::16] = float("nan"), float("inf"), float("-inf")
    X = X.to(DTYPES[kind]).cuda()
    for path in (fx.LOWBIT_MASKED_I8, fx.LOWBIT_PACKED_U4):
        L = make_layer(64, 16, perm, sx)
        L.set_lowbit_path(path)
        general = [np.float32(0.1) * np.float32(2.0 ** -110)]   # outside the short forms' range
        for S in scales(kind) + general:
            for ratio in (0.0, 0.5):
                L.set_lowbit_ratio(ratio)
                if path == fx.LOWBIT_MASKED_I8:
                    for dynamic in (False, True):
                        got, pos = slab(L, X, float(S), dynamic=dynamic)
                        s = pos.cpu().numpy().astype(int) if dynamic else sx[perm].astype(int)
                        lowered = np.arange(4) < 4 * ratio
                        top, bottom = np.where(lowered, 7 << s, 127), np.where(lowered, -8 << s, -128)
                        assert np.array_equal(got[:3, ::16], np.stack([top, top, bottom]).astype(np.int8)), (float(S), ratio, dynamic)
                elif ratio == 0.0:
                    _, x8, _ = L.quantize_lower(X, float(S))
                    assert x8[:192].view(3, 64)[:, ::16].cpu().tolist() == [[127] * 4, [127] * 4, [-128] * 4], float(S)
        L.close()
    fx.flexiq_check_status()


# rows x channels: one row, one chunk, fewer tiles than SMs, ragged last tiles, rows of one chunk per thread and of many, the widest
# rows of the ring for each type (65,536 bytes) and wider ones; rows beyond what the one-launch dynamic kernel holds
@pytest.mark.parametrize("kind", ["f32", "f16", "bf16", "i8"])
@pytest.mark.parametrize("M, K, G", [(1, 16, 16), (3, 144, 16), (197, 384, 32), (5000, 64, 64), (2111, 1360, 16), (2200, 1216, 64),
                                     (9001, 96, 32), (26001, 32, 16), (13000, 64, 64), (333, 4112, 16), (151, 16384, 64), (2, 65536, 32), (2, 132000, 32)])
def test_slab_matches_oracle(kind, M, K, G):
    n_g = K // G
    perm = np.argsort(inputs.uniform(11, K, n_g), kind="stable").astype(np.int32)
    sx = (np.arange(n_g) % 5).astype(np.uint8)
    q = ((inputs.uniform(12, M, M * K) * 256).astype(np.int64) - 128)
    q = (q >> np.tile(np.repeat((inputs.uniform(13, K, n_g) * 6).astype(np.int64), G), M)).astype(np.int8).reshape(M, K)
    X = torch.from_numpy(q).cuda().to(DTYPES[kind])
    if kind != "i8":
        X = X * 0.25                                     # exact in every type
    L = make_layer(K, G, perm, sx)
    cols = (perm[:, None].astype(np.int64) * G + np.arange(G)).reshape(-1)
    dyn_sx = oracle.dynamic_positions(q, G, perm)
    for ratio in (0.0, 0.4, 1.0):
        L.set_lowbit_ratio(ratio)
        n_low = oracle.n_low(ratio, n_g)
        for dynamic in (False, True):
            s = np.where(np.arange(n_g) < n_low, dyn_sx if dynamic else sx[perm], 0).astype(np.int64)
            s = np.repeat(s, G)
            low = np.repeat(np.arange(n_g) < n_low, G)
            v = q[:, cols].astype(np.int64)
            ref = np.where(low, (np.clip(v, -(8 << s), (8 << s) - 1) >> s) << s, v).astype(np.int8)
            got, pos = slab(L, X, 0.25, dynamic=dynamic)
            assert np.array_equal(got, ref), (ratio, dynamic)
            if dynamic:
                assert np.array_equal(pos.cpu().numpy(), dyn_sx)
    fx.flexiq_check_status()
    L.close()


def test_copies_in_flight_land_when_a_wait_expires():
    src = torch.arange(49152, dtype=torch.int64, device="cuda").mul_(40503).bitwise_right_shift_(7).to(torch.uint8)
    res = torch.zeros(5, dtype=torch.int32, device="cuda")
    fx.flexiq_selftest_copy_drain(src, res)
    with pytest.raises(fx.FlexiqError) as e:
        fx.flexiq_check_status()
    assert e.value.code == fx.ERR_TIMEOUT
    assert res.cpu().tolist() == [1, 0, 1, 1, 0]
    fx.flexiq_check_status()                             # reported once
