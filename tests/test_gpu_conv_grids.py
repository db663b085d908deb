"""Convolutions whose tiles are grids of output positions read from halo patches: filters narrower than their padding,
whose output rows are wider than the padded input's left part."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_02822_b200 import binding as fx

pytestmark = pytest.mark.gpu


def check(Nb, H, W, C, N, R, S, stride, pad, G, ratio):
    dev = torch.device("cuda:0")
    rng = np.random.RandomState(Nb + 7 * H + 31 * W + C)
    Wq = rng.randint(-128, 128, (N, R, S, C)).astype(np.int8)
    X = rng.randint(-128, 128, (Nb, H, W, C)).astype(np.int8)
    n_g = C // G
    perm, sx = rng.permutation(n_g).astype(np.int32), rng.randint(0, 5, n_g).astype(np.uint8)
    ws, bias = (rng.rand(N) * 0.01 + 0.001).astype(np.float32), rng.randn(N).astype(np.float32)
    L = fx.Layer(torch.from_numpy(Wq).to(dev), torch.from_numpy(ws).to(dev), torch.from_numpy(bias).to(dev), perm, sx, G, conv=(stride, pad))
    L.set_lowbit_ratio(ratio)
    sw = oracle.weight_positions_conv(Wq, G, perm)
    acc = oracle.mixed_conv_acc(X, Wq, stride, pad, G, perm, sx[perm].copy(), sw, oracle.n_low(ratio, n_g)).reshape(-1, N)
    for _ in range(2):                                   # the second call finds its maps and weights as the first left them
        x4, x8, _ = L.quantize_lower(torch.from_numpy(X).to(dev), 1.0)
        got = {m: L.mixed_conv(x4, x8, Nb, H, W, 0.02 if m else 1.0, 3.0, m).cpu() for m in (fx.OUT_ACC_I32, fx.OUT_REQUANT_I8, fx.OUT_DEQUANT_F16)}
        assert np.array_equal(got[fx.OUT_ACC_I32].numpy().reshape(-1, N), acc)
        assert np.array_equal(got[fx.OUT_REQUANT_I8].numpy().reshape(-1, N), oracle.epilogue_i8(acc, 0.02, ws, bias, 3.0))
        assert np.array_equal(got[fx.OUT_DEQUANT_F16].numpy().reshape(-1, N).view(np.uint16), np.asarray(oracle.epilogue_f16(acc, 0.02, ws, bias)).view(np.uint16).reshape(-1, N))
    fx.flexiq_check_status()
    L.close()


@pytest.mark.parametrize("shape", [(2, 12, 15, 64, 64, 3, 1, 1, 1, 16, 0.5), (1, 9, 31, 128, 48, 2, 2, 1, 2, 16, 0.5), (2, 5, 7, 48, 32, 3, 1, 1, 1, 16, 1.0)])
def test_padding_wider_than_the_filter(shape):
    check(*shape)


# channels beyond a K block or outputs beyond a tile, one and several images per grid row, ragged channels and rows, wide
# images, one- and two-column filters, odd numbers of tiles (the pair's second tile outside)
@pytest.mark.parametrize("shape", [
    (2, 14, 14, 256, 64, 3, 3, 1, 1, 16, 0.5), (3, 7, 7, 512, 128, 3, 3, 1, 1, 16, 0.3), (1, 7, 7, 256, 64, 3, 3, 1, 1, 16, 1.0),
    (5, 7, 7, 144, 144, 3, 3, 1, 1, 16, 0.5), (4, 4, 4, 256, 80, 3, 3, 1, 1, 16, 0.0), (9, 3, 3, 128, 160, 3, 3, 1, 1, 16, 0.5),
    (2, 28, 28, 160, 48, 3, 3, 1, 1, 32, 0.25), (2, 30, 27, 144, 64, 3, 3, 1, 1, 16, 0.6), (1, 56, 56, 192, 32, 3, 3, 1, 1, 64, 0.4),
    (2, 12, 15, 256, 64, 3, 1, 1, 1, 16, 0.5), (2, 12, 15, 256, 64, 1, 3, 1, 1, 16, 0.5), (3, 9, 5, 208, 96, 5, 3, 1, 2, 16, 0.5),
    (1, 5, 90, 256, 16, 3, 3, 1, 1, 16, 0.5), (2, 16, 16, 64, 256, 3, 3, 1, 1, 16, 0.5), (7, 13, 8, 272, 272, 3, 3, 1, 0, 16, 0.7),
    (33, 7, 7, 256, 64, 2, 2, 1, 1, 16, 0.5), (32, 14, 14, 256, 256, 3, 3, 1, 1, 16, 0.5), (31, 7, 7, 512, 512, 3, 3, 1, 1, 16, 0.25)])
def test_streamed_patches(shape):
    check(*shape)
