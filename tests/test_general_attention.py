"""The general fused attention kernel (rows of up to 1024 keys, windows of up to 256 keys with a bias and a
mask), bit for bit against the oracle at the edges of its blocks, tiles and rings."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_13824_gb300 import build as fbuild
from paper_2111_13824_gb300 import fqvit, synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fbuild.build()
    fqvit.load()
    oracle.build()


def _inputs(seed, BH, L, d, pad=0, peaked=False):
    rng = np.random.default_rng(seed)
    ld = (L + 15) // 16 * 16 + pad
    x = rng.integers(-128, 128, size=(BH * L, ld)).astype(np.int8)
    if peaked:  # most keys far below a few
        x[:, :L] = np.where(rng.random((BH * L, L)) < 0.02, x[:, :L], np.minimum(x[:, :L], -60))
    v = rng.integers(-128, 128, size=(BH, L, d)).astype(np.int8)
    return x, v


def _check(x, L, s, v, zp, bias=None, heads=1, window=0, region=None, mask=0):
    kw = dict(bias=bias, heads=heads, window=window) if bias is not None else {}
    mk = dict(region=region, mask_value=mask) if region is not None else {}
    co, _ = oracle.lis_softmax(x, L, s, **kw, **mk)
    want, over = oracle.lis_attn_v(co, v, zp)
    assert not over
    T = lambda a: None if a is None else torch.from_numpy(a).to(DEV)  # noqa: E731
    gkw = dict(bias=T(bias), heads=heads, window=window) if bias is not None else {}
    args = (T(x), s, T(v), T(region), mask)
    got = fqvit.lis_attention_masked(*args, zp_v=zp, **gkw)
    fqvit.sync_status()
    assert np.array_equal(got.cpu().numpy(), want)
    s_v, s_out, zp_out = 0.02, 0.031, 117
    got8 = fqvit.lis_attention_masked_q(*args, zp, s_v, s_out, zp_out, **gkw)
    fqvit.sync_status()
    assert np.array_equal(got8.cpu().numpy(), oracle.attn_requant(want, s_v, s_out, zp_out))


@pytest.mark.parametrize("L", [593, 608, 640, 641, 785, 1009, 1023, 1024])
@pytest.mark.parametrize("zp", [0, -77])
def test_long_rows(L, zp):
    x, v = _inputs(L, 3, L, 64)
    _check(x, L, 0.0421, v, zp)


@pytest.mark.parametrize("L", [65, 80, 100, 127, 128, 129, 144, 197, 257, 577, 900, 1024])
def test_head_dimension_32(L):
    x, v = _inputs(L, 5, L, 32, pad=16)
    _check(x, L, 0.0347, v, 13)


@pytest.mark.parametrize("s", [2.0 ** -7, 0.0173, 0.1, 0.5])
def test_scales(s):
    """The smallest and largest scale, one whose i-exp values rise at a band edge, and the 64-bit sums."""
    for peaked in (False, True):
        x, v = _inputs(7, 4, 700, 64, peaked=peaked)
        _check(x, 700, float(np.float32(s)), v, 5)


@pytest.mark.parametrize("window", [9, 10, 11, 12, 13, 16])
@pytest.mark.parametrize("d,zp", [(32, 0), (32, 31), (64, -9)])
def test_windows_with_bias(window, d, zp):
    L, heads, BH = window * window, 3, 9
    rng = np.random.default_rng(window)
    for brange, s in ((16, 0.0431), (128, 0.0101)):  # the bias's full range: distances past 255
        bias = rng.integers(-brange, brange, size=(heads, (2 * window - 1) ** 2)).astype(np.int8)
        x, v = _inputs(window * d, BH, L, d)
        _check(x, L, s, v, zp, bias=bias, heads=heads, window=window)


@pytest.mark.parametrize("window,side,heads,images,d", [(12, 48, 6, 2, 32), (12, 24, 4, 1, 64), (10, 20, 3, 3, 32),
                                                        (16, 32, 2, 2, 32), (7, 14, 3, 2, 64)])
def test_shifted_windows(window, side, heads, images, d):
    """Bias and shifted-window mask; (7, d = 64) with a zero point of V is beyond the short-row kernel."""
    L, nw = window * window, (side // window) ** 2
    rng = np.random.default_rng(side)
    bias = rng.integers(-40, 41, size=(heads, (2 * window - 1) ** 2)).astype(np.int8)
    region = synth.shifted_window_regions(side, window).numpy()
    for s, mask in ((0.0431, -2320), (0.21, -3), (0.0347, -700)):
        x, v = _inputs(side + window, images * nw * heads, L, d)
        _check(x, L, s, v, -3, bias=bias, heads=heads, window=window, region=region, mask=mask)


def test_one_head_and_partial_tiles():
    for BH, L in ((1, 785), (1, 1024), (2, 66), (1, 65)):
        x, v = _inputs(BH + L, BH, L, 32)
        _check(x, L, 0.05, v, 0)
