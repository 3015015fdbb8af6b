"""Short rows that the short-row kernel does not take (V at a stride of its own, or d = 64 with a zero point and a
bias): one key to a whole 64-key block of the general kernel, which begins at 25 keys, with and without a bias and
a mask, bit for bit against the oracle (exact integers: no tolerance)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_13824_gb300 import build as fbuild
from paper_2111_13824_gb300 import fqvit

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fbuild.build()
    fqvit.load()
    oracle.build()


def _check(seed, BH, L, d, zp, pad_v, bias=None, heads=1, window=0, region=None, mask=0):
    rng = np.random.default_rng(seed)
    kw = dict(bias=bias, heads=heads, window=window) if bias is not None else {}
    mk = dict(region=region, mask_value=mask) if region is not None else {}
    T = lambda a: None if a is None else torch.from_numpy(a).to(DEV)  # noqa: E731
    for low in (-128, 127):  # all codes; one value throughout (every distance 0)
        x = rng.integers(low, 128, size=(BH * L, (L + 15) // 16 * 16)).astype(np.int8)
        v = rng.integers(-128, 128, size=(BH, L, d)).astype(np.int8)
        codes, _ = oracle.lis_softmax(x, L, 0.0421, **kw, **mk)
        want, over = oracle.lis_attn_v(codes, v, zp)
        assert not over
        vd = torch.zeros(BH, L, d + pad_v, dtype=torch.int8, device=DEV)[..., :d]
        vd.copy_(T(v))
        gkw = dict(bias=T(bias), heads=heads, window=window) if bias is not None else {}
        got = fqvit.lis_attention_masked(T(x), 0.0421, vd, T(region), mask, zp_v=zp, **gkw)
        got8 = fqvit.lis_attention_masked_q(T(x), 0.0421, vd, T(region), mask, zp, 0.02, 0.031, 117, **gkw)
        fqvit.sync_status()
        assert np.array_equal(got.cpu().numpy(), want)
        assert np.array_equal(got8.cpu().numpy(), oracle.attn_requant(want, 0.02, 0.031, 117))


@pytest.mark.parametrize("L", [1, 2, 4, 16, 17, 24, 25, 26, 31, 32, 33, 48, 49, 63, 64])
@pytest.mark.parametrize("BH", [1, 400])
def test_rows(L, BH):
    _check(L + BH, BH, L, 64, 21, 16)


@pytest.mark.parametrize("window", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("masked", [False, True])
def test_windows(window, masked):
    L, heads, nw, images = window * window, 3, 4, 40
    rng = np.random.default_rng(window)
    bias = rng.integers(-128, 128, size=(heads, (2 * window - 1) ** 2)).astype(np.int8)
    region = rng.integers(0, 3, size=(nw, L)).astype(np.uint8) if masked else None
    if masked:
        region[1] = 2  # a window of one region
    _check(window, heads * nw * images, L, 64, -33, 0, bias=bias, heads=heads, window=window, region=region,
           mask=-2320 if masked else 0)
