"""The exponent-difference code against the oracle at every distance of a two-key row and in rows that one key
dominates (code 0 against 1, where 3 e = 2S), on the short-row and the general kernel, bit for bit."""
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


def _check(x, L, s, d, bias=None, heads=1, window=0):
    BH = x.shape[0] // L
    v = np.random.default_rng(L).integers(-128, 128, size=(BH, L, d)).astype(np.int8)
    kw = dict(bias=bias, heads=heads, window=window) if bias is not None else {}
    co, _ = oracle.lis_softmax(x, L, s, **kw)
    want, _ = oracle.lis_attn_v(co, v, 3)
    if bias is not None:
        kw["bias"] = torch.from_numpy(bias).to(DEV)
    got = fqvit.lis_attention(torch.from_numpy(x).to(DEV), s, torch.from_numpy(v).to(DEV), 3, **kw)
    fqvit.sync_status()
    assert np.array_equal(got.cpu().numpy(), want)


SCALES = [2.0 ** -7, 0.0101, 0.0173, 0.0431, 0.1, 0.23, 0.3, 0.5]


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("L", [2, 5, 50, 70, 144])
def test_every_distance(s, L):
    """Key i of row r: the maximum; another at distance r; the rest far below."""
    s = float(np.float32(s))
    BH = -(-256 // L)
    x = np.full((BH * L, (L + 15) // 16 * 16), -128, np.int8)
    r = np.arange(BH * L)
    x[r, r % L] = 127
    x[r, (r + 1) % L] = np.clip(127 - r, -128, 127)
    _check(x, L, s, 32)


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("window", [2, 7, 10])
def test_dominant_keys_with_bias(s, window):
    s = float(np.float32(s))
    L, BH = window * window, 12
    rng = np.random.default_rng(window)
    x = np.full((BH * L, (L + 15) // 16 * 16), -90, np.int8)
    r = np.arange(BH * L)
    x[r, r % L] = 100
    near = rng.integers(0, 60, size=BH * L)
    for k in range(1, 4):
        x[r, (r + k) % L] = 100 - near if L > 4 else 100 - 3 * near
    bias = rng.integers(-20, 21, size=(3, (2 * window - 1) ** 2)).astype(np.int8)
    _check(x, L, s, 32, bias=bias, heads=3, window=window)
