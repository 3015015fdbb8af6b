"""Rows of 65 .. 592 keys, d = 64, on both sides of the length where operands stop coming from the i-exp values
and come from a table per row: any scale, dominant keys, and many tiles per CTA, bit for bit."""
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


def _check(x, BH, L, s, zp):
    v = np.random.default_rng(L).integers(-128, 128, size=(BH, L, 64)).astype(np.int8)
    co, _ = oracle.lis_softmax(x, L, s)
    want, over = oracle.lis_attn_v(co, v, zp)
    assert not over
    got = fqvit.lis_attention(torch.from_numpy(x).to(DEV), s, torch.from_numpy(v).to(DEV), zp)
    fqvit.sync_status()
    assert np.array_equal(got.cpu().numpy(), want)


# the first two scales have i-exp values that rise at band edges (floored constants)
@pytest.mark.parametrize("s", [0.008350185749701165, 0.01732846078509329, 2.0 ** -7, 0.0431, 0.3, 0.5])
@pytest.mark.parametrize("L", [65, 128, 191, 384, 385, 577])
def test_codes_at_any_scale(L, s):
    BH, s = 4, float(np.float32(s))
    rng = np.random.default_rng(L)
    x = rng.integers(-128, 128, (BH * L, (L + 15) // 16 * 16), dtype=np.int8)
    x[::3] = rng.integers(60, 90, x[::3].shape, dtype=np.int8)        # narrow rows
    x[1::7] = rng.integers(-128, -100, x[1::7].shape, dtype=np.int8)  # rows far below 0
    r = np.arange(2, BH * L, 5)                                       # a maximum, one key at each distance, the rest far
    x[r] = -128
    x[r, r % L] = 127
    x[r, (r + 1) % L] = np.clip(127 - r % 256, -128, 127)
    _check(x, BH, L, s, 0)


@pytest.mark.parametrize("L,BH", [(65, 700), (127, 400), (129, 600), (320, 150), (384, 120), (400, 120)])
def test_many_tiles(L, BH):
    x = np.random.default_rng(BH).integers(-128, 128, (BH * L, (L + 15) // 16 * 16), dtype=np.int8)
    _check(x, BH, L, float(np.float32(0.0431)), -9)
