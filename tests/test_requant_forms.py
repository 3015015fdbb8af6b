"""The fp32 form of the 8-bit attention output against the oracle, bit for bit: multipliers at the edge of
its condition (c 2^24 = 256 with a zero point of V), accumulators at their largest, on each tensor-core kernel."""
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


# M = (s_v / s_out) 2^-15 = n2 2^-n1: below, at and above 2^-16; small, large and odd ones
RATIOS = [0.4999, 0.5, 0.502, 0.75, 1.0, 1.9999, 0.01, 2.0 ** -16, 37.3, 2.0 ** 15, 2.0 ** 18]


@pytest.mark.parametrize("L,d", [(49, 32), (197, 64), (577, 64), (785, 64), (300, 32)])
@pytest.mark.parametrize("zp_v", [0, -128, 127])
def test_requant_at_extremes(L, d, zp_v):
    rng = np.random.default_rng(1000 + L + zp_v)
    BH = 3
    x = rng.integers(-128, 128, size=(BH * L, (L + 15) // 16 * 16)).astype(np.int8)
    x[::3] = np.where(rng.random(x[::3].shape) < 0.02, 100, -100)      # a few equal maxima
    x[1::3] = 0                                                        # uniform rows
    v = rng.integers(-128, 128, size=(BH, L, d)).astype(np.int8)
    v[:, :, 0], v[:, :, 1], v[:, :, 2] = -128, 127, zp_v
    s = 0.0431
    co, _ = oracle.lis_softmax(x, L, s)
    acc, over = oracle.lis_attn_v(co, v, zp_v)
    assert not over
    xd, vd = torch.from_numpy(x).to(DEV), torch.from_numpy(v).to(DEV)
    for r in RATIOS:
        for zp_out in (0, 131, 255):
            s_v = float(np.float32(r))
            got = fqvit.lis_attention_q(xd, s, vd, zp_v, s_v, 1.0, zp_out)
            assert np.array_equal(got.cpu().numpy(), oracle.attn_requant(acc, s_v, 1.0, zp_out)), (r, zp_out)
    fqvit.sync_status()
