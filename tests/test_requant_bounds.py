"""The fp32 form of the 8-bit attention output at its bound on the accumulators: rows whose operands sum to nearly
1.5 2^15 (equal logits at the lengths just below a code's threshold), V at both ends, zero points of V up to the
largest that the calls take (beyond an int8 code's the 64-bit form), bit for bit against the oracle."""
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


# 3 2^k - 1 keys, on the short-row, the long-row (with and without the operand table) and the general kernel
@pytest.mark.parametrize("L,d", [(47, 32), (191, 64), (383, 64), (577, 64), (191, 32), (767, 64)])
@pytest.mark.parametrize("zp_v", [-255, -128, -5, 100, 127, 255])
def test_largest_accumulators(L, d, zp_v):
    rng = np.random.default_rng(1000 + L + zp_v)
    BH = 2
    x = np.zeros((BH * L, (L + 15) // 16 * 16), np.int8)
    x[1::2] = rng.integers(-128, 128, size=x[1::2].shape)
    v = rng.integers(-128, 128, size=(BH, L, d)).astype(np.int8)
    v[:, :, 0], v[:, :, 1] = -128, 127
    s = 0.0431
    codes, _ = oracle.lis_softmax(x, L, s)
    if L in (47, 191, 383, 767):
        assert (1 << (15 - codes[0].astype(int))).sum() > 1.46 * 2 ** 15
    acc, over = oracle.lis_attn_v(codes, v, zp_v)
    assert not over
    xd, vd = torch.from_numpy(x).to(DEV), torch.from_numpy(v).to(DEV)
    for r in (2.0 ** -12, 0.0037, 0.09, 2.0 / 9.0, 0.31, 0.4999, 0.5, 1.3):
        for zp_out in (0, 117, 255):
            s_v = float(np.float32(r))
            got = fqvit.lis_attention_q(xd, s, vd, zp_v, s_v, 1.0, zp_out)
            assert np.array_equal(got.cpu().numpy(), oracle.attn_requant(acc, s_v, 1.0, zp_out)), (r, zp_out)
    fqvit.sync_status()
