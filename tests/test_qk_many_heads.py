"""Q K^T logits where every CTA walks several heads: operand buffers, chunk-wise K and the staging buffers go
round more than once, on the bulk path (16-byte rows) and on the other, every head against the oracle."""
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


# d = 64, 32, 16: bulk copies from 128 keys on; d = 24, 40: 8-byte rows.  640 keys: all five chunks;
# 129: a second chunk of 16 keys; heads of one tile (128, 64) and of several
@pytest.mark.parametrize("BH,L,d", [(700, 128, 64), (460, 129, 32), (310, 257, 64), (170, 640, 16), (500, 64, 64),
                                    (400, 144, 24), (170, 577, 40)])
def test_heads_follow_one_another(BH, L, d):
    rng = np.random.default_rng(BH + L + d)
    q, k = (rng.integers(-128, 128, size=(BH, L, d), dtype=np.int16).astype(np.int8) for _ in range(2))
    args = (11, -7, 0.031, 0.027, 0.0441, 3)
    want = oracle.qk_logits(q, k, *args, ld=(L + 15) // 16 * 16)
    got = fqvit.qk_logits(torch.from_numpy(q).to(DEV), torch.from_numpy(k).to(DEV), *args)
    fqvit.sync_status()
    assert np.array_equal(got.cpu().numpy(), want)
