"""Logits rows at strides far past their keys: every byte behind the keys is written as zero, bit for bit against
the oracle, over outputs that held something else."""
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


# strides within the keys' 128-byte boxes, to their end, one unit and many boxes past them
@pytest.mark.parametrize("BH,L,d,strides", [(3, 128, 64, (128, 144, 256)), (6, 251, 32, (256, 272, 512)),
                                            (170, 130, 16, (144, 240, 256, 272)), (2, 577, 64, (592, 640, 656, 1024)),
                                            (4, 100, 64, (112, 128, 144, 400))])
def test_padding_is_zero(BH, L, d, strides):
    rng = np.random.default_rng(L)
    q, k = (rng.integers(-128, 128, size=(BH, L, d)).astype(np.int8) for _ in range(2))
    qd, kd = torch.from_numpy(q).to(DEV), torch.from_numpy(k).to(DEV)
    for ld in strides:
        out = torch.full((BH * L, ld), 85, dtype=torch.int8, device=DEV)
        fqvit.qk_logits(qd, kd, 5, -9, 0.03, 0.04, 0.05, 7, out=out)
        fqvit.sync_status()
        assert np.array_equal(out.cpu().numpy(), oracle.qk_logits(q, k, 5, -9, 0.03, 0.04, 0.05, 7, ld=ld)), ld
