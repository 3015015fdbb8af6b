"""Logits, Q and K as views whose rows end where a larger buffer ends (column slices): the kernels' copies
stop with the last row's data.  Bit for bit against the oracle (exact integers: no tolerance)."""
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


def _right_aligned(x, front):
    """x's rows as the last columns of a buffer with `front` more columns ahead of them."""
    buf = torch.full((*x.shape[:-1], front + x.shape[-1]), 77, dtype=torch.int8, device=DEV)
    buf[..., front:] = torch.from_numpy(x).to(DEV)
    return buf[..., front:]


# one operand region, two, the operand table, the general kernel without and with the packing of tiles, and the
# short-row kernel; lengths with whole and part 16-byte units, one tile and several
@pytest.mark.parametrize("BH,L,d", [(3, 97, 64), (7, 197, 64), (300, 197, 64), (4, 577, 64), (3, 785, 64), (40, 1024, 64),
                                    (3, 80, 32), (9, 200, 32), (5, 49, 32)])
def test_logits(BH, L, d):
    rng = np.random.default_rng(L)
    x = rng.integers(-128, 128, size=(BH * L, (L + 15) // 16 * 16)).astype(np.int8)
    v = rng.integers(-128, 128, size=(BH, L, d)).astype(np.int8)
    codes, _ = oracle.lis_softmax(x, L, 0.0421)
    want, over = oracle.lis_attn_v(codes, v, -5)
    assert not over
    for front in (16, 48):
        got = fqvit.lis_attention(_right_aligned(x, front), 0.0421, torch.from_numpy(v).to(DEV), zp_v=-5)
        fqvit.sync_status()
        assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("BH,L,d", [(3, 128, 16), (2, 197, 32), (5, 300, 24), (3, 577, 48), (160, 130, 8)])
def test_q_and_k(BH, L, d):
    rng = np.random.default_rng(L + d)
    q, k = (rng.integers(-128, 128, size=(BH, L, d)).astype(np.int8) for _ in range(2))
    ld = (L + 15) // 16 * 16
    want = oracle.qk_logits(q, k, 3, -7, 0.03, 0.04, 0.05, 11, ld=ld)
    pad = np.zeros((BH, L, -d % 16), np.int8)  # rows in whole 16-byte units
    qv, kv = (_right_aligned(np.concatenate([a, pad], -1), 16)[..., :d] for a in (q, k))
    got = fqvit.qk_logits(qv, kv, 3, -7, 0.03, 0.04, 0.05, 11)
    fqvit.sync_status()
    assert np.array_equal(got.cpu().numpy().reshape(want.shape), want)
