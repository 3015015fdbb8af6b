"""The general attention kernel with several tiles on every CTA: hand-over of the logits buffers (one and two),
of the operand and V rings and of the two accumulator pairs, the walk over many heads, and rows at strides of
their own, bit for bit against the oracle (exact integers: no tolerance)."""
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


def _check(seed, BH, L, d, s, zp, pad_v=0, pad_o=0, bias=None, heads=1, window=0, region=None, mask=0):
    rng = np.random.default_rng(seed)
    x = rng.integers(-128, 128, size=(BH * L, (L + 15) // 16 * 16)).astype(np.int8)
    v = rng.integers(-128, 128, size=(BH, L, d)).astype(np.int8)
    kw = dict(bias=bias, heads=heads, window=window) if bias is not None else {}
    mk = dict(region=region, mask_value=mask) if region is not None else {}
    codes, _ = oracle.lis_softmax(x, L, s, **kw, **mk)
    want, over = oracle.lis_attn_v(codes, v, zp)
    assert not over
    T = lambda a: None if a is None else torch.from_numpy(a).to(DEV)  # noqa: E731
    vd = torch.zeros(BH, L, d + pad_v, dtype=torch.int8, device=DEV)[..., :d]
    vd.copy_(T(v))
    gkw = dict(bias=T(bias), heads=heads, window=window) if bias is not None else {}
    acc = torch.empty(BH, L, d + pad_o, dtype=torch.int32, device=DEV)[..., :d]
    fqvit.lis_attention_masked(T(x), s, vd, T(region), mask, zp_v=zp, acc=acc, **gkw)
    out8 = torch.empty(BH, L, d + 2 * pad_o, dtype=torch.uint8, device=DEV)[..., :d]
    fqvit.lis_attention_masked_q(T(x), s, vd, T(region), mask, zp, 0.02, 0.031, 117, out=out8, **gkw)
    fqvit.sync_status()
    assert np.array_equal(acc.cpu().numpy(), want)
    assert np.array_equal(out8.cpu().numpy(), oracle.attn_requant(want, 0.02, 0.031, 117))


# 640 to 813 tiles of 128 rows on at most 152 CTAs; 1024 keys: one logits buffer; 80 keys: a head per tile, longer
# rows packed; 300 keys with d = 64 come here by the strides of V and the output
@pytest.mark.parametrize("BH,L,d,zp,pad_v,pad_o", [(105, 785, 64, 0, 0, 0), (81, 1024, 64, 19, 0, 0), (800, 80, 32, 0, 0, 0),
                                                   (800, 80, 32, -40, 16, 8), (520, 200, 32, 7, 0, 0),
                                                   (273, 300, 64, -9, 32, 8)])
def test_many_tiles(BH, L, d, zp, pad_v, pad_o):
    _check(BH + L, BH, L, d, 0.0421, zp, pad_v, pad_o)


@pytest.mark.parametrize("window,side,images,heads,zp,shift", [(12, 120, 2, 5, 0, True), (12, 120, 2, 5, 11, False),
                                                               (9, 72, 3, 4, -6, True), (16, 96, 3, 3, 0, True)])
def test_many_windows(window, side, images, heads, zp, shift):
    """324 to 1125 tiles, with and without a mask."""
    rng = np.random.default_rng(side)
    bias = rng.integers(-40, 41, size=(heads, (2 * window - 1) ** 2)).astype(np.int8)
    region = synth.shifted_window_regions(side, window).numpy() if shift else None
    BH = images * (side // window) ** 2 * heads
    _check(side + window, BH, window * window, 32, 0.0431, zp, bias=bias, heads=heads, window=window, region=region,
           mask=-2320 if shift else 0)
