"""Infinities, NaN and the largest finite values in a calibration batch: the error sums are those of the
sequential fp64 additions (an infinite sum and a NaN term give NaN, a huge sum and an infinite term
infinity), and the factors those that comparisons with them choose."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_13824_gb300 import build as fbuild
from paper_2111_13824_gb300 import fqvit

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
INF, NAN = np.float32(np.inf), np.float32(np.nan)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fbuild.build()
    fqvit.load()
    oracle.build()


def _same(got, want):
    """The same bits, any NaN for a NaN."""
    assert np.array_equal(np.isnan(got), np.isnan(want))
    keep = ~np.isnan(want)
    assert np.array_equal(got[keep].view(np.uint64), want[keep].view(np.uint64))


def _batch(rows):
    rng = np.random.default_rng(rows)
    x = rng.normal(size=(rows, 14)).astype(np.float32)
    a, b = rows // 5, rows - 2
    x[a, 0], x[b, 0] = INF, NAN       # an infinite sum, then NaN
    x[a, 1], x[b, 1] = NAN, INF
    x[b, 2] = -INF
    x[a, 3], x[a + 1, 3] = INF, -INF
    x[0, 4] = INF
    x[0, 5] = NAN
    x[0, 6], x[1, 6] = -INF, NAN
    x[:, 7:10] = rng.choice([-3e38, 3e38], size=(rows, 3)).astype(np.float32)  # sums above 2^253
    x[b, 8], x[b, 9] = INF, NAN
    x[:b, 10], x[b, 10] = 0.0, INF    # the first term of the sum
    x[:b, 11], x[b, 11] = 0.0, NAN
    x[a, 12] = -NAN                   # (a NaN with its sign bit set)
    return x


@pytest.mark.parametrize("rows", [5, 40, 300, 1500])
@pytest.mark.parametrize("K", [0, 3, 6])
def test_sums_of_a_shard(rows, K):
    """The range comes from the caller, so the batch may hold anything."""
    x = _batch(rows)
    mnmx = torch.tensor([-3.0, 3.0], device=DEV)
    with np.errstate(all="ignore"):
        want = oracle.calibrate_sse(x, K, -3.0, 3.0)
    got = fqvit.calibrate_sse_partial(torch.from_numpy(x).to(DEV), K, mnmx).cpu().numpy()
    assert np.isnan(want[0]).all() and np.isinf(want[2]).all() and np.isinf(want[8]).all()
    _same(got, want)


@pytest.mark.parametrize("rows", [40, 1500])
@pytest.mark.parametrize("K", [3, 6])
def test_calibration_with_nan(rows, K):
    """NaN has no part in the range; its channels' sums are NaN and their factor 0."""
    x = np.where(np.isinf(_batch(rows)) | (np.abs(_batch(rows)) > 1e38), NAN, _batch(rows))
    x[0, 0] = 1.0  # (the oracle's range starts from this element)
    s_o, zp_o, a_o, sse_o = oracle.calibrate_ptf(x, K=K)
    sse = torch.empty(x.shape[1], K + 1, dtype=torch.float64, device=DEV)
    s, zp, alpha = fqvit.calibrate_ptf(torch.from_numpy(x).to(DEV), K=K, sse=sse)
    assert np.float32(s_o) == np.float32(s.item()) and zp_o == int(zp.item())
    _same(sse.cpu().numpy(), sse_o)
    assert np.array_equal(a_o, alpha.cpu().numpy())
