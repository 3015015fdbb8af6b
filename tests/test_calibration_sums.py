"""The warp-parallel fp64 sums of the PTF calibration against the oracle's sequential ones, bit for bit,
where their rounding is hardest: ties at every step, sums that leave their binade at every step, zero and
denormal terms, and the edges of the row stages, channel blocks and factor groups."""
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


def _check(x, K):
    s_o, zp_o, a_o, sse_o = oracle.calibrate_ptf(x, K=K)
    xd = torch.from_numpy(x).to(DEV)
    sse = torch.empty(x.shape[1], K + 1, dtype=torch.float64, device=DEV)
    s, zp, alpha = fqvit.calibrate_ptf(xd, K=K, sse=sse)
    torch.cuda.synchronize()
    assert np.float32(s_o) == np.float32(s.item()) and zp_o == int(zp.item())
    assert np.array_equal(sse_o.view(np.uint64), sse.cpu().numpy().view(np.uint64))
    assert np.array_equal(a_o, alpha.cpu().numpy())
    q = fqvit.ptf_quantize(xd, float(s.item()), int(zp.item()), alpha)
    assert np.array_equal(oracle.ptf_quantize(x, s_o, zp_o, a_o), q.cpu().numpy())


@pytest.mark.parametrize("K", range(8))
@pytest.mark.parametrize("rows,C", [(1, 1), (31, 3), (129, 17), (1000, 40), (257, 1220)])
def test_shapes(rows, C, K):
    rng = np.random.default_rng(rows + C + K)
    _check((rng.normal(size=(rows, C)) * np.exp(rng.normal(size=C))).astype(np.float32), K)


@pytest.mark.parametrize("kind", ["coarse", "growing", "shrinking", "zeros", "tiny", "mixed"])
def test_hard_sums(kind):
    """coarse: few mantissa bits in the errors, so that almost every addition ties; growing / shrinking:
    errors that double (halve) every few rows; zeros: runs of exact zeros; tiny: errors down to fp32
    denormals; mixed: magnitudes over 40 octaves."""
    rng = np.random.default_rng(len(kind))
    rows, C = 1500, 24
    if kind == "coarse":  # multiples of 2^-12: with s0 = 1 the errors are multiples of 2^-12 as well
        x = (rng.integers(-2 ** 11, 2 ** 11, size=(rows, C)) * 2.0 ** -12 + rng.integers(-90, 90, size=(rows, C)))
        x[0, 0], x[0, 1] = -127.0, 128.0
    elif kind in ("growing", "shrinking"):
        e = np.arange(rows) / 40.0
        x = rng.choice([-1.0, 1.0], size=(rows, C)) * 2.0 ** (e if kind == "growing" else -e)[:, None]
        x *= rng.uniform(1, 2, size=(rows, C))
    elif kind == "zeros":
        x = np.where(rng.random((rows, C)) < 0.9, 0.0, rng.normal(size=(rows, C)))
        x[:, 3] = 0.0
        x[:700, 4] = 0.0
    elif kind == "tiny":
        x = rng.normal(size=(rows, C)) * 2.0 ** rng.uniform(-149, -100, size=(rows, C))
    else:
        x = rng.normal(size=(rows, C)) * 2.0 ** rng.uniform(-30, 10, size=(rows, C))
    for K in (0, 3, 6):
        _check(x.astype(np.float32), K)


def test_odd_strides():
    """Rows that are not multiples of 16 bytes, and an output stride that is not a multiple of 4."""
    rng = np.random.default_rng(1)
    x = rng.normal(size=(300, 50)).astype(np.float32)
    big = torch.zeros(300, 53, device=DEV)
    big[:, :50] = torch.from_numpy(x).to(DEV)
    s_o, zp_o, a_o, _ = oracle.calibrate_ptf(x, K=3)
    s, zp, alpha = fqvit.calibrate_ptf(big[:, :50], K=3)
    assert np.array_equal(a_o, alpha.cpu().numpy()) and np.float32(s_o) == np.float32(s.item())
    out = torch.zeros(300, 51, dtype=torch.uint8, device=DEV)
    fqvit.ptf_quantize(big[:, :50], float(s.item()), int(zp.item()), alpha, out=out[:, :50])
    assert np.array_equal(oracle.ptf_quantize(x, s_o, zp_o, a_o), out[:, :50].cpu().numpy())
