"""The MinMax Linear kernel's tile shapes, rings and requantization forms at the sizes where they can go
wrong, bit for bit against the oracle (exact integers: no tolerance)."""
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


def _check(x, zp_x, s_x, w, s_w, bias, s_y, zp_y, rows=None, pad=0, with_acc=True):
    """The layer on the GPU (x at row stride K + pad) against the oracle on all rows or some."""
    M, K = x.shape
    N = w.shape[0]
    xp = torch.zeros(M, K + pad, dtype=torch.uint8, device=DEV)
    xp[:, :K] = torch.from_numpy(x).to(DEV)
    wh = fqvit.linear_pack_weight(torch.from_numpy(w).to(DEV))
    sw = torch.from_numpy(s_w).to(DEV)
    b = None if bias is None else torch.from_numpy(bias).to(DEV)
    acc = torch.empty(M, N, dtype=torch.int32, device=DEV) if with_acc else None
    y = fqvit.linear_q(xp[:, :K], zp_x, s_x, wh, sw, b, s_y, zp_y, acc=acc)
    fqvit.sync_status()
    r = slice(None) if rows is None else rows
    want_y, want_acc = oracle.linear_q(x[r], zp_x, s_x, w, s_w, bias, s_y, zp_y)
    assert np.array_equal(y.cpu().numpy()[r], want_y)
    if with_acc:
        assert np.array_equal(acc.cpu().numpy()[r], want_acc)


def _case(seed, M, K, N, zp_x):
    rng = np.random.default_rng(seed)
    x = rng.integers(0, 256, size=(M, K)).astype(np.uint8)
    w = rng.integers(-128, 128, size=(N, K)).astype(np.int8)
    s_w = (rng.uniform(0.5, 2, size=N) * 1e-3).astype(np.float32)
    bias = rng.integers(-20000, 20000, size=N).astype(np.int32)
    s_y = float(np.float32(0.02 * 1e-3 * np.sqrt(K) * 60 * 90 / 255))
    return x, zp_x, 0.02, w, s_w, bias, s_y, 117


# single CTAs (few tiles), pairs (many), ragged in M, N and K, one K-step up to several chunks
@pytest.mark.parametrize("M,N,K,zp_x", [(1, 16, 8, 7), (127, 64, 64, 128), (129, 80, 136, 0), (300, 208, 72, 255),
                                        (257, 3360, 200, 100), (1576, 768, 520, 128), (130, 64, 3072, 114)])
def test_tiles(M, N, K, zp_x):
    _check(*_case(M + N + K, M, K, N, zp_x))
    _check(*_case(M + N + K + 1, M, K, N, zp_x), with_acc=False)


@pytest.mark.parametrize("M,N,K,zp_x", [(8200, 1536, 72, 128), (19000, 400, 1032, 140), (9000, 1040, 2056, 8)])
def test_pair_tiles(M, N, K, zp_x):
    """Many tiles: pairs of CTAs.  Rows at the tiles' edges, the ragged end, and a spread between."""
    rows = sorted({0, 127, 128, 255, 256, 511, M // 2, M - 257, M - 256, M - 2, M - 1} | set(range(5, M, M // 20)))
    for with_acc in (False, True):
        _check(*_case(M + K, M, K, N, zp_x), rows=rows, with_acc=with_acc)


@pytest.mark.parametrize("pad", [8, 16, 24])
@pytest.mark.parametrize("M,N,K", [(300, 96, 200), (8200, 1040, 136)])
def test_row_strides(pad, M, N, K):
    """Rows at strides that are and are not multiples of 16 bytes (TMA and direct loads of X)."""
    _check(*_case(pad, M, K, N, 131), rows=list(range(0, M, max(1, M // 60))) + [M - 1], pad=pad)


@pytest.mark.parametrize("zp_x", [0, 128, 255])
@pytest.mark.parametrize("M,N", [(128, 64), (8200, 1536)])
def test_sums_at_two_to_the_24(zp_x, M, N):
    """A chunk's sums right up to 2^24 in magnitude (every large product of one sign), then unit products:
    a bit lost anywhere in the fp32 accumulation shows in the integer."""
    K = 1024 if zp_x == 128 else 512
    rng = np.random.default_rng(zp_x)
    big = 255 if zp_x == 0 else 0                     # x - zp_x = 255, -128 or -255
    x = np.full((M, K), big, np.uint8)
    unit = rng.random((M, K)) < 0.02
    x[unit] = zp_x + 1 if zp_x < 255 else zp_x - 1    # x - zp_x = +-1
    w = np.where(np.arange(N)[:, None] % 2 == 0, 127, -128).astype(np.int8) * np.ones((1, K), np.int8)
    ones = rng.random((N, K)) < 0.01
    w[ones] = 1
    rows = None if M < 1000 else list(range(0, M, 300)) + [M - 1]
    _check(x, zp_x, 0.01, w, np.full(N, 1e-3, np.float32), None, 50.0, 128, rows=rows)


@pytest.mark.parametrize("K", [64, 2048])
def test_requantization_forms(K):
    """Channels inside and outside the fp32 form: shifts 22 and 23, N1 <= 0, biases at 2^24 and beyond."""
    rng = np.random.default_rng(K)
    M, N = 200, 64
    x = rng.integers(0, 256, size=(M, K)).astype(np.uint8)
    w = rng.integers(-128, 128, size=(N, K)).astype(np.int8)
    for Ms, bias in (([2.0 ** -15, 1.99 * 2.0 ** -15], None), ([2.0 ** -16], None), ([1.5, 3e2, 4e3], None),
                     ([2.0 ** -12], [1 << 24, -(1 << 24)]), ([2.0 ** -12], [(1 << 24) + 1, -(1 << 30)]),
                     ([2.0 ** -31, 2.0 ** -33], [1 << 30])):
        s_w = np.resize(np.array(Ms, np.float32) * np.float32(4.0), N)
        b = None if bias is None else np.resize(np.array(bias, np.int32), N)
        _check(x, 120, 0.5, w, s_w, b, 2.0, 100)
        _check(x, 120, 0.5, w, s_w, b, 2.0, 100, with_acc=False)


def test_layer_run_in_place():
    """N == K: the output written over the activations."""
    x, zp_x, s_x, w, s_w, b, s_y, zp_y = _case(3, 3000, 384, 384, 128)
    xd = torch.from_numpy(x).to(DEV)
    wh = fqvit.linear_pack_weight(torch.from_numpy(w).to(DEV))
    args = (zp_x, s_x, wh, torch.from_numpy(s_w).to(DEV), torch.from_numpy(b).to(DEV), s_y, zp_y)
    want = fqvit.linear_q(xd, *args)
    got = fqvit.linear_q(xd, *args, out=xd)
    fqvit.sync_status()
    assert torch.equal(got, want)
