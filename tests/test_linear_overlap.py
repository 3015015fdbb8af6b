"""Linear layers whose outputs overlap their activations: y shifted, y at a stride of its own, y in the columns
behind x, and the accumulators, at row strides that do and do not suit tensor loads, on single CTAs and on pairs,
against the oracle on the original activations (exact integers: no tolerance)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_13824_gb300 import build as fbuild
from paper_2111_13824_gb300 import fqvit

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
SIZES = [(300, 96, 208), (300, 96, 200), (8200, 1040, 136), (8200, 1040, 144)]  # M, N, K


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fbuild.build()
    fqvit.load()
    oracle.build()


def _layer(M, N, K):
    rng = np.random.default_rng(M + N + K)
    x = rng.integers(0, 256, size=(M, K)).astype(np.uint8)
    w = rng.integers(-128, 128, size=(N, K)).astype(np.int8)
    s_w = (rng.uniform(0.5, 2, size=N) * 1e-3).astype(np.float32)
    bias = rng.integers(-20000, 20000, size=N).astype(np.int32)
    s_y = float(np.float32(0.02 * 1e-3 * np.sqrt(K) * 60 * 90 / 255))
    rows = np.unique(np.r_[0:M:max(1, M // 50), M - 1])
    want_y, want_acc = oracle.linear_q(x[rows], 131, 0.02, w, s_w, bias, s_y, 117)
    args = (131, 0.02, fqvit.linear_pack_weight(torch.from_numpy(w).to(DEV)), torch.from_numpy(s_w).to(DEV),
            torch.from_numpy(bias).to(DEV), s_y, 117)
    return x, args, rows, want_y, want_acc


def _place(buf, rows, cols, ld, at):
    return buf.as_strided((rows, cols), (ld, 1), at)


@pytest.mark.parametrize("M,N,K", SIZES)
@pytest.mark.parametrize("pad", [0, 16, 24])
def test_output_over_the_activations(M, N, K, pad):
    """x at 4096 with row stride K + pad; y from 16 bytes before it to far behind its start."""
    x, args, rows, want_y, _ = _layer(M, N, K)
    ld_x = K + pad
    for at, ld_y in ((4096, N), (4096 - 16, N + 32), (4096 + 48, N), (4096 + (M // 2) * ld_x // 16 * 16, N)):
        buf = torch.zeros(4096 + max(M * ld_x, 4096 + (M // 2) * ld_x + M * (N + 32)), dtype=torch.uint8, device=DEV)
        xv = _place(buf, M, K, ld_x, 4096)
        xv.copy_(torch.from_numpy(x).to(DEV))
        y = fqvit.linear_q(xv, *args, out=_place(buf, M, N, ld_y, at))
        fqvit.sync_status()
        assert np.array_equal(y.cpu().numpy()[rows], want_y), (at, ld_y)


@pytest.mark.parametrize("M,N,K", SIZES)
def test_output_in_the_columns_behind(M, N, K):
    x, args, rows, want_y, _ = _layer(M, N, K)
    k16 = (K + 15) // 16 * 16
    buf = torch.zeros(M, k16 + N, dtype=torch.uint8, device=DEV)
    buf[:, :K] = torch.from_numpy(x).to(DEV)
    y = fqvit.linear_q(buf[:, :K], *args, out=buf[:, k16:])
    fqvit.sync_status()
    assert np.array_equal(y.cpu().numpy()[rows], want_y)
    assert np.array_equal(buf[:, :K].cpu().numpy(), x)


@pytest.mark.parametrize("M,N,K", SIZES)
def test_accumulators_over_the_activations(M, N, K):
    x, args, rows, want_y, want_acc = _layer(M, N, K)
    buf = torch.zeros(4096 + 4 * M * (N + 4) + M * K, dtype=torch.uint8, device=DEV)
    for at, ld in ((4096, N), (4096 - 16, N + 4), (4096 + 32, N)):
        xv = _place(buf, M, K, K, 4096)
        xv.copy_(torch.from_numpy(x).to(DEV))
        acc = buf.view(torch.int32).as_strided((M, N), (ld, 1), at // 4)
        y = fqvit.linear_q(xv, *args, acc=acc)
        fqvit.sync_status()
        assert np.array_equal(y.cpu().numpy()[rows], want_y), (at, ld)
        assert np.array_equal(acc.cpu().numpy()[rows], want_acc), (at, ld)
