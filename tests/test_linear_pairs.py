"""Linear calls on pairs of CTAs right behind one another: with programmatic launches the next kernel's CTAs
take over an SM as soon as a pair has left it, so every barrier arrival of the pair has to have landed by
then.  Bit for bit against the oracle and against the first call (exact integers: no tolerance)."""
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


def _layer(seed, M, N, K):
    rng = np.random.default_rng(seed)
    x = rng.integers(0, 256, size=(M, K)).astype(np.uint8)
    w = rng.integers(-128, 128, size=(N, K)).astype(np.int8)
    s_w = (rng.uniform(0.5, 2, size=N) * 1e-3).astype(np.float32)
    bias = rng.integers(-20000, 20000, size=N).astype(np.int32)
    s_y = float(np.float32(0.02 * 1e-3 * np.sqrt(K) * 60 * 90 / 255))
    xd, sw, b = (torch.from_numpy(a).to(DEV) for a in (x, s_w, bias))
    wh = fqvit.linear_pack_weight(torch.from_numpy(w).to(DEV))
    out = torch.empty(M, N, dtype=torch.uint8, device=DEV)
    rows = sorted({0, 127, 128, 255, 256, M // 2, M - 1} & set(range(M)))
    want, _ = oracle.linear_q(x[rows], 131, 0.02, w, s_w, bias, s_y, 117)
    return (xd, 131, 0.02, wh, sw, b, s_y, 117), out, rows, want


# fewer K-steps than operand stages (4), than weight stages (8), and more than both
@pytest.mark.parametrize("K", [64, 200, 576])
def test_pairs_back_to_back(K):
    pair, single = _layer(K, 8200, 1536, K), _layer(K + 1, 300, 96, K)  # (pairs of CTAs; single CTAs)
    outs = [[torch.empty_like(out) for _ in range(12)] for _, out, _, _ in (pair, single)]
    for i in range(12):
        for (args, _, _, _), o in zip((pair, single), outs):
            fqvit.linear_q(*args, out=o[i])
    fqvit.sync_status()
    for (_, _, rows, want), o in zip((pair, single), outs):
        assert np.array_equal(o[0].cpu().numpy()[rows], want)
        for y in o[1:]:
            assert torch.equal(y, o[0])
