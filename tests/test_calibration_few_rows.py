"""Calibration of few rows (a thread per error sum) on both sides of the rule that chooses it, at the edges of
its row groups, channel blocks and factor groups, bit for bit against the oracle."""
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


# threads below 36 + C (K + 1) / 64 rows: 36, 38, 48, 164 and 292
@pytest.mark.parametrize("C,K,rows", [(1, 0, (1, 2, 35, 36)), (33, 3, (3, 4, 5, 37, 38)), (192, 3, (7, 47, 48)),
                                      (1025, 7, (6, 163, 164, 165)), (4096, 3, (32, 291, 292))])
def test_few_rows(C, K, rows):
    rng = np.random.default_rng(C + K)
    for n in rows:
        x = (rng.normal(size=(n, C)) * np.exp(rng.normal(size=C))).astype(np.float32)
        s_o, zp_o, a_o, sse_o = oracle.calibrate_ptf(x, K=K)
        buf = torch.zeros(n, C + 3, device=DEV)  # rows at a stride of their own
        buf[:, :C] = torch.from_numpy(x).to(DEV)
        for xd in (torch.from_numpy(x).to(DEV), buf[:, :C]):
            sse = torch.empty(C, K + 1, dtype=torch.float64, device=DEV)
            s, zp, alpha = fqvit.calibrate_ptf(xd, K=K, sse=sse)
            assert np.float32(s_o) == np.float32(s.item()) and zp_o == int(zp.item())
            assert np.array_equal(sse_o.view(np.uint64), sse.cpu().numpy().view(np.uint64))
            assert np.array_equal(a_o, alpha.cpu().numpy())
            part = fqvit.calibrate_sse_partial(xd, K, torch.tensor([float(x.min()), float(x.max())], device=DEV))
            assert torch.equal(part, sse)
