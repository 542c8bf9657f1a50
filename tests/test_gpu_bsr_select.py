"""The error-controlled selection where it changes from one CTA to a grid (1024 pairs: between 44 and 45 block rows),
and for the smallest lattices: decisions equal to the oracle's, budgets that cut inside a tie group among them."""
import numpy as np
import pytest

from oracle import bsr_oracle as bo
from test_gpu_bsr import _keep_gpu, _spread_blocks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [1, 2, 22, 23, 44, 45])
def test_decisions_at_the_line(nb):
    from paper_1507_02087_gb300 import sp2
    X32, proto = _spread_blocks(nb, nb)
    tie = float(np.linalg.norm((proto * 1e-5).astype(np.float32).astype(np.float64)) ** 2)
    for tau in (0.0, 1e-160, 1e-7, 1e-4, 3e-3, np.sqrt(7.5 * tie), 1e3):
        keep = _keep_gpu(sp2, X32, tau, 1)
        assert np.array_equal(keep, bo.keep_mask_error(X32.astype(np.float64), 32, tau)), tau
