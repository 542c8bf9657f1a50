"""The spectral-norm estimate in one launch (lz_cluster_kernel in csrc/sp2_lanczos.cu) at the sizes where its split
of the entries over 16 CTAs, their warps and the rows kept in shared memory changes, and beside its largest size,
against the exact spectrum of X_0.

32 Lanczos steps from a fixed start vector approach max |x - x^2| from below; here the spectrum is dense near its
top, and the bound that the other tests of the estimate use is 1e-2.  The matrix and the products are rounded to
FP32, about 1e-7 of the norm each.
"""
import numpy as np
import pytest
import torch

from paper_1507_02087_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp16x3"])
@pytest.mark.parametrize("N", [2, 15, 16, 17, 33, 511, 512, 513, 865, 1009, 1279, 1280, 1281])
def test_estimate_of_the_scaled_matrix(N, precision):
    from paper_1507_02087_gb300 import sp2
    case = inputs.dense_gapped(N, max(1, N // 2), gap=0.1, seed=N)
    lo, hi = -1.25, 1.75
    with sp2.Purifier(N, max(1, N // 2), precision, norm="spectral", max_iter=4, guard=False) as P:
        P.set_bounds((lo, hi))
        P.run(case.F.cuda())
        info = P.info()
    x = (hi - np.asarray(case.lam)) / (hi - lo)
    for k in range(3):
        e = float(np.max(np.abs(x - x * x)))
        assert (1 - 1e-2) * e <= info["v"][k] <= (1 + 1e-5) * e, (k, info["v"][k], e)
        x = x * x if info["p"][k + 1] else 2 * x - x * x
