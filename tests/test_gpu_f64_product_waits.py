"""The waits of the FP64 product on the tensor cores (csrc/sp2_f64_tc.cu) where a run ends during the launch.

A wait that gives up ends the run while other clusters are still starting, so that some CTAs of a cluster may find it
over and others not.  Every CTA stays until its cluster is done: the testing entry lets some CTAs of every cluster
find the run over at their start, and lets waits run out, without a fault.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

SPLITS = [2, 4, 8]


def product(X, ks, hook, wait_ms=0):
    from paper_1507_02087_gb300 import sp2
    out = torch.full_like(X, float("nan"))
    status = sp2.lib().sp2_test_f64_product(X.data_ptr(), X.shape[0], 64, ks, hook, wait_ms, out.data_ptr(), None,
                                            torch.cuda.current_stream().cuda_stream)
    return out, status


@pytest.fixture(scope="module")
def X():
    g = torch.Generator().manual_seed(11)
    return torch.randn(300, 300, generator=g, dtype=torch.float64).cuda()


@pytest.mark.parametrize("ks", SPLITS)
@pytest.mark.parametrize("hook", [2, 3])         # all but the first CTA of a cluster, or only the first
def test_ctas_that_find_the_run_over_stay_in_their_cluster(X, ks, hook):
    want, status = product(X, ks, 0)
    assert status == 0 and torch.allclose(want, X @ X.T, rtol=0, atol=1e-10)
    _, status = product(X, ks, hook, wait_ms=50)
    assert status == 4                           # SP2_ERR_TIMEOUT: the others wait for their sums in vain
    again, status = product(X, ks, 0)            # the context stays usable
    assert status == 0 and torch.equal(again, want)


@pytest.mark.parametrize("ks", [1] + SPLITS)
def test_waits_that_run_out_end_the_launch(X, ks):
    want, _ = product(X, ks, 0)
    got, status = product(X, ks, 1, wait_ms=50)
    assert status == 4                           # SP2_ERR_TIMEOUT
    assert torch.equal(got[256:, 256:], want[256:, 256:])    # a tile of another cluster
    again, status = product(X, ks, 0)            # the context stays usable
    assert status == 0 and torch.equal(again, want)


def test_arguments_are_checked(X):
    from paper_1507_02087_gb300 import sp2
    L = sp2.lib()
    for N, bn, ks, hook, wait in [(0, 64, 1, 0, 0), (8193, 64, 1, 0, 0), (300, 32, 2, 0, 0), (300, 64, 3, 0, 0),
                                  (300, 128, 1, 0, 0), (300, 64, 1, 4, 0), (300, 64, 1, 1, 2001)]:
        assert L.sp2_test_f64_product(X.data_ptr(), N, bn, ks, hook, wait, X.data_ptr(), None, None) == 1
