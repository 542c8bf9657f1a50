"""FP64 products on the tensor cores (csrc/sp2_f64_tc.cu): sizes at the edges of the tiles and of the
blocks of k-columns, and matrices whose rows differ in scale, against products in extended precision.

A run capped at one or two steps returns the polynomial of X_0 itself.  Bound on an element of
S = X X^T, with 2^e_i the scale of row i (2^e_i <= 4 max|x_i| or <= 2 ||x_i||, so 2^e_i <= 4 ||x_i||): digits
rounded at 2^-57 2^e_i per value, products left out below 2^-64 sqrt(K), and one rounding to FP64.
That is at most 8 eps ||x_i|| ||x_j|| sqrt(K) with room to spare (eps = 2^-53).
"""
import numpy as np
import pytest
import torch

from paper_1507_02087_gb300 import inputs

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def one_square(F, bounds, nocc):
    """X_0 as the library forms it, and X_1 of a run that ends at the cap after one step."""
    from paper_1507_02087_gb300 import sp2
    N = F.shape[0]
    with sp2.Purifier(N, nocc, "fp64", max_iter=1, guard=False) as P:
        P.set_bounds(bounds)
        X1 = P.run(torch.from_numpy(F).cuda()).cpu().numpy()
        info = P.info()
    assert info["status"] == 0 and info["n_iter"] == 1
    lo, hi = bounds
    X0 = (hi * np.eye(N) - F) / (hi - lo)
    return X0, X1, int(info["p"][1])


def check(X0, X1, p):
    N = X0.shape[0]
    L = X0.astype(np.longdouble)
    S = L @ L
    ref = S if p else 2 * L - S
    norms = np.linalg.norm(X0, axis=1)
    bound = 8 * EPS * np.sqrt(N) * np.outer(norms, norms) + 2 * EPS * np.abs(ref).astype(float)
    err = np.abs((X1.astype(np.longdouble) - ref).astype(float))
    assert np.all(err <= bound), float(np.max(err / np.maximum(bound, 1e-300)))
    assert np.array_equal(X1, X1.T)


@pytest.mark.parametrize("N", [129, 160, 191, 192, 193, 256, 321, 448, 513])
@pytest.mark.parametrize("fill", [0.2, 0.8])
def test_one_square_at_tile_edges(N, fill):
    nocc = int(fill * N)                                    # both polynomials
    F = inputs.dense_gapped(N, nocc, gap=0.1, seed=N).F.numpy()
    check(*one_square(F, (-1.5, 1.5), nocc))


@pytest.mark.parametrize("N", [700, 1001, 1500, 2049, 3000])     # k ranges split over 4, 2, 4, 1 and 1 CTAs, or so
def test_one_square_against_fp64_matmul(N):
    F = torch.randn(N, N, dtype=torch.float64, generator=torch.Generator().manual_seed(N)).cuda()
    F = (F + F.T) / (4 * N ** 0.5)
    nocc = N // 3
    from paper_1507_02087_gb300 import sp2
    with sp2.Purifier(N, nocc, "fp64", max_iter=1, guard=False) as P:
        P.set_bounds((-1.5, 1.5))
        X1 = P.run(F)
        info = P.info()
    X0 = (1.5 * torch.eye(N, dtype=torch.float64, device="cuda") - F) / 3.0
    S = X0 @ X0                                              # its own error is within the same bound
    ref = S if info["p"][1] else 2 * X0 - S
    norms = torch.linalg.norm(X0, dim=1)
    bound = 16 * EPS * N ** 0.5 * torch.outer(norms, norms) + 2 * EPS * ref.abs()
    assert bool(((X1 - ref).abs() <= bound).all()) and torch.equal(X1, X1.T)
    v = float(torch.linalg.norm(X0 - S))
    assert info["v"][0] == pytest.approx(v, rel=1e-12)
    assert info["trace"][1] == pytest.approx(float(torch.trace(ref)), rel=1e-12)


@pytest.mark.parametrize("scale", [1e-6, 1e-30, 1e-120])
def test_one_square_of_rows_of_different_scale(scale):
    # a block-diagonal matrix whose X_0 has rows of norm 1, of norm `scale` and zero rows
    N = 300
    g = np.random.Generator(np.random.PCG64(7))
    A = g.standard_normal((N, N)) / N
    w = np.where(np.arange(N) % 3 == 0, 1.0, np.where(np.arange(N) % 3 == 1, scale, 0.0))
    X = w[:, None] * (A + A.T) * w[None, :]
    X0, X1, p = one_square(-X, (-1.0, 0.0), 100)            # lmax = 0: X_0 = -F exactly
    check(X0, X1, p)


def test_a_row_with_an_overflow_ends_the_run():
    # finite input whose square is not: reported, as by the FP64 units
    from paper_1507_02087_gb300 import sp2
    N = 200
    F = inputs.dense_gapped(N, 100, gap=0.1, seed=3).F.numpy() * 1e200
    with sp2.Purifier(N, 100, "fp64") as P:
        P.set_bounds((-1.0, 1.0))                           # far too narrow
        P.run(torch.from_numpy(F).cuda())
        assert P.info()["status"] == 3


@pytest.mark.parametrize("mode,xi", [("mcw", 0.0), ("mcw-acc", 0.05)])
@pytest.mark.parametrize("N", [130, 257, 500])
def test_mcweeny_products_at_tile_edges(N, mode, xi):
    from oracle import mcweeny_oracle as om
    from oracle import sp2_oracle as o
    from paper_1507_02087_gb300 import sp2
    case = inputs.dense_gapped(N, N // 2, gap=0.05, seed=N)
    with sp2.Purifier(N, N // 2, "fp64") as P:
        P.set_mcweeny(mode, 0.0, xi)
        D = P.run(case.F.cuda()).cpu().numpy()
        info = P.info()
    ref = om.mcweeny(case.F.numpy(), 0.0, xi=xi, accelerate=(mode == "mcw-acc"),
                     bounds=(info["lambda_min"], info["lambda_max"]))
    assert info["status"] == 0 and abs(info["n_iter"] - ref.n) <= 1
    assert o.rel_error(D, ref.D, N // 2) <= 1e-12


@pytest.mark.parametrize("left,mcw,used", [(90, False, 67), (150, False, 126), (150, True, 101), (250, True, 218)])
def test_a_handle_without_room_for_the_digits_uses_the_fp64_units(left, mcw, used):
    # MB left on the device at create: two iterates take 67, the digits 59 each, the McWeeny square 34.
    # At 90 the digits fail; at 150 the square takes their place.
    from paper_1507_02087_gb300 import sp2
    N, MB = 2048, 1 << 20
    case = inputs.dense_gapped(N, N // 2, gap=0.05, seed=1)
    F, D = case.F.cuda(), torch.empty(N, N, dtype=torch.float64, device="cuda")
    free = lambda: torch.cuda.mem_get_info()[0]

    def solve():
        before = free()
        with sp2.Purifier(N, N // 2, "fp64") as P:
            if mcw:
                P.set_mcweeny("mcw-acc", 0.0, 0.05)
            took = (before - free()) / 1e6
            P.run(F, D)
            return D.cpu(), P.info(), took

    want, winfo, _ = solve()                                 # with room; loads the kernels too
    torch.cuda.empty_cache()
    hog = []
    try:
        for size in (1 << 30, 64 * MB, 16 * MB, 2 * MB):
            while free() > left * 10**6 + size:
                hog.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
        got, info, took = solve()
    except torch.cuda.OutOfMemoryError:
        pytest.skip("the device's free memory moved")
    finally:
        del hog
        torch.cuda.empty_cache()
    assert used - 5 <= took <= used + 8, took
    # (where the runs stop may differ: the units' rounding floor is higher)
    assert info["status"] == winfo["status"] == 0
    assert float(torch.linalg.norm(got - want)) <= 1e-11 * (N / 2) ** 0.5
