"""The 8 x 8 tiles of the smallest FP64 problems (N <= 128, csrc/sp2_dense_f64.cu), and the Lanczos estimate of
the spectral stop on either side of the size up to which its vector is kept in shared memory."""
import numpy as np
import pytest
import torch

from paper_1507_02087_gb300 import inputs

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.mark.parametrize("N", [2, 7, 8, 9, 63, 64, 65, 120, 127, 128])
@pytest.mark.parametrize("fill", [0.3, 0.7])
def test_one_square(N, fill):
    # one step from X_0 (formed here as the library forms it): an FMA chain of N terms, halved
    from paper_1507_02087_gb300 import sp2
    nocc = max(1, int(fill * N))
    F = inputs.dense_gapped(N, nocc, gap=0.1, seed=N).F.numpy()
    with sp2.Purifier(N, nocc, "fp64", max_iter=1, guard=False) as P:
        P.set_bounds((-1.5, 1.5))
        X1 = P.run(torch.from_numpy(F).cuda()).cpu().numpy()
        info = P.info()
    X0 = (1.5 * np.eye(N) - F) / 3.0
    L = X0.astype(np.longdouble)
    S = L @ L
    ref = S if info["p"][1] else 2 * L - S
    bound = (N + 4) * EPS * (np.abs(X0) @ np.abs(X0)) + 4 * EPS * np.abs(X0)
    assert np.all(np.abs((X1.astype(np.longdouble) - ref).astype(float)) <= bound)
    assert np.array_equal(X1, X1.T)
    assert info["v"][0] == pytest.approx(float(np.linalg.norm((L - S).astype(float))), rel=1e-12)


@pytest.mark.parametrize("N", [60, 100, 128])
@pytest.mark.parametrize("mode", [None, "mcw", "mcw-acc"])
def test_runs_against_the_oracle(N, mode):
    from oracle import mcweeny_oracle as om
    from oracle import sp2_oracle as o
    from paper_1507_02087_gb300 import sp2
    case = inputs.dense_gapped(N, N // 2, gap=0.05, seed=N)
    with sp2.Purifier(N, N // 2, "fp64", norm="fro" if mode else "mixed") as P:
        if mode:
            P.set_mcweeny(mode, 0.0, 0.05)
        D = P.run(case.F.cuda()).cpu().numpy()
        info = P.info()
    bounds = (info["lambda_min"], info["lambda_max"])
    if mode:
        ref = om.mcweeny(case.F.numpy(), 0.0, xi=0.05, accelerate=mode == "mcw-acc", bounds=bounds)
    else:
        ref = o.sp2(case.F.numpy(), N // 2, norm="mixed", block=64, bounds=bounds)
    assert info["status"] == 0 and abs(info["n_iter"] - ref.n) <= 1
    assert o.rel_error(D, ref.D, N // 2) <= 1e-11
    for i in range(min(len(ref.v), info["hist_len"])):
        if ref.v[i] > 1e-7:
            assert info["v"][i] == pytest.approx(ref.v[i], rel=1e-8)


@pytest.mark.parametrize("scale", [1.0, 3e-4, 7e7, 1e-200, 1e250])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_scaling_is_the_correctly_rounded_quotient(scale, seed):
    # diagonal F: every step is one rounding per element, so X_6 equals the scalar recursion's bit for bit only if
    # every X_0 entry is the quotient (lmax - f) / (lmax - lmin) as IEEE division rounds it.  (Six steps: where the
    # run itself stops is decided by traces at the rounding floor.)
    from oracle import sp2_oracle as o
    from paper_1507_02087_gb300 import sp2
    g = np.random.Generator(np.random.PCG64(seed))
    N, nocc = 128, 50
    lam = scale * np.concatenate([g.uniform(-1, -0.02, nocc), g.uniform(0.03, 1.0, N - nocc)])
    g.shuffle(lam)
    F = torch.from_numpy(np.diag(lam)).cuda()
    with sp2.Purifier(N, nocc, "fp64", max_iter=6, guard=False) as P:
        D = P.run(F).cpu().numpy()
        info = P.info()
    lo, hi = o.gershgorin_bounds(np.diag(lam))
    xs, n, reason, *_ = o.sp2_scalar(lam, nocc, lo, hi, max_iter=6, guard=False)
    assert info["n_iter"] == n == 6 and np.array_equal(np.diag(D), np.array(xs))


@pytest.mark.parametrize("N", [33, 2431, 2433, 16384, 16448])
def test_spectral_estimate_of_a_known_matrix(N):
    # diagonal F with three eigenvalues: X_0 = 0.1 I but for a few entries of 0.5 and 0.99, so e_0 = 1/4 exactly,
    # well separated: 32 Lanczos steps find it to FP32 rounding (the Krylov space ends after three)
    from paper_1507_02087_gb300 import sp2
    F = torch.zeros(N, N, dtype=torch.float64, device="cuda")
    d = F.diagonal()
    d.fill_(0.8)                                             # X_0 = (1 - F) / 2
    d[::7] = 0.0
    d[1::11] = -0.98
    with sp2.Purifier(N, N // 2, "fp64", max_iter=1, guard=False, norm="spectral") as P:
        P.set_bounds((-1.0, 1.0))
        P.run(F)
        info = P.info()
    assert info["status"] == 0 and info["v"][0] == pytest.approx(0.25, rel=1e-5)
