"""The digit scheme of the FP64 products (csrc/sp2_f64_tc.cu), restated in integers.

Row i is d_0 .. d_6 (8 bits each, signed) times 2^(e_i - 8 (a + 1)); V_s sums the digit products with a + b = s over k,
for s <= 7.  The kernel adds the V_s as 64-bit integers in units of 2^(e_i + e_j - 62), so V_0 .. V_5 exactly, and
rounds V_6 2^-2 and V_7 2^-10 to whole units each time it drains them: at most once in four blocks of 32 k-columns
and once more at the end of each CTA's share, so at most ld / 128 + ks half units for each of the two sums.  Then
one rounding to FP64.  `kept_sums` has the exact value, and an element of the product has to be within
ld / 128 + ks units and half an FP64 unit of it, with any split.
"""
import numpy as np
import pytest
import torch

SHAPES = [(32, 1), (64, 1), (64, 2), (64, 4), (64, 8)]
ND, NS = 7, 8


def exponents(X):
    m = np.frexp(np.abs(X).max(axis=1))[1]                  # max |x| in [2^(m - 1), 2^m)
    norm = np.frexp(np.linalg.norm(X, axis=1) * 1.0005)[1]  # ||x|| < 2^norm
    return np.maximum(m + 1, norm).astype(np.int64)


def fixed_point(X, e):
    a = np.abs(np.ldexp(X, 56 - e[:, None]))
    f = np.floor(a)
    return (np.sign(X) * (f + (a - f >= 0.5))).astype(np.int64)


def digits(X, e):
    y = fixed_point(X, e)
    d = [None] * ND
    for a in range(ND - 1, 0, -1):
        d[a] = (y & 255).astype(np.uint8).astype(np.int8).astype(np.int64)
        y = (y - d[a]) >> 8
    d[0] = y
    assert np.abs(y).max() <= 128
    return d


def kept_sums(d, drop=()):
    """(whole units, 1024ths of a unit): the kept sums, exactly."""
    f = [x.astype(np.float64) for x in d]                    # integer products and sums far below 2^53: exact
    V = [sum(f[a] @ f[s - a].T for a in range(max(0, s - ND + 1), min(s, ND - 1) + 1)) for s in range(NS)]
    V = [v.astype(np.int64) * (s not in drop) for s, v in enumerate(V)]
    return sum(V[s] << (46 - 8 * s) for s in range(6)), V[6] * 256 + V[7]


def units_off(S, e, whole, part):
    """Distance of S from the kept sums in units of 2^(e_i + e_j - 62), and half an FP64 unit of S in them."""
    t = np.ldexp(S, 62 - e[:, None] - e[None, :])
    d = (t.astype(np.longdouble) - whole.astype(np.longdouble)) - part.astype(np.longdouble) / 1024
    return np.abs(d).astype(np.float64), np.abs(t) * 2.0 ** -53


def limit(N, ks):
    return (N + 63) // 64 * 64 / 128 + ks


def round_to_fp64(whole, part, e):
    """What a kernel that rounds once, at the end, would return."""
    return np.ldexp((whole + ((part + 512) >> 10)).astype(np.float64), e[:, None] + e[None, :] - 62)


def gaussian(N, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    X = g.standard_normal((N, N)) / N ** 0.5
    return (X + X.T) / 2


def graded(N, seed):
    """A local matrix: entries decay by ten per eight off the diagonal."""
    i = np.arange(N)
    return gaussian(N, seed) * 10.0 ** (-np.abs(i[:, None] - i[None, :]) / 8.0)


def near_the_limit(N):
    """Rows of one value whose lower digits are all -128, so that V_2 .. V_7 come near 2^24 between two drains; in every
    other row an entry of the opposite sign cancels most of the product with the others, so that nothing hides in the
    rounding of the sum."""
    values = [np.ldexp(top * 2.0 ** 48 - 128 * ((2 ** 48 - 1) // 255), -56) for top in range(1, 128)]
    c = next(c for c in values if 0.25 <= c * (N - 1) ** 0.5 < 0.5)      # e_i = 0
    X = np.full((N, N), c)
    X[0::2, 5] = c * (N - 1) ** 0.5
    X[1::2, 5] = -c * (N - 1) ** 0.5
    return X


MATRICES = {"gaussian": lambda N: gaussian(N, N), "graded": lambda N: graded(N, N), "limit": near_the_limit}


def exact_product(X):
    """X X^T to far more than FP64: the products of 26-bit halves are exact, their sums in extended precision."""
    h = X.astype(np.float32).astype(np.float64)
    l = X - h
    L = np.longdouble
    return ((h.astype(L) @ h.T.astype(L)) + (h.astype(L) @ l.T.astype(L)) + (l.astype(L) @ h.T.astype(L)) +
            (l.astype(L) @ l.T.astype(L)))


def documented_bound(X, S):
    N = X.shape[0]
    n = np.linalg.norm(X, axis=1)
    return (2.0 ** -54 * N ** 0.5 + 2.0 ** -59 * N) * np.outer(n, n) * 1.001 + 2.0 ** -53 * np.abs(S)


@pytest.mark.parametrize("kind", MATRICES)
def test_the_scheme_keeps_the_documented_bound(kind):
    X = MATRICES[kind](300)
    e = exponents(X)
    norms = np.linalg.norm(X, axis=1)
    assert np.all(np.ldexp(1.0, e) <= 4 * norms) and np.all(norms < np.ldexp(1.0, e))
    S = round_to_fp64(*kept_sums(digits(X, e)), e)
    err = np.abs(S - exact_product(X)).astype(np.float64)
    assert np.all(err <= documented_bound(X, S)), float((err / documented_bound(X, S)).max())


def test_small_elements_lose_relative_accuracy():
    # what the bound leaves open: entries far below their rows' norms.  FP64 multiply-adds keep them
    X = graded(400, 1)
    e = exponents(X)
    S, R = round_to_fp64(*kept_sums(digits(X, e)), e), exact_product(X)
    far = np.abs(np.subtract.outer(np.arange(400), np.arange(400))) > 120
    rel = (np.abs(S - R) / np.abs(R)).astype(np.float64)
    assert np.median(rel[far]) > 1e-3 and np.median((np.abs(X @ X.T - R) / np.abs(R)).astype(np.float64)[far]) < 1e-13
    assert np.linalg.norm((S - R).astype(np.float64)) < 1e-15 * np.linalg.norm(S)


@pytest.mark.parametrize("lost", range(NS))
def test_a_lost_sum_is_outside_the_limit(lost):
    # the tests below see any of the eight sums go missing, the lightest (V_7, 2^-10 of a unit each) among them
    X = gaussian(300, 300)
    e = exponents(X)
    d = digits(X, e)
    off, half = units_off(round_to_fp64(*kept_sums(d, drop=(lost,)), e), e, *kept_sums(d))
    assert np.mean(off > limit(300, 8) + half) > 0.5


def test_the_limit_matrix_comes_near_the_accumulators_limit():
    d = digits(near_the_limit(256), exponents(near_the_limit(256)))
    f = [x[0, 128:].astype(np.int64) for x in d]
    peak = {s: sum(int(f[a] @ f[s - a]) for a in range(max(0, s - ND + 1), min(s, ND - 1) + 1)) for s in range(2, NS)}
    assert peak[7] > 0.7 * 2 ** 24 and max(abs(v) for v in peak.values()) <= 2 ** 24


@pytest.mark.gpu
@pytest.mark.parametrize("kind", MATRICES)
@pytest.mark.parametrize("bn,ks", SHAPES)
@pytest.mark.parametrize("N", [129, 300, 449, 700])
def test_product_on_the_gpu(N, bn, ks, kind):
    from paper_1507_02087_gb300 import sp2
    X = MATRICES[kind](N)
    Xd = torch.from_numpy(X).cuda()
    out, exps = torch.empty_like(Xd), torch.empty(N, dtype=torch.int32, device="cuda")
    assert sp2.lib().sp2_test_f64_product(Xd.data_ptr(), N, bn, ks, 0, 0, out.data_ptr(), exps.data_ptr(),
                                          torch.cuda.current_stream().cuda_stream) == 0
    S, e = out.cpu().numpy(), exps.cpu().numpy().astype(np.int64)
    norms = np.linalg.norm(X, axis=1)
    assert np.all(norms < np.ldexp(1.0, e)) and np.all(np.ldexp(1.0, e) <= 4 * norms)
    assert np.all(np.abs(X).max(axis=1) <= np.ldexp(1.0, e - 1)) and np.array_equal(S, S.T)
    off, half = units_off(S, e, *kept_sums(digits(X, e)))
    assert np.all(off <= limit(N, ks) + half), float((off / (limit(N, ks) + half)).max())
