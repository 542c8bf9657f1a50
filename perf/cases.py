"""The measured workloads of the library: what a program that purifies Fock matrices asks of it.

Each case names one use of a public class (`Purifier`, `BatchPurifier`, `BsrPurifier`) with its size
and options.  `prepare` makes the inputs on the GPU and the handle such a program keeps between
calls (an SCF loop purifies one matrix after another of the same size); `run` is one purification
F -> D through that handle.

Dense inputs: F = Q diag(lam) Q^T with the occupied eigenvalues uniform in [-1, -gap/2], the virtual
ones uniform in [gap/2, 1] and Q = I - 2 V (V^T V)^-1 V^T, a reflection through the span of N/2
Gaussian vectors: an orthogonal matrix with delocalised columns that needs matrix products only.
The exact density matrix is then Q_occ Q_occ^T.  Block-sparse inputs: the gapped tight-binding
lattice of the benchmark (onsite +-1 with disorder, hopping -0.3), whose 32 x 32 blocks are the
x-lines of the lattice.
"""
import math

import numpy as np
import torch

from paper_1507_02087_gb300 import sp2

DISORDER = 0.05


def _dense(name, N, nocc, gap, precision, **more):
    return dict(name=name, kind="dense", N=N, nocc=nocc, gap=gap, precision=precision, **more)


def listed():
    return [
        # FP64, the default precision of a handle.  The smallest call: a molecule of a few atoms,
        # where launches and latency are everything.
        _dense("fp64_n64", 64, 30, 0.1, "fp64"),
        # A small molecule at full precision (the N = 400 workload of the benchmark).
        _dense("fp64_n400", 400, 200, 0.1, "fp64"),
        # The size of the paper's dense example with the stop on the spectral norm, on which the
        # stop is defined; one above and below multiples of the tile sizes on purpose.
        _dense("fp64_spectral_n1001", 1001, 500, 0.01, "fp64", norm="spectral"),
        # The accelerated McWeeny expansion: chemical potential and a gap estimate are known.
        _dense("fp64_mcw_acc_n1500", 1500, 600, 0.05, "fp64", expansion="mcw-acc"),
        # A mid-size basis at full precision.
        _dense("fp64_n2048", 2048, 1024, 0.01, "fp64"),
        # The same small molecule on the tensor-core path.
        _dense("fp16x3_n400", 400, 200, 0.1, "fp16x3"),
        # An SCF step that knows homo and lumo from the step before: the accelerated expansion, one
        # row more than a whole number of tiles, in the tf32 mode.
        _dense("tf32x3_acc_n2049", 2049, 700, 0.01, "tf32x3", expansion="acc"),
        # An odd size and a third filled, in the bf16x6 mode (the default of a batch).
        _dense("bf16x6_n3001", 3001, 1000, 0.02, "bf16x6"),
        # The headline workload: a large dense matrix with a small gap.
        _dense("fp16x3_n8192", 8192, 4096, 0.01, "fp16x3"),
        # Many molecules of uneven size at once (the batch workload of the benchmark).
        dict(name="batch64_fp16x3", kind="batch", count=64, nmin=128, nmax=2048, precision="fp16x3"),
        # Block-sparse with error-controlled truncation: a small lattice whose block rows fill
        # neither the tiles nor the bitmap words.
        dict(name="bsr_error_11x10", kind="bsr", Ly=11, Lz=10, tau=1e-4, rule="error", norm="fro"),
        # Block-sparse at the benchmark's size with the mixed-norm truncation and stop.
        dict(name="bsr_mixed_32x32", kind="bsr", Ly=32, Lz=32, tau=1e-4, rule="mixed", norm="mixed"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.random()
    gap = round(math.exp(rng.uniform(math.log(0.005), math.log(0.1))), 5)
    if pick < 0.75:
        fp64 = pick < 0.4
        precision = "fp64" if fp64 else rng.choice(["fp16x3", "fp16x3", "bf16x6", "tf32x3"])
        N = _log_int(rng, 48, 2048) if fp64 else _log_int(rng, 100, 8192 if precision == "fp16x3" else 4096)
        case = dict(kind="dense", N=N, nocc=max(1, int(N * rng.uniform(0.1, 0.9))), gap=gap, precision=precision)
        kinds = ["sp2", "sp2", "acc"] + (["mcw", "mcw-acc"] if fp64 else [])
        case["expansion"] = rng.choice(kinds)
        case["norm"] = rng.choice(["fro", "fro", "mixed", "spectral"])
        return case
    if pick < 0.85:
        nmax = _log_int(rng, 256, 2048)
        return dict(kind="batch", count=rng.randint(2, 64), nmin=rng.randint(48, 128), nmax=nmax,
                    precision=rng.choice(["fp16x3", "bf16x6"]))
    rule = rng.choice(["block", "error", "mixed"])
    return dict(kind="bsr", Ly=rng.randint(4, 24), Lz=rng.randint(1, 24), tau=rng.choice([1e-5, 1e-4, 1e-3]),
                rule=rule, norm="mixed" if rule == "mixed" else "fro")


# ---- inputs ----------------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _spectrum_and_basis(N, nocc, gap, seed):
    g = _generator(seed)
    u = torch.rand(N, generator=g, device="cuda", dtype=torch.float64)
    lam = gap / 2 + (1.0 - gap / 2) * u
    lam[:nocc].neg_()
    V = torch.randn(N, max(1, N // 2), generator=g, device="cuda", dtype=torch.float64)
    L = torch.linalg.cholesky(V.T @ V)
    W = torch.linalg.solve_triangular(L, V.T, upper=False)      # orthonormal rows
    Q = -2.0 * (W.T @ W)
    Q.diagonal().add_(1.0)
    return lam, Q


def _dense_problem(N, nocc, gap, seed):
    lam, Q = _spectrum_and_basis(N, nocc, gap, seed)
    F = (Q * lam) @ Q.T
    F = 0.5 * (F + F.T)
    inner = (float(lam[:nocc].max()), float(lam[nocc:].min())) if 0 < nocc < N else None
    return F.contiguous(), inner


def _batch_problems(case, seed):
    g = np.random.Generator(np.random.PCG64(1))                # the sizes are the case's, not the seed's
    logs = g.uniform(math.log(case["nmin"]), math.log(case["nmax"]), size=case["count"])
    gaps = g.uniform(0.005, 0.1, size=case["count"])
    return [(int(round(math.exp(x))), int(round(math.exp(x))) // 2, float(gp), seed * 1009 + k)
            for k, (x, gp) in enumerate(zip(logs, gaps))]


def _lattice_pairs(Ly, Lz):
    """(I, J) of the stored blocks, sorted: each x-line, and its neighbours in y and z (periodic)."""
    I = np.arange(Ly * Lz)
    y, z = I % Ly, I // Ly
    ends = [I, (y + 1) % Ly + Ly * z, (y - 1) % Ly + Ly * z, y + Ly * ((z + 1) % Lz), y + Ly * ((z - 1) % Lz)]
    return np.unique(np.stack([np.tile(I, 5), np.concatenate(ends)], axis=1), axis=0)


def _lattice(case, seed):
    Ly, Lz, b = case["Ly"], case["Lz"], 32
    nb = Ly * Lz
    I = torch.arange(nb, device="cuda")
    x = torch.arange(b, device="cuda")
    parity = (x[None, :] + (I % Ly + I // Ly)[:, None]) % 2
    noise = torch.randn(nb, b, generator=_generator(seed), device="cuda", dtype=torch.float64)
    onsite = torch.where(parity == 0, 1.0, -1.0).double() + DISORDER * noise
    pairs = _lattice_pairs(Ly, Lz)
    row_ptr = np.zeros(nb + 1, dtype=np.int32)
    row_ptr[1:] = np.cumsum(np.bincount(pairs[:, 0], minlength=nb))
    diagonal = torch.from_numpy(np.flatnonzero(pairs[:, 0] == pairs[:, 1])).cuda()
    vals = (-0.3 * torch.eye(b, device="cuda", dtype=torch.float64)).repeat(len(pairs), 1, 1)
    ring = torch.zeros(b, b, device="cuda", dtype=torch.float64)
    ring[x, (x + 1) % b] = -0.3
    ring[(x + 1) % b, x] = -0.3
    vals[diagonal] = ring + torch.diag_embed(onsite)
    return torch.from_numpy(row_ptr).cuda(), torch.from_numpy(pairs[:, 1].astype(np.int32)).cuda(), vals.contiguous()


# ---- the measured calls ------------------------------------------------------------------------

def prepare(case, seed):
    if case["kind"] == "bsr":
        rp, ci, vals = _lattice(case, seed)
        N = 32 * case["Ly"] * case["Lz"]
        p = sp2.BsrPurifier(N, N // 2, case["tau"], rule=case["rule"], norm=case["norm"])
        return dict(kind="bsr", p=p, F=(rp, ci, vals), D=torch.empty(N, N, device="cuda", dtype=torch.float64))
    if case["kind"] == "batch":
        probs = _batch_problems(case, seed)
        Fs = [_dense_problem(*q)[0] for q in probs]
        p = sp2.BatchPurifier([q[0] for q in probs], [q[1] for q in probs], case["precision"])
        return dict(kind="batch", p=p, F=Fs, D=[torch.empty_like(F) for F in Fs])
    N, nocc, gap = case["N"], case["nocc"], case["gap"]
    F, inner = _dense_problem(N, nocc, gap, seed)
    p = sp2.Purifier(N, nocc, case["precision"], norm=case.get("norm", "fro"))
    expansion = case.get("expansion", "sp2")
    if expansion == "acc":
        p.set_homo_lumo((inner[0] - 1e-3, inner[0], inner[1], inner[1] + 1e-3))
    elif expansion in ("mcw", "mcw-acc"):
        # the middle of the gap, and a width around it that holds an eigenvalue
        p.set_mcweeny(expansion, mu=0.5 * (inner[0] + inner[1]), xi=1.001 * (inner[1] - inner[0]))
    return dict(kind="dense", p=p, F=F, D=torch.empty_like(F))


def run(state):
    if state["kind"] == "bsr":
        return state["p"].run(*state["F"], D=state["D"])
    return state["p"].run(state["F"], state["D"])


# ---- the work of one pass and the exact results ------------------------------------------------

def _dense_work(N, gap, expansion="sp2"):
    # F in, D out; N^2 (N + 1) flops a symmetric product.  Products: about 3.3 squares per doubling of
    # the scaled gap (bounds about 0.92 sqrt(N) wide for these matrices) and 11 for the purification;
    # the accelerated expansions take about half.
    n = 3.3 * math.log2(max(2.0, 0.92 * math.sqrt(N)) / gap) + 12
    n *= {"sp2": 1.0, "acc": 0.55, "mcw": 1.05, "mcw-acc": 0.57}[expansion]
    return 16.0 * N * N, n * N * N * (N + 1.0)


def work(case):
    if case["kind"] == "dense":
        b, f = _dense_work(case["N"], case["gap"], case.get("expansion", "sp2"))
    elif case["kind"] == "batch":
        both = [_dense_work(N, gap) for N, _, gap, _ in _batch_problems(case, 0)]
        b, f = sum(x for x, _ in both), sum(y for _, y in both)
    else:
        # blocks of D decay with the distance of the x-lines: about pi r^2 of them in a block row, r
        # growing with log(1 / tau); half the products of the last pattern on average, 15 squares
        nb = case["Ly"] * case["Lz"]
        c = min(nb, math.pi * (0.97 * math.log(1.0 / case["tau"])) ** 2)
        b, f = 8.0 * (32.0 * nb) ** 2 + 5.0 * nb * 8192, 15.0 * nb * c * c / 4 * 2 * 32 ** 3
    return {"bytes": b, "flops": f}


def _projector(N, nocc, gap, seed):
    Qo = _spectrum_and_basis(N, nocc, gap, seed)[1][:, :nocc]
    return Qo @ Qo.T


def exact(case, seed):
    if case["kind"] == "dense":
        return _projector(case["N"], case["nocc"], case["gap"], seed)
    if case["kind"] == "batch":
        return [_projector(*q) for q in _batch_problems(case, seed)]
    nb = case["Ly"] * case["Lz"]
    if nb > 128:
        return None                                             # an eigensolver would take too long
    rp, ci, vals = _lattice(case, seed)
    row = torch.repeat_interleave(torch.arange(nb, device="cuda"), (rp[1:] - rp[:-1]).long())
    F = torch.zeros(nb, nb, 32, 32, device="cuda", dtype=torch.float64)
    F[row, ci.long()] = vals
    U = torch.linalg.eigh(F.permute(0, 2, 1, 3).reshape(32 * nb, 32 * nb))[1][:, :16 * nb]
    return U @ U.T
