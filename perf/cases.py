"""The work this library is used for, as measurable cases.

A case describes driven systems (Eq. 1 of the multimode Floquet method), a precision and the results
asked for; ``prepare`` makes the systems from a seed and the plan or handle a program keeps, ``run``
is one pass through the public API (the ``mmf`` binding of include/mmf.h), ``work`` what a pass
cannot do without, and ``exact`` the same results from a dense 64-bit eigendecomposition in torch.

Kinds:
  sequence  the paper's call sequence for one system through the single-system handle, host results
  batch     a batch plan: coefficients and times uploaded, solved, results left in torch tensors
  evolve    U(t, t0) on a time grid from eigenpairs that are already on the device
  serve     a burst of requests to the continuous-batching server, each waited for
"""

import math
import os

import numpy as np
import torch

from paper_2005_03426_gb300 import mmf
from paper_2005_03426_gb300 import workloads as W

TUNING = os.path.join(os.path.dirname(os.path.abspath(mmf.__file__)), "tuning_gb300.txt")
PRECISION = {"fp64": mmf.MMF_FP64, "mixed": mmf.MMF_MIXED}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one qubit through the paper's one-system calls, FP64 as in the paper: the smallest call,
        # where plan creation, launches and host waits count
        {"name": "qubit_sequence_fp64", "kind": "sequence", "family": "qubit", "precision": "fp64", "N1": 20, "nt": 64},
        # the paper's spectroscopy sweep: 200 drive frequencies of one qubit, n = 82, FP64, captured
        # in a graph and repeated
        {"name": "qubit_sweep_fp64", "kind": "batch", "family": "qubit", "precision": "fp64", "count": 200, "N1": 20,
         "nt": 64, "graph": True},
        # one spin-1 system at two incommensurate frequencies, n = 1323: the latency of one solve
        {"name": "spin1_one_mixed", "kind": "batch", "family": "spin1", "precision": "mixed", "count": 1, "N1": 10,
         "N2": 10, "nt": 64, "graph": False},
        # 64 amplitude pairs of it: the benchmark's sweep
        {"name": "spin1_sweep_mixed", "kind": "batch", "family": "spin1", "precision": "mixed", "count": 64, "N1": 10,
         "N2": 10, "nt": 64, "graph": False},
        # the same systems on the plain FP64 path
        {"name": "spin1_sweep_fp64", "kind": "batch", "family": "spin1", "precision": "fp64", "count": 8, "N1": 10,
         "N2": 10, "nt": 64, "graph": False},
        # an uneven batch in one plan: 2..8 levels, one or two modes, dimensions 18 to 2000
        {"name": "uneven_mixed", "kind": "batch", "family": "uneven", "precision": "mixed", "count": 256, "nmax": 2000,
         "shapes": 0, "nt": 64, "graph": False},
        # small and middling uneven systems in FP64
        {"name": "uneven_fp64", "kind": "batch", "family": "uneven", "precision": "fp64", "count": 96, "nmax": 500,
         "shapes": 1, "nt": 64, "graph": False},
        # spectrum of the driven lattice (256 sites, n = 1792) against the drive frequency
        {"name": "lattice_spectrum_mixed", "kind": "batch", "family": "lattice", "precision": "mixed", "count": 16,
         "D": 256, "N1": 3, "nt": 0, "graph": False},
        # one large system: 8 levels, three modes, n = 5832
        {"name": "three_modes_mixed", "kind": "batch", "family": "three", "precision": "mixed", "count": 1, "D": 8,
         "N1": 4, "N2": 4, "N3": 4, "nt": 256, "graph": False},
        # time evolution on a fine grid from resident eigenpairs
        {"name": "evolve_mixed", "kind": "evolve", "family": "spin1", "precision": "mixed", "N1": 10, "N2": 10,
         "nt": 512},
        # a burst of requests: qubits, spin-1 systems and uneven draws, a third each
        {"name": "serve_burst_mixed", "kind": "serve", "precision": "mixed", "count": 24, "shapes": 2, "nt": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sequence", "sequence", "qubit", "spin1", "spin1", "spin1_fp64", "uneven", "uneven", "uneven_fp64",
                       "lattice", "three", "evolve", "evolve", "serve"])
    if kind == "sequence":
        c = {"kind": "sequence", "family": rng.choice(["qubit", "spin1"]), "precision": rng.choice(["fp64", "mixed"])}
        if c["family"] == "qubit":
            c["N1"] = rng.randint(4, 60)
        else:
            c["N1"], c["N2"] = rng.randint(2, 6), rng.randint(2, 5)
        return {**c, "nt": _log_int(rng, 8, 256)}
    if kind == "qubit":
        return {"kind": "batch", "family": "qubit", "precision": rng.choice(["fp64", "mixed"]),
                "count": _log_int(rng, 8, 400), "N1": rng.randint(4, 30), "nt": _log_int(rng, 8, 128),
                "graph": rng.random() < 0.5}
    if kind == "spin1":
        return {"kind": "batch", "family": "spin1", "precision": "mixed", "count": _log_int(rng, 1, 64),
                "N1": rng.randint(4, 10), "N2": rng.randint(3, 10), "nt": _log_int(rng, 8, 128), "graph": False}
    if kind == "spin1_fp64":
        return {"kind": "batch", "family": "spin1", "precision": "fp64", "count": _log_int(rng, 1, 8),
                "N1": rng.randint(4, 10), "N2": rng.randint(3, 10), "nt": _log_int(rng, 8, 128), "graph": False}
    if kind == "uneven":
        return {"kind": "batch", "family": "uneven", "precision": "mixed", "count": _log_int(rng, 8, 256),
                "nmax": _log_int(rng, 200, 2000), "shapes": rng.randint(100, 10 ** 6), "nt": _log_int(rng, 8, 128),
                "graph": False}
    if kind == "uneven_fp64":
        return {"kind": "batch", "family": "uneven", "precision": "fp64", "count": _log_int(rng, 8, 96),
                "nmax": _log_int(rng, 100, 500), "shapes": rng.randint(100, 10 ** 6), "nt": _log_int(rng, 8, 128),
                "graph": False}
    if kind == "lattice":
        return {"kind": "batch", "family": "lattice", "precision": "mixed", "count": _log_int(rng, 1, 16),
                "D": rng.randint(64, 256), "N1": rng.randint(2, 3), "nt": 0, "graph": False}
    if kind == "three":
        N = [rng.randint(2, 4) for _ in range(3)]
        return {"kind": "batch", "family": "three", "precision": "mixed", "count": 1, "D": rng.randint(4, 8), "N1": N[0],
                "N2": N[1], "N3": N[2], "nt": _log_int(rng, 16, 256), "graph": False}
    if kind == "evolve":
        return {"kind": "evolve", "family": "spin1", "precision": rng.choice(["fp64", "mixed"]), "N1": rng.randint(4, 10),
                "N2": rng.randint(3, 10), "nt": _log_int(rng, 32, 512)}
    return {"kind": "serve", "precision": "mixed", "count": rng.randint(6, 24), "shapes": rng.randint(100, 10 ** 6),
            "nt": _log_int(rng, 16, 64)}


# ------------------------------------------------------------------ systems
def _uneven_shapes(count, seed, nmax):
    """(D, truncations) as W.uneven_batch draws them: 2..8 levels, one or two modes, N in 4..30, n <= nmax."""
    rng, out = W.SplitMix64(seed), []
    while len(out) < count:
        D = rng.integer(2, 8)
        Ns = [rng.integer(4, 30) for _ in range(rng.integer(1, 2))]
        if D * math.prod(2 * N + 1 for N in Ns) <= nmax:
            out.append((D, Ns))
    return out


def _problems(case, seed):
    rng = W.SplitMix64(seed)
    if case["kind"] == "serve":
        # a third each of qubits (n = 82), spin-1 systems (n = 1323) and uneven draws, in turn
        shapes = _uneven_shapes(case["count"], case["shapes"], 2000)
        out = []
        for i in range(case["count"]):
            if i % 3 == 0:
                out.append(W.two_level(rng.uniform_in(0.2, 2.0), N=20))
            elif i % 3 == 1:
                a1 = rng.uniform_in(0.05, 0.5)
                out.append(W.spin1_bichromatic(a1, rng.uniform_in(0.05, 0.5)))
            else:
                out.append(W.random_multimode(rng, *shapes[i]))
        return out
    count = case.get("count", 1)
    if case["family"] == "qubit":
        if count == 1:
            return [W.two_level(rng.uniform_in(0.2, 2.0), N=case["N1"])]
        amp = rng.uniform_in(0.3, 0.7)
        return [W.two_level(float(w), N=case["N1"], Omega=amp) for w in np.linspace(0.2, 2.0, count)]
    if case["family"] == "spin1":
        return W.spin1_amplitude_set(count, seed=seed, N1=case["N1"], N2=case["N2"])
    if case["family"] == "uneven":
        return [W.random_multimode(rng, D, Ns) for D, Ns in _uneven_shapes(count, case["shapes"], case["nmax"])]
    if case["family"] == "lattice":
        lo = rng.uniform_in(0.2, 0.3)
        return W.lattice_sweep(count, lo=lo, hi=1.0, D=case["D"], N=case["N1"])
    D = case["D"]
    lam = np.array([rng.uniform_in(0.0, 2.0) for _ in range(D)])
    Q = W.haar_unitary(rng, D)
    H0 = (Q * lam[None, :]) @ Q.conj().T
    return [W.Problem(D=D, H0=0.5 * (H0 + H0.conj().T), omegas=[0.5, math.sqrt(2.0) / 2.0, math.sqrt(3.0) / 2.0],
                      Ns=[case["N1"], case["N2"], case["N3"]],
                      couplings=[[W.hermitian_gaussian(rng, D, 0.05)] for _ in range(3)])]


def _times(p, nt):
    return W.time_grid(p, nt)


# ------------------------------------------------------------------ state and pass
class _State:
    pass


_STREAM = []


def _stream():
    """The program's CUDA stream: the library's work and the results' copies are enqueued on it."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0].cuda_stream


def prepare(case, seed):
    s = _State()
    s.case = case
    s.problems = _problems(case, seed)
    s.nt = case["nt"]
    s.ctx = mmf.Context(0, stream=_stream())
    s.ctx.load_tuning(TUNING)
    s.precision = PRECISION[case["precision"]]
    s.systems = [mmf.System(s.ctx, p) for p in s.problems]
    s.t = [_times(p, s.nt) for p in s.problems]
    if case["kind"] == "batch":
        s.batch = mmf.Batch(s.ctx, s.systems, s.precision, s.nt)
        s.batch.set_times(0.0, np.stack(s.t))
        if case["graph"]:
            s.batch.graph(True)
        s.E = torch.zeros(s.batch.nE, dtype=torch.float64, device="cuda")
        s.U = torch.zeros(max(s.batch.nU, 1), dtype=torch.complex128, device="cuda")
        s.P = torch.zeros(s.batch.nP, dtype=torch.float64, device="cuda")
        k = _first(case, s.problems)
        more = k < len(s.problems)
        s.cut = [s.batch.offE[k] if more else s.batch.nE, s.batch.offU[k] if more else s.batch.nU,
                 s.batch.offP[k] if more else s.batch.nP]
    elif case["kind"] == "evolve":
        s.systems[0].build(s.precision)
        s.systems[0].diagonalise()
        s.t_dev = torch.from_numpy(s.t[0]).cuda()
        torch.cuda.synchronize()  # the times are read on the program's stream
        s.U = torch.zeros((s.nt, s.systems[0].D, s.systems[0].D), dtype=torch.complex128, device="cuda")
        # the plan for this number of times
        s.systems[0].time_evolution_dev(0.0, s.nt, s.t_dev.data_ptr(), s.U.data_ptr(),
                                        _stream())
    elif case["kind"] == "serve":
        s.server = mmf.Server(s.ctx, slots=4, max_batch=16, precision=s.precision)
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "sequence":
        y = s.systems[0]
        y.build(s.precision)
        y.diagonalise()
        return {"E": y.quasienergies(), "U": y.time_evolution(s.t[0]), "P": y.transition_avg()}
    stream = _stream()
    if kind == "batch":
        s.batch.upload()
        s.batch.run()
        if s.nt == 0:  # a spectrum
            s.batch.results_dev(s.E.data_ptr(), 0, 0, stream)
            return {"first": {"E": s.E[:s.cut[0]]}, "rest": {"E": s.E[s.cut[0]:]}}
        s.batch.results_dev(s.E.data_ptr(), s.U.data_ptr(), s.P.data_ptr(), stream)
        return {"first": {"E": s.E[:s.cut[0]], "U": s.U[:s.cut[1]], "P": s.P[:s.cut[2]]},
                "rest": {"E": s.E[s.cut[0]:], "U": s.U[s.cut[1]:], "P": s.P[s.cut[2]:]}}
    if kind == "evolve":
        s.systems[0].time_evolution_dev(0.0, s.nt, s.t_dev.data_ptr(), s.U.data_ptr(), stream)
        return {"U": s.U}
    tickets = [s.server.submit(y, t) for y, t in zip(s.systems, s.t)]
    got = [s.server.wait(k) for k in tickets]
    k = _first(s.case, s.problems)
    return {"first": _packed(got[:k]), "rest": _packed(got[k:])}


def _packed(results):
    """E, U, Pbar of several systems one after another."""
    if not results:
        return {"E": np.zeros(0), "U": np.zeros(0, dtype=np.complex128), "P": np.zeros(0)}
    return {"E": np.concatenate([r[0].ravel() for r in results]),
            "U": np.concatenate([r[1].ravel() for r in results]),
            "P": np.concatenate([r[2].ravel() for r in results])}


# ------------------------------------------------------------------ what a pass cannot do without
def _band(p):
    """Half-bandwidth of H_F for the couplings of these families (harmonic 1)."""
    b, S = 1, 1
    i, j = np.nonzero(p.H0)
    if i.size:
        b = max(b, int(np.abs(i - j).max()))
    for N, cl in zip(p.Ns, p.couplings):
        if N > 0:
            i, j = np.nonzero(cl[0])
            if i.size:
                b = max(b, p.D * S + int((j - i).max()))
        S *= 2 * N + 1
    return b


def work(case):
    """Inputs (coefficients, times) read and results (E, U, Pbar) written once; real floating-point
    operations: the reduction of H_F to tridiagonal form (on its band where that is less), the n
    eigenvectors from it, and the Fourier sums of U."""
    nbytes = flops = 0.0
    for p in _problems(case, 1):
        n, nt = p.n, case["nt"]
        nbytes += 16 * p.D ** 2 * (1 + sum(p.nharm())) + 8 * nt + 16 * nt * p.D ** 2
        flops += 8.0 * nt * n * n
        if case["kind"] == "evolve":
            nbytes += 16.0 * n * n + 8 * n
        else:
            nbytes += 8 * n + 8 * p.D ** 2
            flops += min(16.0 / 3.0 * n ** 3, 24.0 * n * n * _band(p)) + 8.0 * n ** 3
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ the results in 64 bits
EXACT_N3 = 2.5e10  # sum of n^3 of the systems whose results `exact` gives, beyond the first system
EXACT_ONE = 6000   # largest single system


def _first(case, problems):
    """How many systems, from the first on, `exact` gives results for."""
    total, k = 0.0, 0
    for p in problems:
        total += float(p.n) ** 3
        if k and total > EXACT_N3:
            break
        k += 1
    return k


def _floquet(p):
    """Dense H_F (mode 1 innermost, first block n = -N): diagonal blocks H0 - (n.w) 1, block (m + h,
    m) of mode l coupled by V^{l,h} above the diagonal and its conjugate transpose below."""
    n, D, M = p.n, p.D, p.M
    H = torch.zeros((M, D, M, D), dtype=torch.complex128)
    widths = [2 * N + 1 for N in p.Ns]
    H0 = torch.from_numpy(np.ascontiguousarray(p.H0.astype(np.complex128)))
    strides = [math.prod(widths[:l]) for l in range(len(widths))]
    for b in range(M):
        nv = [(b // S) % w - N for S, w, N in zip(strides, widths, p.Ns)]
        H[b, :, b, :] = H0 - sum(k * om for k, om in zip(nv, p.omegas)) * torch.eye(D, dtype=torch.complex128)
        for l, cl in enumerate(p.couplings):
            for h, V in enumerate(cl, start=1):
                if nv[l] + h <= p.Ns[l]:
                    c = b + h * strides[l]
                    Vt = torch.from_numpy(np.ascontiguousarray(V.astype(np.complex128)))
                    H[b, :, c, :] += Vt
                    H[c, :, b, :] += Vt.conj().T
    return H.reshape(n, n)


def _solve(p, t):
    H = _floquet(p)
    if p.n > 160:
        H = H.cuda()
    E, Z = torch.linalg.eigh(H)
    n, D, M = p.n, p.D, p.M
    Z3 = Z.reshape(M, D, n)
    widths = [2 * N + 1 for N in p.Ns]
    strides = [math.prod(widths[:l]) for l in range(len(widths))]
    ndotw = np.zeros(M)
    b0 = sum(N * S for N, S in zip(p.Ns, strides))
    for b in range(M):
        ndotw[b] = sum(((b // S) % w - N) * om for S, w, N, om in zip(strides, widths, p.Ns, p.omegas))
    tt = torch.from_numpy(np.asarray(t)).to(Z.device)
    nw = torch.from_numpy(ndotw).to(Z.device)
    Z0 = Z3[b0]                                         # <i, 0 | lambda>
    U = torch.zeros((len(t), D, D), dtype=torch.complex128, device=Z.device)
    for j in range(D):
        F = torch.polar(torch.ones((len(t), M), dtype=torch.float64, device=Z.device), -tt[:, None] * nw[None, :])
        Phi = F @ Z3[:, j, :]                           # sum_n e^{-i n.w t} <j, n | lambda>
        Phi = Phi * torch.polar(torch.ones((len(t), n), dtype=torch.float64, device=Z.device), -tt[:, None] * E[None, :])
        U[:, j, :] = Phi @ Z0.conj().T
    # time average: consecutive eigenvalues closer than 1e-8 max|E| are one degenerate cluster
    gap = (E[1:] - E[:-1]) >= 1e-8 * E.abs().max()
    cid = torch.cat([torch.zeros(1, dtype=torch.int64, device=Z.device), gap.to(torch.int64).cumsum(0)])
    P = torch.zeros((D, D), dtype=torch.float64, device=Z.device)
    for i in range(D):
        for j in range(D):
            A = torch.zeros((M, int(cid[-1]) + 1), dtype=torch.complex128, device=Z.device)
            A.index_add_(1, cid, Z3[:, j, :] * Z0[i].conj()[None, :])
            P[i, j] = A.abs().square().sum()
    return E.cpu().numpy(), U.cpu().numpy(), P.cpu().numpy()


def exact(case, seed):
    problems = _problems(case, seed)
    if max(p.n for p in problems[:1]) > EXACT_ONE:
        return None
    k = _first(case, problems)
    got = []
    for p in problems[:k]:
        if case["nt"] == 0:
            H = _floquet(p)
            got.append((torch.linalg.eigvalsh(H.cuda()).cpu().numpy(), None, None))
        else:
            got.append(_solve(p, _times(p, case["nt"])))
    if case["kind"] == "sequence":
        return {"E": got[0][0], "U": got[0][1], "P": got[0][2]}
    if case["kind"] == "evolve":
        return {"U": got[0][1]}
    if case["nt"] == 0:
        return {"first": {"E": np.concatenate([g[0] for g in got])}, "rest": {"E": None}}
    return {"first": _packed(got), "rest": {"E": None, "U": None, "P": None}}
