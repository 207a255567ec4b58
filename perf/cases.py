"""The work a user of this simulator has it do, as a list of measurable cases.

Kinds of case (key "kind"):

  gates   dense Haar gates applied one qsim_apply call each (the gate microbenchmark's rule: every
          width 1..kmax equally often, uniformly random distinct targets; some with a control)
  fused   a layered circuit of 1- and 2-qubit gates, fused by qsim_fuse at its default width and
          applied in one call (general circuit simulation)
  hhl     one HHL solve on the full-GPU path: run, then read the solution out.  form "passes":
          structured phase estimation with the QFTs as Fourier passes and the readout sums from
          the run; form "paper": the paper's gate-level circuit; dilate: a non-symmetric system
          through its Hermitian dilation (the Newton-Raphson power-flow step)
  batch   many small HHL systems (N-1 contingencies) in one persistent launch; count 1 is the
          latency path of a single small system
  serve   a burst of independent requests through the serving pool

Sizes are those of this repository's benchmark workloads and tests (7-, 16-, 22- and 27-qubit
solves, 512 contingencies, gates of 1..6 targets, 2..7 data qubits) or lie between them.
"""
import math

import numpy as np
import torch

import paper_2402_08136_gb300 as qs

DTYPES = {"c64": torch.complex64, "c128": torch.complex128}
BYTES = {"c64": 8, "c128": 16}
DEV = "cuda"
STATS = ("p_success", "p_clock0", "norm2", "norm_x")


def listed():
    return [
        # one 4x4 system on the 4-bit clock grid, answer on the host: the latency of the smallest solve
        {"name": "solve7-c128", "kind": "batch", "dtype": "c128", "count": 1, "nb_lo": 2, "nb_hi": 2, "m_lo": 4,
         "m_hi": 4, "form": "paper"},
        # a contingency screening: 512 N-1 systems of 7..16 qubits in one launch
        {"name": "batch512-c64", "kind": "batch", "dtype": "c64", "count": 512, "nb_lo": 2, "nb_hi": 5, "m_lo": 4,
         "m_hi": 10, "form": "passes"},
        # a smaller screening where the answers are wanted in double precision
        {"name": "batch96-c128", "kind": "batch", "dtype": "c128", "count": 96, "nb_lo": 2, "nb_hi": 5, "m_lo": 4,
         "m_hi": 10, "form": "passes"},
        # the gate microbenchmark's rule on a state well above L2, single precision
        {"name": "gates28-c64", "kind": "gates", "dtype": "c64", "n": 28, "kmax": 6, "per_k": 2, "control": False},
        # the same in double precision, on an odd qubit count and with a controlled gate per width
        {"name": "gates25-c128", "kind": "gates", "dtype": "c128", "n": 25, "kmax": 6, "per_k": 2, "control": True},
        # an ordinary circuit on a state that stays in L2
        {"name": "fused22-c64", "kind": "fused", "dtype": "c64", "n": 22, "layers": 4},
        # the same in double precision
        {"name": "fused21-c128", "kind": "fused", "dtype": "c128", "n": 21, "layers": 4},
        # the precision solve: 64x64 system, 20 clock qubits, both precisions
        {"name": "hhl27-c64", "kind": "hhl", "dtype": "c64", "N": 64, "m": 20, "form": "passes", "dilate": False},
        {"name": "hhl27-c128", "kind": "hhl", "dtype": "c128", "N": 64, "m": 20, "form": "passes", "dilate": False},
        # the paper's gate-level circuit, hundreds of short operations, on a padded system
        {"name": "hhl17-paper-c128", "kind": "hhl", "dtype": "c128", "N": 13, "m": 12, "form": "paper", "dilate": False},
        # one Newton step of a power flow: non-symmetric system, dilated to 128x128
        {"name": "hhl22-dilated-c64", "kind": "hhl", "dtype": "c64", "N": 64, "m": 14, "form": "passes", "dilate": True},
        # a burst of requests of mixed size at the serving pool
        {"name": "serve48-c64", "kind": "serve", "dtype": "c64", "count": 48, "n_lo": 8, "n_hi": 20},
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, math.floor(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["gates", "gates", "fused", "fused", "hhl", "hhl", "batch", "serve"])
    dtype = rng.choice(["c64", "c128"])
    if kind == "gates":
        return {"kind": kind, "dtype": dtype, "n": rng.randint(16, 28 if dtype == "c64" else 25), "kmax": rng.randint(2, 6),
                "per_k": rng.randint(1, 2), "control": rng.random() < 0.5}
    if kind == "fused":
        return {"kind": kind, "dtype": dtype, "n": rng.randint(12, 26 if dtype == "c64" else 23), "layers": rng.randint(2, 6)}
    if kind == "hhl":
        dilate = rng.random() < 0.3
        if rng.random() < 0.25:  # gate-level circuits: up to a few hundred operations
            N, m, form, dilate = rng.randint(3, 32), rng.randint(6, 12), "paper", False
        else:
            N, m, form = (rng.randint(9, 64), rng.randint(8, 14), "passes") if dilate else (rng.randint(4, 64), rng.randint(8, 20), "passes")
        return {"kind": kind, "dtype": dtype, "N": N, "m": m, "form": form, "dilate": dilate}
    if kind == "batch":
        nb, m = rng.randint(2, 3), rng.randint(4, 6)
        return {"kind": kind, "dtype": dtype, "count": _log_int(rng, 1, 512 if dtype == "c64" else 192), "nb_lo": nb,
                "nb_hi": rng.randint(nb, 5), "m_lo": m, "m_hi": rng.randint(m, 10), "form": "passes"}
    return {"kind": kind, "dtype": dtype, "count": _log_int(rng, 8, 48), "n_lo": rng.randint(8, 10),
            "n_hi": rng.randint(14, 20 if dtype == "c64" else 18)}


# ----------------------------------------------------------------------------- inputs
def _haar(rng, d):
    # QR of a complex Gaussian matrix with the phases of R's diagonal divided out (Mezzadri 2007)
    q, r = np.linalg.qr(rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d)))
    p = np.diagonal(r)
    return np.ascontiguousarray(q * (p / np.abs(p))[None, :])


def _grid(rng, N):
    """Reduced DC power-flow matrix of a random connected (N+1)-bus grid (average degree 3) and
    random injections: symmetric positive definite, N x N."""
    B = N + 1
    edges = {(int(rng.integers(0, i)), i) for i in range(1, B)}  # a random tree keeps it connected
    want = min(B * (B - 1) // 2, int(math.ceil(1.5 * B)))
    while len(edges) < want:
        a, b = sorted(int(v) for v in rng.integers(0, B, size=2))
        if a != b:
            edges.add((a, b))
    L = np.zeros((B, B))
    for a, b in sorted(edges):
        s = rng.uniform(5.0, 20.0)
        L[a, a] += s
        L[b, b] += s
        L[a, b] -= s
        L[b, a] -= s
    return L[1:, 1:].copy(), rng.standard_normal(N)


def _snap(A, m):
    """The spectrum moved to integers 1..2^m-1: every phase is exact on an m-bit clock."""
    w, V = np.linalg.eigh(A)
    k = np.clip(np.floor(w * ((2 ** m - 1) / w[-1]) + 0.5), 1, 2 ** m - 1)
    A = (V * k) @ V.T
    return 0.5 * (A + A.T)


def _state(case, seed):
    n, dt = case["n"], DTYPES[case["dtype"]]
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    psi = torch.empty(1 << n, dtype=dt, device=DEV)
    torch.view_as_real(psi).normal_(0.0, 2.0 ** (-(n + 1) / 2.0), generator=g)
    return psi


def _gate_list(case, seed):
    """[(targets, U, controls)] of a gates or fused case."""
    rng, n, out = np.random.default_rng([7, seed]), case["n"], []
    if case["kind"] == "gates":
        for k in range(1, case["kmax"] + 1):
            for j in range(case["per_k"]):
                c = 1 if case["control"] and j == 0 else 0
                q = [int(v) for v in rng.choice(n, size=k + c, replace=False)]
                out.append((q[:k], _haar(rng, 2 ** k), q[k:]))
        return out
    for _ in range(case["layers"]):
        out += [([q], _haar(rng, 2), []) for q in range(n)]
        p = [int(v) for v in rng.permutation(n)]
        out += [([p[i], p[i + 1]], _haar(rng, 4), []) for i in range(0, n - 1, 2)]
    return out


def _systems(case, seed):
    """[(A, b, m, t)] of an hhl, batch or serve case (t = 0: chosen by the library)."""
    rng, out = np.random.default_rng([11, seed]), []
    if case["kind"] == "hhl":
        if not case["dilate"]:
            return [(*_grid(rng, case["N"]), case["m"], 0.0)]
        A, b = _grid(rng, case["N"])
        # a power-flow Jacobian is close to symmetric: 10 % of unsymmetric coupling on the lines
        return [(A * (1.0 + 0.1 * rng.standard_normal(A.shape)), b, case["m"], 0.0)]
    sizes = np.random.default_rng(case["count"])  # the mix of sizes belongs to the case, the systems to the seed
    for _ in range(case["count"]):
        if case["kind"] == "serve":
            n = int(sizes.integers(case["n_lo"], case["n_hi"] + 1))
            nb = int(sizes.integers(2, min(6, n - 5) + 1))
            m = n - 1 - nb
        else:
            nb = int(sizes.integers(case["nb_lo"], case["nb_hi"] + 1))
            m = int(sizes.integers(case["m_lo"], case["m_hi"] + 1))
        A, b = _grid(rng, 2 ** nb)
        if case.get("form") == "paper":
            out.append((_snap(A, m), b, m, 2 * math.pi / 2 ** m))
        else:
            out.append((A, b, m, 0.0))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gates":
        circuits = [qs.Circuit(case["n"]).add_gate(t, U, c) for t, U, c in _gate_list(case, seed)]
        return {"kind": kind, "psi": _state(case, seed), "circuits": circuits}
    if kind == "fused":
        c = qs.Circuit(case["n"])
        for t, U, _ in _gate_list(case, seed):
            c.add_gate(t, U)
        return {"kind": kind, "psi": _state(case, seed), "circuits": [qs.qsim_fuse(c)]}
    systems = _systems(case, seed)
    if kind == "serve":
        pool = qs.Pool(1 << 30)
        dt = qs.QSIM_C128 if case["dtype"] == "c128" else qs.QSIM_C64
        return {"kind": kind, "pool": pool, "systems": systems, "dtype": dt}
    opts = dict(structured=True, fft_qft=True) if case["form"] == "passes" else {}
    if case.get("dilate"):
        opts["dilate"] = True
    hs = [qs.hhl_build(A, b, m, t, **opts) for A, b, m, t in systems]
    fused = [qs.qsim_fuse(h.as_circuit(), 3 if kind == "batch" else 4) for h in hs]
    states = [torch.empty(1 << h.info()["n"], dtype=DTYPES[case["dtype"]], device=DEV) for h in hs]
    if kind == "batch":
        return {"kind": kind, "batch": qs.hhl_batch_create(hs, states, fused)}
    sums = torch.empty(qs.QSIM_READOUT_SUMS_DOUBLES, dtype=torch.float64, device=DEV)
    return {"kind": kind, "h": hs[0], "circuit": fused[0], "psi": states[0], "sums": sums, "form": case["form"]}


def run(state):
    kind = state["kind"]
    if kind in ("gates", "fused"):
        for c in state["circuits"]:
            qs.qsim_apply(state["psi"], c)
        return state["psi"]
    if kind == "batch":
        x, st = state["batch"].solve()
        return {"x": x, **{k: st[k] for k in STATS}}
    if kind == "hhl":
        psi, h = state["psi"], state["h"]
        if state["form"] == "passes":
            qs.hhl_run_sums(psi, h, state["sums"], state["circuit"])
            r = qs.hhl_readout_sums(psi, h, state["sums"])
        else:
            qs.hhl_run(psi, h, state["circuit"])
            r = qs.hhl_readout(psi, h)
        return {"psi": psi, "x": r["x"], **{k: r[k] for k in STATS}}
    pool = state["pool"]
    tickets = [pool.submit(A, b, m, dtype=state["dtype"], structured=True) for A, b, m, _ in state["systems"]]
    left = len(tickets)
    while left:
        left -= len(pool.take_completed())
    r = [pool.poll(t) for t in tickets]
    return {"x": np.concatenate([v["x"] for v in r]), **{k: np.array([v[k] for v in r]) for k in STATS}}


# ----------------------------------------------------------------------------- 64-bit results
def _apply_exact(psi, n, targets, U, controls):
    """psi (complex128) after one dense gate: gather each group, multiply, scatter."""
    fix = sorted(targets + controls)
    off = torch.tensor([sum(((c >> b) & 1) << t for b, t in enumerate(targets)) for c in range(1 << len(targets))], device=psi.device)
    Ut = torch.from_numpy(np.ascontiguousarray(U.T)).to(psi.device)
    groups, cm = 1 << (n - len(fix)), sum(1 << q for q in controls)
    step = max(1, (1 << 24) >> len(targets))
    for s in range(0, groups, step):
        g = torch.arange(s, min(groups, s + step), device=psi.device)
        for q in fix:
            g = ((g >> q) << (q + 1)) | (g & ((1 << q) - 1))
        i = (g | cm)[:, None] + off[None, :]
        psi[i] = psi[i] @ Ut


def _spectrum(A, b, m, t, dilate):
    """What the procedure fixes before the circuit: padded eigenpairs, b, t, C, clock values."""
    N, x_off = len(b), 0
    A, b = np.asarray(A, dtype=np.float64), np.asarray(b, dtype=np.float64)
    if dilate:
        Z = np.zeros((N, N))
        A, b, x_off = np.block([[Z, A], [A.T, Z]]), np.concatenate([b, np.zeros(N)]), N
    n = len(b)
    D = 1 << max(1, (n - 1).bit_length())
    lam, V = np.linalg.eigh(A)
    signed, top, low = lam[0] < 0, np.abs(lam).max(), np.abs(lam).min()
    lam, W = np.concatenate([lam, np.full(D - n, top)]), np.eye(D)
    W[:n, :n] = V
    M = 1 << m
    t = t or 2 * math.pi * ((M / 2 if signed else M) - 1.0) / (M * top)
    step = 2 * math.pi / (t * M)
    C = max(1.0, math.floor(low / step * (1 + 1e-9))) * step
    k = np.arange(M, dtype=np.float64)
    k = np.where(k >= M // 2, k - M, k) if signed else k
    r = np.zeros(M)
    r[k != 0] = np.clip(C / step / k[k != 0], -1.0, 1.0)
    nrm = np.linalg.norm(b)
    beta = W.T @ np.concatenate([b / nrm, np.zeros(D - n)])
    return N, x_off, lam, W, beta, t, C, r, nrm


def _phases(x, m):
    """exp(i x c) for c = 0..2^m-1 and every x: products of two tables in extended precision."""
    h = (m + 1) // 2
    pi2 = 2 * np.longdouble("3.14159265358979323846264338327950288")
    tab = []
    for size, scale in ((1 << h, 1), (1 << (m - h), 1 << h)):
        a = np.fmod(np.longdouble(x)[None, :] * np.arange(size, dtype=np.int64).astype(np.longdouble)[:, None] * scale, pi2)
        tab.append(torch.from_numpy(np.exp(1j * a.astype(np.float64))).to(DEV))
    return (tab[1][:, None, :] * tab[0][None, :, :]).reshape(1 << m, -1)


def _solve_exact(A, b, m, t, dilate=False, whole=True):
    """Final state (whole) and readout of one HHL solve, in the eigenbasis of A with torch FFTs."""
    N, x_off, lam, W, beta, t, C, r, nrm = _spectrum(A, b, m, t, dilate)
    M, D = 1 << m, len(lam)
    P = _phases(lam * t, m)
    Wt = torch.from_numpy(W.T.astype(np.complex128)).to(DEV)
    F = torch.fft.fft(P * torch.from_numpy(beta).to(DEV)[None, :], dim=0) / M  # QPE, inverse QFT
    s = torch.from_numpy(r).to(DEV)[:, None]
    c = torch.sqrt((1 - s.abs()) * (1 + s.abs()))
    halves, norms = [], []
    for f in ((c, s) if whole else (s,)):
        Y = torch.fft.ifft(F * f, dim=0) * math.sqrt(M)
        Y.mul_(P.conj())
        if whole:
            Y = Y @ Wt
            w = Y.reshape((M, D))
            for j in range(m):  # Hadamard on clock bit j
                v = w.reshape(M >> (j + 1), 2, 1 << j, D)
                w = torch.stack((v[:, 0] + v[:, 1], v[:, 0] - v[:, 1]), dim=1).mul_(math.sqrt(0.5)).reshape(M, D)
            Y = w
            sl = Y[0]
        else:
            sl = (Y.sum(0) / math.sqrt(M)) @ Wt
        norms.append(float((F * f).abs().square().sum()))
        halves.append(Y.reshape(-1))
    prob, p0 = norms[-1], float(sl.abs().square().sum())
    norm_x = math.sqrt(prob) / C
    x = (sl[x_off:x_off + N] / math.sqrt(p0) * norm_x * nrm).cpu().numpy()
    st = {"p_success": prob, "p_clock0": p0, "norm2": float(F.abs().square().sum()), "norm_x": norm_x}
    return (torch.cat(halves) if whole else None), x, st


def exact(case, seed):
    if case["kind"] in ("gates", "fused"):
        psi = _state(case, seed).to(torch.complex128)
        for t, U, c in _gate_list(case, seed):
            _apply_exact(psi, case["n"], t, U, c)
        return psi
    systems = _systems(case, seed)
    if case["kind"] == "hhl":
        psi, x, st = _solve_exact(*systems[0], dilate=case["dilate"])
        return {"psi": psi, "x": x, **st}
    r = [_solve_exact(*s, whole=False) for s in systems]
    return {"x": np.concatenate([v[1] for v in r]), **{k: np.array([v[2][k] for v in r]) for k in STATS}}


# ----------------------------------------------------------------------------- work
def work(case):
    """Each call's input read once and its output written once; multiply-adds of the dense gates
    and 5 N log2 N for each Fourier transform."""
    S, kind = BYTES[case["dtype"]], case["kind"]
    if kind == "gates":
        amps = 2.0 ** case["n"]
        share = [0.5 if case["control"] and j == 0 else 1.0 for j in range(case["per_k"])]
        return {"bytes": 2 * S * amps * sum(share) * case["kmax"],
                "flops": 8 * amps * sum(share) * sum(2 ** k for k in range(1, case["kmax"] + 1))}
    if kind == "fused":
        amps, n = 2.0 ** case["n"], case["n"]
        return {"bytes": 2 * S * amps, "flops": case["layers"] * amps * 8 * (2 * n + 4 * (n // 2))}
    total = {"bytes": 0.0, "flops": 0.0}
    if kind == "hhl":
        sizes = [(max(1, (case["N"] * (2 if case["dilate"] else 1) - 1).bit_length()), case["m"])]
    else:  # the mean size of the case, times its count
        if kind == "serve":
            ns = range(case["n_lo"], case["n_hi"] + 1)
            sizes = [(min(4, n - 5), n - 1 - min(4, n - 5)) for n in ns]
        else:
            sizes = [(nb, m) for nb in range(case["nb_lo"], case["nb_hi"] + 1) for m in range(case["m_lo"], case["m_hi"] + 1)]
    for nb, m in sizes:
        amps = 2.0 ** (nb + m + 1)
        # small systems hand back x alone; a full solve also leaves its final state
        total["bytes"] += (S * amps if kind == "hhl" else 16.0 * 2 ** nb) + 16.0 * 4 ** nb
        total["flops"] += amps * (4 * 2 ** nb + 5 * m + 5 * m + 2 * m + 16)
    many = 1.0 if kind == "hhl" else case["count"] / len(sizes)
    return {k: v * many for k, v in total.items()}
