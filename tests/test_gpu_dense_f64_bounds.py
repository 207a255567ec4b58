"""complex128 gates amplitude by amplitude: each output within the bound of an FP64 sum of its own terms.

A sum of n products in FP64, in any order, is within n 2^-53 sum |u_rc| |x_c| of the exact value (n = 2 2^k real products
per part; one more rounding each for the result).  Both the gate and the oracle are held to that bound, so they may
differ by twice as much, whatever other amplitudes the group or the state holds.
"""
import numpy as np
import pytest
import torch

import synth
from oracle import core as ocore

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs(cuda_device):
    from paper_2402_08136_gb300 import build
    build.build()
    import paper_2402_08136_gb300 as q
    return q


def check(qs, psi, n, t, U, ctl=(), terms=None):
    """terms: products per part of each row, where a row has fewer than 2 2^k."""
    psi = np.ascontiguousarray(psi, dtype=np.complex128)
    ref, mag = psi.copy(), np.abs(psi).astype(np.complex128)
    ocore.apply_gate(ref, t, U, list(ctl))
    ocore.apply_gate(mag, t, np.abs(U).astype(np.complex128), list(ctl))
    st = torch.from_numpy(psi).cuda()
    qs.qsim_apply(st, qs.Circuit(n).add_gate(t, U, list(ctl)))
    out = st.cpu().numpy()
    assert qs.qsim_device_status() == 0
    if terms is None:
        m = 2.0 * len(U)
    else:
        m = np.asarray(terms, dtype=float)[rows(n, t)]
    worst = np.max(np.abs(out - ref) / np.maximum(2 * (m + 1) * 2.0 ** -53 * mag.real, 1e-300))
    assert worst <= 1, (n, t, worst)


def rows(n, t):
    idx = np.arange(1 << n)
    return sum(((idx >> q) & 1) << b for b, q in enumerate(t))


def haar(rng, d, real=False):
    if not real:
        return synth.haar_unitary(rng, d)
    return np.linalg.qr(rng.standard_normal((d, d)))[0].astype(np.complex128)


# (targets, qubits): warp-level digit kernels, and from 4 targets on the tcgen05 ones
SIZES = [(1, 12), (2, 12), (3, 12), (4, 12), (4, 18), (5, 13), (5, 19), (6, 13), (6, 18), (6, 19)]


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("k,n", [s for s in SIZES if s[0] >= 2])
def test_controlled_gates_as_dense_ones(qs, k, n, real):
    """The lower half of the rows only scale their amplitude; that half is 1e12 times the other one, or the other way
    round, or is not finite."""
    rng = np.random.default_rng(10 * k + n)
    D = 1 << k
    for scale in (1e-12, 1e12):
        for phase in (1.0, -1.0 if real else np.exp(0.7j)):
            U = np.eye(D, dtype=np.complex128) * phase
            U[D // 2:, D // 2:] = haar(rng, D // 2, real)
            for t in (list(range(k)), synth.random_targets(rng, n, k)):
                psi = synth.gaussian_state_np(k, n)
                psi[rows(n, t) >= D // 2] *= scale
                check(qs, psi, n, t, U)
    psi = synth.gaussian_state_np(k, n)
    t = synth.random_targets(rng, n, k)
    idle = np.flatnonzero(rows(n, t) < D // 2)
    psi[idle[5]], psi[idle[-1]] = np.inf, complex(0, np.nan)
    st = torch.from_numpy(psi).cuda()
    qs.qsim_apply(st, qs.Circuit(n).add_gate(t, U))
    out = st.cpu().numpy()
    hit = ~np.isfinite(out)
    # 0 * inf: every row of the two groups is not finite, as in a plain sum (for a real U in the part of the value)
    same = np.isin(np.arange(1 << n) & ~sum(1 << q for q in t), [i & ~sum(1 << q for q in t) for i in (idle[5], idle[-1])])
    assert np.array_equal(hit, same)


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("k,n", SIZES)
def test_small_angles(qs, k, n, real):
    """Gates close to the identity, on amplitudes of one size and on ones that differ by 1e12 and more inside a group:
    the small outputs come from small entries times large amplitudes."""
    rng = np.random.default_rng(100 * k + n + real)
    D = 1 << k
    for angle in (1e-3, 1e-7, 1e-10, 1e-17):
        Z = rng.standard_normal((D, D)) + (0 if real else 1j * rng.standard_normal((D, D)))
        U = np.eye(D) + angle * (Z - Z.conj().T)
        for what in ("even", "one", "wide"):
            psi = synth.gaussian_state_np(k, n)
            t = synth.random_targets(rng, n, k)
            if what == "one":  # one amplitude of every group
                psi[rows(n, t) != D // 2] = 0
            elif what == "wide":
                psi *= 10.0 ** rng.uniform(-20, 0, 1 << n)
            check(qs, psi, n, t, U.astype(np.complex128))


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("k,n", SIZES)
def test_mixed_scales(qs, k, n, real):
    """Dense gates, and gates with rows and columns of very different size, on states whose amplitudes differ by target
    index, by group or at random."""
    rng = np.random.default_rng(1000 * k + n + real)
    D = 1 << k
    for gate in ("dense", "rows", "columns"):
        U = haar(rng, D, real)
        if gate == "rows":
            U = U * 10.0 ** rng.uniform(-12, 0, D)[:, None]
        elif gate == "columns":
            U = U * 10.0 ** rng.uniform(-12, 0, D)[None, :]
        for what in ("index", "group", "any", "half"):
            t = synth.random_targets(rng, n, k)
            psi = synth.gaussian_state_np(k, n)
            if what == "index":
                psi *= (10.0 ** rng.uniform(-12, 0, D))[rows(n, t)]
            elif what == "group":
                psi *= (10.0 ** rng.uniform(-60, 60, 1 << n))[np.arange(1 << n) & ~sum(1 << q for q in t)]
            elif what == "any":
                psi *= 10.0 ** rng.uniform(-30, 0, 1 << n)
            else:
                psi[rows(n, t) % 2 == 0] *= 1e-14
            check(qs, psi, n, t, U)


@pytest.mark.parametrize("k,blocks,real", [(2, (3, 1), False), (3, (7, 1), False), (3, (6, 1, 1), True), (4, (13, 3), False),
                                           (4, (14, 1, 1), False), (5, (31, 1), True), (5, (30, 2), False), (6, (63, 1), True),
                                           (6, (62, 2), True), (6, (40, 24), True), (6, (50, 13, 1), False),
                                           (6, (60, 1, 1, 1, 1), False)])
def test_short_rows(qs, k, blocks, real):
    """Short rows next to full ones: a sum of few terms is held to its own few terms, a row of one entry to one product,
    also where another block's amplitudes are 1e12 times as large."""
    rng = np.random.default_rng(k + len(blocks))
    D = 1 << k
    U = np.zeros((D, D), dtype=np.complex128)
    block = np.zeros(D, dtype=int)
    at = 0
    for i, b in enumerate(blocks):
        U[at:at + b, at:at + b] = haar(rng, b, real)
        block[at:at + b] = i
        at += b
    col = rng.permutation(D)
    U, block = U[rng.permutation(D)][:, col], block[col]
    terms = 2 * np.count_nonzero(U, axis=1)
    for n, ctl in ((k + 7, 0), (k + 9, 1), (k + 14, 0)):
        for scale in (1.0, 1e-12, 1e12):
            q = [int(v) for v in rng.permutation(n)]
            psi = synth.gaussian_state_np(k, n)
            psi[(block == 0)[rows(n, q[:k])]] *= scale
            check(qs, psi, n, q[:k], U, q[k:k + ctl], terms)


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("k,n", [s for s in SIZES if s[0] >= 4])
def test_rows_that_hardly_mix(qs, k, n, real):
    """One or two rows with a single large entry, on the diagonal or off it, and rounding noise beside it (1e-17 down to
    1e-50, some zeros), as an eigensolver leaves it for a part of the system that stands alone; also all rows (a gate
    next to a diagonal one)."""
    rng = np.random.default_rng(7 * k + n + real)
    D = 1 << k
    for alone in (1, 2, D):
        for moved in (False, True):
            M = D - alone
            U = np.zeros((D, D), dtype=np.complex128)
            if M:
                U[:M, :M] = haar(rng, M, real)
            for i in range(M, D):
                U[i, i] = -1.0 if real else np.exp(1j * i)
            noise = 10.0 ** -rng.uniform(16.5, 50, (D, D)) * (rng.random((D, D)) < 0.9)
            noise = noise * (rng.choice([-1.0, 1.0], (D, D)) if real else np.exp(1j * rng.uniform(0, 6, (D, D))))
            edge = np.ones((D, D), dtype=bool)
            edge[:M, :M] = False
            edge[np.arange(D), np.arange(D)] = False
            U[edge] = noise[edge]
            if moved:
                U = U[rng.permutation(D)][:, rng.permutation(D)]
            for what in ("even", "far", "near", "wide", "one"):
                t = synth.random_targets(rng, n, k)
                psi = synth.gaussian_state_np(k, n)
                col = np.argmax(np.abs(U), axis=1) if alone == D else np.flatnonzero((np.abs(U) > 1e-9).sum(0) == 1)
                hit = np.isin(rows(n, t), col)
                if what == "far":
                    psi[hit] *= 1e-30
                elif what == "near":
                    psi[~hit] *= 1e-19
                elif what == "wide":
                    psi *= 10.0 ** rng.uniform(-25, 0, 1 << n)
                elif what == "one":
                    psi[rows(n, t) != col[0]] = 0
                check(qs, psi, n, t, U)


@pytest.mark.parametrize("n,ctl,digits", [(17, 0, True), (18, 0, False), (18, 1, True), (19, 1, False)])
def test_real_single_targets(qs, n, ctl, digits):
    """Both sides of the rule that leaves real 1-target gates to FP64 (2^18 amplitudes, controls apart)."""
    rng = np.random.default_rng(n + ctl)
    for U in (np.array([[1, 1], [1, -1]]) / 2 ** 0.5, haar(rng, 2, True)):
        q = [int(v) for v in rng.permutation(n)]
        before = qs.qsim_launch_counts()["dense_tc"]
        check(qs, synth.gaussian_state_np(n, n), n, q[:1], U.astype(np.complex128), q[1:1 + ctl])
        assert (qs.qsim_launch_counts()["dense_tc"] > before) == digits
