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
