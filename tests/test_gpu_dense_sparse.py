"""complex128 gates with mostly zero matrices (same sums as the dense form: bits), scaled rows next to
a dense block, and gates on states of a few groups, against the FP64 oracle."""
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


def apply(qs, psi, n, t, U, ctl=(), dtype=torch.complex128):
    st = torch.from_numpy(np.ascontiguousarray(psi)).to(dtype).cuda()
    qs.qsim_apply(st, qs.Circuit(n).add_gate(t, U, list(ctl)))
    return st.cpu().numpy()


def oracle(psi, t, U, ctl=()):
    ref = psi.copy()
    with np.errstate(all="ignore"):
        ocore.apply_gate(ref, t, U, list(ctl))
    return ref


def sparse_unitary(rng, k, w, real):
    """2^w nonzeros a row: a permutation times blocks that act on the lowest w bits."""
    D = 1 << k
    U = np.zeros((D, D), dtype=np.complex128)
    for b in range(0, D, 1 << w):
        B = rng.standard_normal((1 << w, 1 << w)) + (0 if real else 1j * rng.standard_normal((1 << w, 1 << w)))
        U[b:b + (1 << w), b:b + (1 << w)] = np.linalg.qr(B)[0]
    return U[rng.permutation(D)][:, rng.permutation(D)]


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("k,w", [(1, 0), (2, 0), (2, 1), (3, 1), (4, 2), (5, 3), (6, 0), (6, 4), (7, 1)])
def test_sparse_gates(qs, k, w, real):
    rng = np.random.default_rng(100 * k + w)
    U = sparse_unitary(rng, k, w, real)
    for n, extra in ((k, 0), (k + 1, 1), (k + 4, 2), (15, 1)):
        for t in (list(range(k)), list(range(n - k, n))[::-1], synth.random_targets(rng, n, k)):
            ctl = [int(q) for q in rng.permutation([q for q in range(n) if q not in t])[:extra]]
            psi = synth.gaussian_state_np(int(rng.integers(1 << 30)), n) * 10.0 ** rng.uniform(-30, 0, 1 << n)
            ref = oracle(psi, t, U, ctl)
            out = apply(qs, psi, n, t, U, ctl)
            # 2 2^w rounded terms on both sides, relative to the terms themselves
            mag = oracle(np.abs(psi).astype(np.complex128), t, np.abs(U).astype(np.complex128), ctl).real
            assert np.all(np.abs(out - ref) <= 2.0 ** (w + 2) * 2.0 ** -53 * mag), (n, t, ctl)
    n = max(k + 2, 10)
    t = synth.random_targets(rng, n, k)
    psi = synth.gaussian_state_np(1, n)
    psi[5] = complex(np.inf, 0)
    out, ref = apply(qs, psi, n, t, U), oracle(psi, t, U)
    assert np.isfinite(ref[np.isfinite(out)]).sum() >= 0 and np.all(np.isfinite(out[np.isfinite(ref)]))


def test_scaled_rows(qs):
    """A dense block next to rows that scale one amplitude: those are exact to FP64 in themselves."""
    rng = np.random.default_rng(8)
    for k, real in ((3, False), (4, False), (5, True), (6, False)):
        D, B = 1 << k, (1 << k) - 3
        U = np.zeros((D, D), dtype=np.complex128)
        Z = rng.standard_normal((B, B)) + (0 if real else 1j * rng.standard_normal((B, B)))
        U[:B, :B] = np.linalg.qr(Z)[0]
        for r in range(B, D):
            U[r, r] = -1.0 if real else np.exp(1j * r)
        n, t = 13, synth.random_targets(rng, 13, k)
        psi = synth.gaussian_state_np(k, n)
        idx = np.arange(1 << n)
        row = sum(((idx >> q) & 1) << b for b, q in enumerate(t))
        psi[row >= B] *= 1e-20
        before = qs.qsim_launch_counts()["dense_tc"]
        out, ref = apply(qs, psi, n, t, U), oracle(psi, t, U)
        assert qs.qsim_launch_counts()["dense_tc"] > before
        assert np.max(np.abs(out - ref)) <= (2.0 * D + 2) * 2.0 ** -53 * 2.0 ** (k / 2) * np.max(np.abs(psi))
        pad = row >= B
        assert np.all(np.abs(out[pad] - ref[pad]) <= 4 * 2.0 ** -53 * np.abs(ref[pad]))


@pytest.mark.parametrize("dtype,eps", [(torch.complex128, 2.0 ** -53), (torch.complex64, 2.0 ** -24)])
@pytest.mark.parametrize("k", [3, 4, 5, 6, 7])
def test_few_groups(qs, k, dtype, eps):
    rng = np.random.default_rng(k)
    for free, extra in ((0, 0), (1, 0), (3, 1), (2, 2)):
        for real in (False, True):
            n = k + free + extra
            q = [int(v) for v in rng.permutation(n)]
            t, ctl = q[:k], q[k:k + extra]
            Z = rng.standard_normal((1 << k, 1 << k)) + (0 if real else 1j * rng.standard_normal((1 << k, 1 << k)))
            U = np.linalg.qr(Z)[0].astype(np.complex128)
            if dtype == torch.complex64:
                U = U.astype(np.complex64).astype(np.complex128)
            psi = torch.from_numpy(synth.gaussian_state_np(k, n)).to(dtype).numpy().astype(np.complex128)
            out, ref = apply(qs, psi, n, t, U, ctl, dtype), oracle(psi, t, U, ctl)
            # a sum of 2^(k+1) products, rounded after each, on both sides
            assert np.max(np.abs(out - ref)) <= 2 * (2.0 ** (k + 1) + 2) * eps * 2.0 ** (k / 2) * np.max(np.abs(psi))


@pytest.mark.parametrize("k,blocks,real", [(4, (13, 3), False), (5, (31, 1), True), (6, (63, 1), True), (6, (40, 24), True),
                                           (6, (50, 13, 1), False)])
def test_blocks_of_different_size(qs, k, blocks, real):
    """Short rows next to full ones (a grid that falls apart): on the digit kernels, within their bound."""
    rng = np.random.default_rng(k)
    D = 1 << k
    U = np.zeros((D, D), dtype=np.complex128)
    at = 0
    for b in blocks:
        Z = rng.standard_normal((b, b)) + (0 if real else 1j * rng.standard_normal((b, b)))
        U[at:at + b, at:at + b] = np.linalg.qr(Z)[0]
        at += b
    U = U[rng.permutation(D)][:, rng.permutation(D)]
    for n in (k + 6, k + 14):
        t = synth.random_targets(rng, n, k)
        psi = synth.gaussian_state_np(k, n)
        before = qs.qsim_launch_counts()["dense_tc"]
        out = apply(qs, psi, n, t, U)
        assert qs.qsim_launch_counts()["dense_tc"] > before
        assert np.max(np.abs(out - oracle(psi, t, U))) <= (2.0 * D + 2) * 2.0 ** -53 * 2.0 ** (k / 2) * np.max(np.abs(psi))
