"""Wide complex128 gates on the tcgen05 kernels against the FP64 oracle (same arithmetic and tolerance as
the warp-level digit kernels, see test_gpu_dense_f64.py), at the smallest state that takes them, with every
kind of target set, controls, scaled rows, and tiles that leave the fixed-point range."""
import numpy as np
import pytest
import torch

import synth
from oracle import core as ocore

pytestmark = pytest.mark.gpu

# (targets, real U, groups of a tile, log2)
FORMS = [(4, False, 7), (5, False, 7), (6, True, 6), (6, False, 6)]


@pytest.fixture(scope="module")
def qs(cuda_device):
    from paper_2402_08136_gb300 import build
    build.build()
    import paper_2402_08136_gb300 as q
    return q


def tolerance(k, x):
    return (2.0 ** (k + 1) + 2) * 2.0 ** -53 * 2.0 ** (k / 2) * np.max(np.abs(x))


def unitary(rng, k, real):
    if not real:
        return synth.haar_unitary(rng, 1 << k)
    return np.linalg.qr(rng.standard_normal((1 << k, 1 << k)))[0].astype(np.complex128)


def apply(qs, psi, n, t, U, ctl=()):
    st = torch.from_numpy(np.ascontiguousarray(psi)).cuda()
    before = qs.qsim_launch_counts()["dense_tc"]
    qs.qsim_apply(st, qs.Circuit(n).add_gate(t, U, list(ctl)))
    out = st.cpu().numpy()
    assert qs.qsim_launch_counts()["dense_tc"] == before + 1
    assert qs.qsim_device_status() == 0
    return out


def oracle(psi, t, U, ctl=()):
    ref = psi.copy()
    with np.errstate(all="ignore"):
        ocore.apply_gate(ref, t, U, list(ctl))
    return ref


@pytest.mark.parametrize("k,real,gb", FORMS)
def test_targets_sizes(qs, k, real, gb):
    rng = np.random.default_rng(10 * k + real)
    for extra, more in ((0, 0), (1, 0), (2, 1), (0, 2)):  # controls, qubits beyond 2^7 tiles
        n = k + gb + 7 + extra + more
        for t in (list(range(k)), list(range(1, k + 1)), list(range(n - k, n))[::-1], synth.random_targets(rng, n, k)):
            ctl = [int(q) for q in rng.permutation([q for q in range(n) if q not in t])[:extra]]
            psi = synth.gaussian_state_np(int(rng.integers(1 << 30)), n)
            U = unitary(rng, k, real)
            assert np.max(np.abs(apply(qs, psi, n, t, U, ctl) - oracle(psi, t, U, ctl))) <= tolerance(k, psi), (n, t, ctl)


@pytest.mark.parametrize("k,real,gb", FORMS)
def test_values(qs, k, real, gb):
    rng = np.random.default_rng(k)
    n = k + gb + 7
    t = synth.random_targets(rng, n, k)
    U = unitary(rng, k, real)
    base = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    for what in ("zero", "basis", "wide", "1e-300", "1e-315", "inf", "nan"):
        psi = base.copy()
        if what == "zero":
            psi[:] = 0
        elif what == "basis":
            psi[:] = 0
            psi[1234] = 1j
        elif what == "wide":
            psi *= 10.0 ** rng.uniform(-30, 0, 1 << n)
        elif what in ("inf", "nan"):
            psi[[777, 1 << (n - 1)]] = complex(0.0, float(what))
        else:
            psi *= float(what)
        out, ref = apply(qs, psi, n, t, U), oracle(psi, t, U)
        if what in ("inf", "nan"):  # the plain form of a real U leaves the zero imaginary parts out
            hit = ~np.isfinite(out)
            assert hit.any() and np.all(~np.isfinite(ref[hit]))
            fine = np.isfinite(ref)
            assert np.max(np.abs(out[fine] - ref[fine])) <= tolerance(k, base)
        else:
            assert np.max(np.abs(out - ref)) <= max(tolerance(k, psi), 2.0 ** -1073), what


@pytest.mark.parametrize("k,real,gb", FORMS)
def test_scaled_rows(qs, k, real, gb):
    rng = np.random.default_rng(k + 50)
    D, B = 1 << k, (1 << k) - 5
    U = np.zeros((D, D), dtype=np.complex128)
    U[:B, :B] = np.linalg.qr(rng.standard_normal((B, B)) + (0 if real else 1j * rng.standard_normal((B, B))))[0]
    for r in range(B, D):
        U[r, r] = -1.0 if real else np.exp(1j * r)
    n = k + gb + 7
    for t in (list(range(k)), synth.random_targets(rng, n, k)):
        psi = synth.gaussian_state_np(k, n)
        idx = np.arange(1 << n)
        pad = sum(((idx >> q) & 1) << b for b, q in enumerate(t)) >= B
        psi[pad] *= 1e-20
        out, ref = apply(qs, psi, n, t, U), oracle(psi, t, U)
        assert np.max(np.abs(out - ref)) <= tolerance(k, psi)
        assert np.all(np.abs(out[pad] - ref[pad]) <= 4 * 2.0 ** -53 * np.abs(ref[pad]))
