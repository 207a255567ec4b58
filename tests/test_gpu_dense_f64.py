"""complex128 dense gates as digit products on the tensor cores against the FP64 oracle.

Tolerance per amplitude: the oracle adds 2 2^k products per real, each sum rounded to 53 bits, so it
is within 2^(k+1) 2^-53 sum_c |u_rc| |x_c| of the exact value, and sum_c |u_rc| |x_c| <= |x|_2 over
the group <= 2^(k/2) max |x| for a unitary U; the digit form is within 2^-56 of the group's scale
(at most twice its largest real) per sqrt(2^k) terms, below that, plus its one rounding.
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


def tolerance(k, x):
    return (2.0 ** (k + 1) + 2) * 2.0 ** -53 * 2.0 ** (k / 2) * np.max(np.abs(x))


def apply(qs, psi, n, t, U, ctl=()):
    """The gate's result and whether it ran on the tensor cores."""
    st = torch.from_numpy(np.ascontiguousarray(psi)).cuda()
    before = qs.qsim_launch_counts()["dense_tc"]
    qs.qsim_apply(st, qs.Circuit(n).add_gate(t, U, list(ctl)))
    torch.cuda.synchronize()
    return st.cpu().numpy(), qs.qsim_launch_counts()["dense_tc"] > before


def unitary(rng, k, real):
    if not real:
        return synth.haar_unitary(rng, 1 << k)
    return np.linalg.qr(rng.standard_normal((1 << k, 1 << k)))[0].astype(np.complex128)


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6])
def test_widths_sizes_targets(qs, k, real):
    rng = np.random.default_rng(10 * k + real)
    low = max(3, k) + (2 if real and k >= 4 else 3)  # the smallest state that fills one warp tile
    for n, extra in ((low, 0), (low + 1, 1), (low + 5, 2), (17, 1)):
        for t in (list(range(k)), list(range(n - k, n))[::-1], synth.random_targets(rng, n, k)):
            free = [q for q in range(n) if q not in t]
            ctl = [int(q) for q in rng.permutation(free)[:extra]]
            psi = synth.gaussian_state_np(int(rng.integers(1 << 30)), n)
            U = unitary(rng, k, real)
            ref = psi.copy()
            ocore.apply_gate(ref, t, U, ctl)
            out, tc = apply(qs, psi, n, t, U, ctl)
            assert np.max(np.abs(out - ref)) <= tolerance(k, psi), (n, t, ctl)
            assert tc == (n - len(ctl) >= low)


@pytest.mark.parametrize("k,real", [(1, False), (3, True), (4, False), (5, True), (6, False)])
def test_values_outside_the_fixed_point_range(qs, k, real):
    """Zeros, a wide range inside a group, exponents near the ends, denormals, infinities, NaN."""
    rng = np.random.default_rng(k)
    n = 13
    t = synth.random_targets(rng, n, k)
    U = unitary(rng, k, real)
    base = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    for what in ("zero", "basis", "wide", "1e300", "1e-300", "1e-315", "inf", "nan"):
        psi = base.copy()
        if what == "zero":
            psi[:] = 0
        elif what == "basis":
            psi[:] = 0
            psi[1234] = 1j
        elif what == "wide":
            psi *= 10.0 ** rng.uniform(-30, 0, 1 << n)
        elif what in ("inf", "nan"):
            psi[777] = complex(0.0, float(what))
        else:
            psi *= float(what)
        out, tc = apply(qs, psi, n, t, U)
        assert tc
        ref = psi.copy()
        with np.errstate(all="ignore"):
            ocore.apply_gate(ref, t, U)
        if what in ("inf", "nan"):  # the plain form of a real U leaves the zero imaginary parts out
            hit = ~np.isfinite(out)
            assert hit.any() and np.all(~np.isfinite(ref[hit.nonzero()]))
            fine = np.isfinite(ref)
            assert np.max(np.abs(out[fine] - ref[fine])) <= tolerance(k, base)
        else:
            assert np.max(np.abs(out - ref)) <= max(tolerance(k, psi), 2.0 ** -1073)


def test_identity_rows_and_sparse_gates(qs):
    rng = np.random.default_rng(3)
    n = 12
    psi = synth.gaussian_state_np(5, n)
    # a block next to an identity (a padded eigenvector matrix): identity rows keep their bits
    U = np.eye(64, dtype=np.complex128)
    U[:50, :50] = np.linalg.qr(rng.standard_normal((50, 50)))[0]
    out, tc = apply(qs, psi, n, list(range(6)), U)
    assert tc
    ref = psi.copy()
    ocore.apply_gate(ref, list(range(6)), U)
    assert np.max(np.abs(out - ref)) <= tolerance(6, psi)
    pad = (np.arange(1 << n) & 63) >= 50
    assert np.array_equal(out[pad], psi[pad])
    # a permutation is exact whatever the range of its amplitudes
    psi *= 10.0 ** rng.uniform(-30, 0, 1 << n)
    P = np.roll(np.eye(8), 3, axis=0).astype(np.complex128)
    out, tc = apply(qs, psi, n, [2, 7, 9], P)
    ref = psi.copy()
    ocore.apply_gate(ref, [2, 7, 9], P)
    assert not tc and np.array_equal(out, ref)
