"""complex128 Fourier and Walsh-Hadamard passes in fixed point against numpy's FFT.

Tolerance: a K-qubit transform in FP64 by radix-2 steps is within about 6 K 2^-53 |x|_2 of the exact
result per column (numpy's, and the pass's FP64 form), the fixed-point form within a few units of
2^-56 of the column's largest value; twiddle factors add two roundings.  Per amplitude, with |x|_2 <=
2^(K/2) max |x| over a column: 8 (K + 2) 2^-53 2^(K/2) max |x|.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs(cuda_device):
    from paper_2402_08136_gb300 import build
    build.build()
    import paper_2402_08136_gb300 as q
    return q


def columns(n, f0, K):
    i = np.arange(1 << n)
    rest = i[((i >> f0) & ((1 << K) - 1)) == 0]
    return rest, rest[:, None] | (np.arange(1 << K)[None, :] << f0)


def reference(psi, n, f0, K, kind, src):
    rest, idx = columns(n, f0, K)
    x = psi[idx]
    if kind == "walsh":
        y = x
        for b in range(K):
            v = y.reshape(len(rest), -1, 2, 1 << b)
            y = np.stack((v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]), axis=2).reshape(len(rest), -1)
        y = y * 2.0 ** (-K / 2)
    else:
        sign = 1 if kind == "dft+" else -1
        y = (np.fft.ifft(x, axis=1) * 2.0 ** K if sign > 0 else np.fft.fft(x, axis=1)) * 2.0 ** (-K / 2)
        if src:
            w = np.zeros(len(rest), dtype=np.int64)
            for j, q in enumerate(src):
                w |= ((rest >> q) & 1) << j
            N = 1 << (K + len(src))
            y = y * np.exp(sign * 2j * np.pi * ((w[:, None] * np.arange(1 << K)[None, :]) % N) / N)
    out = psi.copy()
    out[idx] = y
    return out


def run(qs, psi, n, f0, K, kind, src):
    c = qs.Circuit(n)
    t = list(range(f0, f0 + K))
    c.add_walsh(t) if kind == "walsh" else c.add_dft(t, 1 if kind == "dft+" else -1, src)
    st = torch.from_numpy(np.ascontiguousarray(psi)).cuda()
    qs.qsim_apply(st, c)
    return st.cpu().numpy()


@pytest.mark.parametrize("kind", ["walsh", "dft+", "dft-"])
@pytest.mark.parametrize("K", [5, 6, 7, 8, 9, 10])
def test_fields(qs, K, kind):
    """Field at the bottom, in the middle and at the top; no, low and high twiddle sources; a state
    that is one field; one lane."""
    for n, f0, src in ((K, 0, []), (K + 1, 1, [0]), (K + 2, 0, [K, K + 1]), (K + 5, 3, [0, 1, 2]), (K + 5, 5, []),
                       (K + 5, 2, [K + 2, K + 3]), (K + 4, 4, [1, 3])):
        psi = synth.gaussian_state_np(K + f0, n)
        s = [] if kind == "walsh" else src
        out, ref = run(qs, psi, n, f0, K, kind, s), reference(psi, n, f0, K, kind, s)
        assert np.max(np.abs(out - ref)) <= 8 * (K + 2) * 2.0 ** -53 * 2.0 ** (K / 2) * np.max(np.abs(psi)), (n, f0, s)


@pytest.mark.parametrize("kind", ["dft+", "dft-"])
@pytest.mark.parametrize("K", [9, 10])
def test_tile_twiddles(qs, K, kind):
    """Sources on both sides of the rule for one twiddle table a tile: none, one or all of them in a lane; tiles of
    few and of many lanes; more tiles than SMs."""
    for n, f0, src in ((K + 8, 4, [K + 4, K + 5]), (K + 9, 4, [3]), (K + 9, 5, [4, K + 5, K + 8]), (K + 9, 3, [2, K + 4]),
                       (K + 11, 4, [0, 1, 2, 3]), (K + 11, 4, [K + 4 + i for i in range(7)])):
        psi = synth.gaussian_state_np(K + f0, n)
        out, ref = run(qs, psi, n, f0, K, kind, src), reference(psi, n, f0, K, kind, src)
        assert np.max(np.abs(out - ref)) <= 8 * (K + 2) * 2.0 ** -53 * 2.0 ** (K / 2) * np.max(np.abs(psi)), (n, f0, src)


@pytest.mark.parametrize("kind", ["walsh", "dft+", "dft-"])
@pytest.mark.parametrize("K", [6, 9, 10])
def test_values(qs, K, kind):
    """Zero columns, spikes over small values, a wide range, exponents near the ends, denormals,
    infinities and NaN (a tile that holds one runs in FP64; other tiles do not change)."""
    rng = np.random.default_rng(K)
    n, f0 = K + 5, 4
    base = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    rest, idx = columns(n, f0, K)
    for what in ("zero", "spike", "wide", "1e300", "1e-300", "1e-315", "nan", "inf"):
        psi = base.copy()
        if what == "zero":
            psi[idx[::3]] = 0
        elif what == "spike":
            psi *= 1e-9
            psi[idx[:, 5]] = 1j
        elif what == "wide":
            psi *= 10.0 ** rng.uniform(-30, 0, 1 << n)
        elif what in ("nan", "inf"):
            psi[idx[3, 7]] = complex(float(what), 0.0)
        else:
            psi *= float(what)
        out = run(qs, psi, n, f0, K, kind, [])
        with np.errstate(all="ignore"):
            ref = reference(psi, n, f0, K, kind, [])
        if what in ("nan", "inf"):
            # every amplitude of the column (the other part stays finite where only 1 and i multiply)
            assert not np.isfinite(out[idx[3]]).any()
            keep = np.delete(idx, 3, axis=0)
            out, ref, psi = out[keep], ref[keep], psi[keep]
        tol = 8 * (K + 2) * 2.0 ** -53 * 2.0 ** (K / 2) * np.max(np.abs(psi))
        assert np.max(np.abs(out - ref)) <= max(tol, 2.0 ** (K - 1074)), what
        if what == "zero":
            assert np.all(out[idx[::3]] == 0)
