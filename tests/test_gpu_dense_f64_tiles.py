"""Wide complex128 gates on states of many tiles per SM, some of which leave the fixed-point range.

What the loading warps of a CTA tell its reading warps about a tile (exponents, whether it runs in FP64) goes through
a few slots that the CTA's tiles share.  Here every CTA has 13 tiles or more, so each slot is used several times, and
the tiles that hold an infinity, a NaN, values near 1e-300 or subnormals lie next to each other, a slot's reuse apart
or anywhere.

Tolerance: that of test_gpu_dense_f64.py, with the largest value of the amplitude's own group in place of the state's.
"""
import numpy as np
import pytest
import torch

import synth
from oracle import core as ocore
from test_gpu_dense_f64_tc import FORMS, unitary

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs(cuda_device):
    from paper_2402_08136_gb300 import build
    build.build()
    import paper_2402_08136_gb300 as q
    return q


def reference(psi, t, U, real):
    """The oracle's result; for a real U part by part, so that an infinity stays in its part as in the kernels."""
    with np.errstate(all="ignore"):
        if not real:
            ref = psi.copy()
            ocore.apply_gate(ref, t, U)
            return ref
        ref = np.empty_like(psi)
        for part in ("real", "imag"):
            p = getattr(psi, part).astype(np.complex128)
            ocore.apply_gate(p, t, U)
            setattr(ref, part, p.real)
        return ref


@pytest.mark.parametrize("pattern", ["run", "every4", "any"])
@pytest.mark.parametrize("k,real,gb", FORMS)
def test_marked_tiles(qs, k, real, gb, pattern):
    rng = np.random.default_rng(100 * k + real)
    n = k + gb + 11
    t = synth.random_targets(rng, n, k)
    U = unitary(rng, k, real)
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tile = np.arange(1 << 11)
    at = tile // sms  # the tile's place in its CTA
    marked = {"run": (at % 8) < 5, "every4": at % 4 == 1, "any": rng.random(1 << 11) < 0.3}[pattern]
    free = [q for q in range(n) if q not in t]
    for j in np.flatnonzero(marked):
        g = int(j) << gb | int(rng.integers(1 << gb))
        base = sum(((g >> b) & 1) << q for b, q in enumerate(free))
        idx = base + sum(((np.arange(1 << k) >> b) & 1) << q for b, q in enumerate(t))
        what = ("inf", "nan", "1e-300", "1e-310", "1e-315")[int(rng.integers(5))]
        if what in ("inf", "nan"):
            psi[idx[int(rng.integers(1 << k))]] = complex(float(what), 0.5)
        else:
            psi[idx] *= float(what)
    ref = reference(psi, t, U, real)
    st = torch.from_numpy(psi).cuda()
    before = qs.qsim_launch_counts()["dense_tc"]
    qs.qsim_apply(st, qs.Circuit(n).add_gate(t, U))
    out = st.cpu().numpy()
    assert qs.qsim_launch_counts()["dense_tc"] == before + 1
    assert qs.qsim_device_status() == 0
    top = np.where(np.isfinite(psi), np.abs(psi), 0).reshape((2,) * n).max(axis=tuple(n - 1 - q for q in t), keepdims=True)
    tol = np.broadcast_to((2.0 ** (k + 1) + 2) * 2.0 ** -53 * 2.0 ** (k / 2) * top + 2.0 ** (k - 1073), (2,) * n).reshape(-1)
    for part in ("real", "imag"):
        o, r = getattr(out, part), getattr(ref, part)
        fine = np.isfinite(r)
        assert not fine.all() or part == "imag"
        assert np.array_equal(np.isfinite(o), fine)
        assert np.all(np.abs(o[fine] - r[fine]) <= tol[fine])
