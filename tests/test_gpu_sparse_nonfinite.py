"""Mostly-zero complex128 gates on states with infinities and NaN: they spread as in a sum over whole rows (0 times an
infinity is a NaN), to every row of the group and to no other group."""
import numpy as np
import pytest
import torch

import synth
from oracle import core as ocore
from test_gpu_dense_sparse import sparse_unitary

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs(cuda_device):
    from paper_2402_08136_gb300 import build
    build.build()
    import paper_2402_08136_gb300 as q
    return q


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("k,w", [(2, 1), (3, 1), (4, 2), (5, 3), (6, 4), (7, 1)])
def test_nonfinite(qs, k, w, real):
    rng = np.random.default_rng(10 * k + real)
    n = max(k + 4, 13)
    U = sparse_unitary(rng, k, w, real)
    for value in (complex(np.inf, 0.25), complex(0.5, -np.inf), complex(np.nan, 1.0)):
        t = synth.random_targets(rng, n, k)
        psi = synth.gaussian_state_np(k, n)
        at = int(rng.integers(1 << n))
        psi[at] = value
        ref = psi.copy()
        mag = np.abs(np.where(np.isfinite(psi.real), psi.real, 0) + 1j * np.where(np.isfinite(psi.imag), psi.imag, 0)).astype(np.complex128)
        with np.errstate(all="ignore"):
            if real:  # part by part: the plain form of a real U leaves the zero imaginary parts out
                for part in ("real", "imag"):
                    p = getattr(psi, part).astype(np.complex128)
                    ocore.apply_gate(p, t, U)
                    setattr(ref, part, p.real)
            else:
                ocore.apply_gate(ref, t, U)
            ocore.apply_gate(mag, t, np.abs(U).astype(np.complex128))
        st = torch.from_numpy(psi).cuda()
        qs.qsim_apply(st, qs.Circuit(n).add_gate(t, U))
        out = st.cpu().numpy()
        group = np.isin(np.arange(1 << n) & ~sum(1 << q for q in t), [at & ~sum(1 << q for q in t)])
        for part in ("real", "imag"):
            o, r = getattr(out, part), getattr(ref, part)
            fine = np.isfinite(r)
            assert np.array_equal(np.isfinite(o), fine)
            assert np.all(fine[~group])
            assert np.all(np.abs(o[fine] - r[fine]) <= 2.0 ** (w + 2) * 2.0 ** -53 * mag.real[fine] + 1e-300)
        assert not np.isfinite(out[group]).any()
