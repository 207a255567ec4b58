"""Mostly-zero complex128 gates on both sides of the rule that gives a real U with half of its rows to the tiled kernels
(2^20 amplitudes, controls apart): the same sums either way, each within the bound of its own terms."""
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


@pytest.mark.parametrize("n,extra", [(19, 0), (20, 0), (20, 1), (21, 1)])
@pytest.mark.parametrize("k,w", [(1, 0), (2, 1), (3, 2), (4, 3), (3, 1)])
def test_both_sides(qs, k, w, n, extra):
    rng = np.random.default_rng(100 * k + n)
    U = sparse_unitary(rng, k, w, True) if k > 1 else np.array([[0, 1], [1, 0]], dtype=np.complex128)
    q = [int(v) for v in rng.permutation(n)]
    t, ctl = q[:k], q[k:k + extra]
    psi = synth.gaussian_state_np(k, n) * 10.0 ** rng.uniform(-30, 0, 1 << n)
    ref, mag = psi.copy(), np.abs(psi).astype(np.complex128)
    ocore.apply_gate(ref, t, U, ctl)
    ocore.apply_gate(mag, t, np.abs(U).astype(np.complex128), ctl)
    st = torch.from_numpy(psi).cuda()
    qs.qsim_apply(st, qs.Circuit(n).add_gate(t, U, ctl))
    out = st.cpu().numpy()
    assert np.all(np.abs(out - ref) <= 2.0 ** (w + 2) * 2.0 ** -53 * mag.real)
