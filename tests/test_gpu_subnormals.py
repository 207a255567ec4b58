"""complex128 states of subnormal numbers, with and without set bits in their high words (1e-310, 1e-315): gates,
passes and the batched executor take them in FP64 and keep their values.  Tolerance: those of test_gpu_dense_f64.py
and test_gpu_dft_fx.py where no result is representable more finely than 2^-1074."""
import numpy as np
import pytest
import torch

import synth
from oracle import core as ocore
from test_gpu_dft_fx import columns, reference, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs(cuda_device):
    from paper_2402_08136_gb300 import build
    build.build()
    import paper_2402_08136_gb300 as q
    return q


@pytest.mark.parametrize("scale", [1e-310, 1e-315])
@pytest.mark.parametrize("kind", ["walsh", "dft+", "dft-"])
def test_passes(qs, kind, scale):
    rng = np.random.default_rng(3)
    for n, f0, K in ((9, 2, 5), (12, 3, 6), (13, 3, 10), (15, 4, 10)):
        rest, idx = columns(n, f0, K)
        psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
        psi[idx[::2]] *= scale  # next to columns in the ordinary range, and alone
        for x in (psi, psi * 2.0 ** 1 * scale):
            ref = reference(x, n, f0, K, kind, [])
            c, t = qs.Circuit(n), list(range(f0, f0 + K))
            c.add_walsh(t) if kind == "walsh" else c.add_dft(t, 1 if kind == "dft+" else -1, [])
            st = torch.from_numpy(x).cuda()
            qs.qsim_apply_batched([st], [c])
            for out in (st.cpu().numpy(), run(qs, x, n, f0, K, kind, [])):
                for cols in (idx[::2], idx[1::2]):
                    tol = 8 * (K + 2) * 2.0 ** -53 * 2.0 ** (K / 2) * np.max(np.abs(x[cols]))
                    assert np.max(np.abs(out[cols] - ref[cols])) <= max(tol, 2.0 ** (K - 1074)), (n, K)


@pytest.mark.parametrize("scale", [1e-310, 1e-315])
@pytest.mark.parametrize("k,n", [(1, 12), (3, 12), (4, 12), (4, 18), (5, 13), (6, 13), (6, 19)])
def test_gates(qs, k, n, scale):
    rng = np.random.default_rng(k)
    U, t = synth.haar_unitary(rng, 1 << k), synth.random_targets(rng, n, k)
    psi = synth.gaussian_state_np(k, n) * scale
    ref = psi.copy()
    ocore.apply_gate(ref, t, U)
    st = torch.from_numpy(psi).cuda()
    qs.qsim_apply(st, qs.Circuit(n).add_gate(t, U))
    out = st.cpu().numpy()
    assert np.max(np.abs(out)) > 0
    assert np.max(np.abs(out - ref)) <= 2.0 ** (k + 2 - 1074)
