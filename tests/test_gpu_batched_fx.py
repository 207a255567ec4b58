"""complex128 passes inside the batched executor in fixed point (reference and tolerance of
test_gpu_dft_fx.py), and batches whose two launches overlap."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_dft_fx import columns, reference

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs(cuda_device):
    from paper_2402_08136_gb300 import build
    build.build()
    import paper_2402_08136_gb300 as q
    return q


@pytest.mark.parametrize("kind", ["walsh", "dft+", "dft-"])
def test_fields_and_values(qs, kind):
    rng = np.random.default_rng(4)
    circs, states, refs, tols = [], [], [], []
    # in shared memory (up to 13 qubits) and in tiles (above); 5 stages, 5 + 1, 5 + 5; one column
    for n, f0, K, src in ((5, 0, 5, []), (11, 2, 6, [0, 1]), (13, 3, 10, [0, 1, 2]), (13, 8, 5, [2, 3]), (12, 2, 9, []),
                          (14, 4, 10, [1, 2, 3]), (16, 5, 10, []), (15, 9, 6, [0, 1, 2, 3])):
        for what in ("gauss", "zero", "spike", "wide", "1e-300", "1e-315", "nan"):
            psi = synth.gaussian_state_np(n, n) * 2.0 ** (n / 2)
            rest, idx = columns(n, f0, K)
            if what == "zero":
                psi[idx[::2]] = 0
            elif what == "spike":
                psi *= 1e-9
                psi[idx[:, 3]] = 1j
            elif what == "wide":
                psi *= 10.0 ** rng.uniform(-30, 0, 1 << n)
            elif what == "nan":
                psi[idx[-1, 1]] = complex(np.nan, 0)
            elif what != "gauss":
                psi *= float(what)
            s = [] if kind == "walsh" else src
            c = qs.Circuit(n)
            t = list(range(f0, f0 + K))
            c.add_walsh(t) if kind == "walsh" else c.add_dft(t, 1 if kind == "dft+" else -1, s)
            with np.errstate(all="ignore"):
                refs.append(reference(psi, n, f0, K, kind, s))
            circs.append(c)
            states.append(torch.from_numpy(psi).cuda())
            fine = np.abs(psi[np.isfinite(psi)])
            tols.append((idx, what, max(8 * (K + 2) * 2.0 ** -53 * 2.0 ** (K / 2) * fine.max(), 2.0 ** (K - 1074))))
    qs.qsim_apply_batched(states, circs)
    for st, ref, (idx, what, tol) in zip(states, refs, tols):
        out = st.cpu().numpy()
        if what == "nan":
            assert not np.isfinite(out[idx[-1]]).any()
            keep = idx[:-1]
            out, ref = out[keep], ref[keep]
        if out.size:
            assert np.max(np.abs(out - ref)) <= tol, (idx.shape, what)


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
def test_team_and_single_launches_overlap(qs, dtype):
    """A batch of circuits on teams and on single CTAs gives the same bits as each circuit alone, over
    repeated runs, and what follows on the stream sees both launches' results."""
    rng = np.random.default_rng(9)
    circs, psis = [], []
    for n in (16, 15, 16, 9, 12, 7, 13, 15, 10, 8):
        c = qs.Circuit(n)
        for _ in range(3):
            c.add_gate(synth.random_targets(rng, n, 4), synth.haar_unitary(rng, 16))
        c.add_walsh(list(range(2, 7)))
        circs.append(c)
        psis.append(torch.from_numpy(synth.gaussian_state_np(n, n)).to(dtype).cuda())
    alone = [p.clone() for p in psis]
    for c, p in zip(circs, alone):
        qs.qsim_apply_batched([p], [c])
    states = [p.clone() for p in psis]
    b = qs.qsim_batch_create(circs, states)
    for _ in range(5):
        for s, p in zip(states, psis):
            s.copy_(p)
        b.run()
        got = [s.clone() for s in states]  # on the same stream, right behind the second launch
        torch.cuda.synchronize()
        for g, a in zip(got, alone):
            assert torch.equal(torch.view_as_real(g), torch.view_as_real(a))
