"""hhl_readout_sums and the streams of other work: it follows the latest replay of a graph that holds its run, on
whichever stream that replay is, and waits for nothing else."""
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


def problem(qs, m, b, dtype=torch.complex64):
    p = synth.hhl27_problem()
    h = qs.hhl_build(p["A"], b, m, structured=True, fft_qft=True)
    st = torch.empty(1 << h.info()["n"], dtype=dtype, device="cuda")
    return h, qs.qsim_fuse(h.as_circuit(), 4), st, torch.zeros(qs.QSIM_READOUT_SUMS_DOUBLES, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("replay_on", ["default", "other"])
def test_follows_the_replay(qs, cuda_device, replay_on):
    b = synth.hhl27_problem()["b"]
    h, c, st, sums = problem(qs, 17, b)  # 24 qubits: a replay takes far longer than the call of the readout
    s, r = torch.cuda.Stream(), torch.cuda.Stream()
    qs.hhl_run_sums(st, h, sums, c, stream=s)
    s.synchronize()
    want = qs.hhl_readout_sums(st, h, sums, stream=s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        qs.hhl_run_sums(st, h, sums, c, stream=s)
    for _ in range(5):
        with torch.cuda.stream(torch.cuda.default_stream() if replay_on == "default" else r):
            st.zero_()
            sums.zero_()
            for _ in range(3):
                g.replay()
        got = qs.hhl_readout_sums(st, h, sums, stream=s)
        assert got["p_success"] == want["p_success"] and np.array_equal(got["x"], want["x"])
        torch.cuda.synchronize()


def test_replay_after_the_problem_is_gone(qs, cuda_device):
    """The circuit's graph stays valid without the problem that the run was captured with."""
    h, c, st, sums = problem(qs, 12, synth.hhl27_problem()["b"])
    s = torch.cuda.Stream()
    qs.hhl_run_sums(st, h, sums, c, stream=s)
    s.synchronize()
    want = st.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        qs.hhl_run_sums(st, h, sums, c, stream=s)
    del h
    st.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(st), torch.view_as_real(want))


def test_waits_for_nothing_else(qs, cuda_device):
    h, c, st, sums = problem(qs, 12, synth.hhl27_problem()["b"])
    s = torch.cuda.Stream()
    qs.hhl_run_sums(st, h, sums, c, stream=s)
    want = qs.hhl_readout_sums(st, h, sums, stream=s)
    torch.cuda.synchronize()
    torch.cuda._sleep(1_000_000_000)  # about half a second of other work on the default stream
    qs.hhl_run_sums(st, h, sums, c, stream=s)
    got = qs.hhl_readout_sums(st, h, sums, stream=s)
    assert not torch.cuda.default_stream().query()
    assert np.array_equal(got["x"], want["x"])
    torch.cuda.synchronize()
