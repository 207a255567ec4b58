"""complex128 gates whose digits are all at the ends of their range, so that the sums of the digit kernels come as close to
2^24 as they can (64 and 128 products) before they cancel: the results have to be exact to the kernels' last kept bit.

x = +-(2^61 .. 2^62 units, digits -128 below the top one), U = digits +128: every product of two lower digits is +-2^14.
The terms of a sum all have one sign, or its first half drives it up and the second half back; the results are computed in
integers here.
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


# 62-bit integers with at most 53 significant bits, top digit 64 and 32
X = (64 << 56) - 128 * sum(1 << (8 * i) for i in range(1, 7))
V = (32 << 56) + 128 * sum(1 << (8 * i) for i in range(2, 7))


@pytest.mark.parametrize("cancel", [True, False])
@pytest.mark.parametrize("k,real,n", [(1, False, 10), (2, False, 10), (3, False, 12), (4, False, 12), (4, True, 12), (4, False, 18),
                                      (5, False, 13), (5, True, 13), (5, False, 19), (6, False, 13), (6, True, 13),
                                      (6, True, 18), (6, False, 18), (6, False, 19)])
def test_sums_at_their_ends(qs, k, real, n, cancel):
    rng = np.random.default_rng(10 * k + n + real)
    D = 1 << k
    assert float(X) == X and float(V) == V and X < 1 << 62
    u = float(V) / 2.0 ** 62  # below 1, above 1/8
    U = np.full((D, D), u if real else complex(u, -u), dtype=np.complex128)
    t = synth.random_targets(rng, n, k)
    idx = np.arange(1 << n)
    row = sum(((idx >> q) & 1) << b for b, q in enumerate(t))
    sign = np.where(row < D // 2, 1, -1 if cancel else 1)
    if D > 2 and cancel:  # a few terms more or less in the second half: sums that do not cancel
        sign = np.where((row >= D // 2) & (rng.random(1 << n) < 0.1), 0, sign)
    re = sign * X
    im = sign * (X - (1 << 20))
    psi = (re.astype(np.float64) + 1j * im.astype(np.float64)) / 2.0 ** 62
    group = idx & ~sum(1 << q for q in t)
    sum_re, sum_im = {}, {}
    for g, a, b in zip(group.tolist(), re.tolist(), im.tolist()):
        sum_re[g] = sum_re.get(g, 0) + a
        sum_im[g] = sum_im.get(g, 0) + b
    st = torch.from_numpy(psi).cuda()
    before = qs.qsim_launch_counts()["dense_tc"]
    qs.qsim_apply(st, qs.Circuit(n).add_gate(t, U))
    out = st.cpu().numpy()
    assert qs.qsim_launch_counts()["dense_tc"] > before
    worst = 0.0
    for i, g in enumerate(group.tolist()):
        yr = V * sum_re[g] + (0 if real else V * sum_im[g])
        yi = V * sum_im[g] - (0 if real else V * sum_re[g])
        worst = max(worst, abs(int(out[i].real * 2.0 ** 80) * 2 ** 44 - yr), abs(int(out[i].imag * 2.0 ** 80) * 2 ** 44 - yi))
    # half of the last kept bit (2^(13 - 68) of 2^124 at most), the digit pairs left out (7 per product, each below 2^62
    # of the 2^124) and the rounding to 53 bits
    terms = D if real else 2 * D
    assert worst <= 2.0 ** (124 - 56) + 7 * terms * 2.0 ** 62 + 2.0 ** -53 * terms * V * X
