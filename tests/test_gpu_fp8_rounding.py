"""The FP8 form's products are rounded to FP64 once: sums of more than 53 bits whose digits
are exact come out as the nearest double, whatever follows below the half unit."""
import fractions

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def zb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06204_gb300 import build
    build.build()
    from paper_1806_06204_gb300 import binding
    return binding


def dev(a):
    import torch
    return torch.from_numpy(np.asfortranarray(a)).cuda()


# column j holds `terms` integers of 53 bits and a 1 that meets the row's 2^-t: their sum is an
# integer of 54 to 60 bits plus 2^-t.  Every entry is a whole number of the format's units
# (2^-55 of twice the next power of two) and every digit pair lies in the kept levels, so the
# exact sum is known and the result is its nearest double.
@pytest.mark.parametrize("terms", [2, 3, 5, 9, 30, 64])
@pytest.mark.parametrize("t", [1, 4, 8])
def test_sums_beyond_53_bits_round_once(zb, terms, t):
    rng = np.random.default_rng(100 * terms + t)
    n = 96
    B = np.ones((terms + 1, n))
    for j in range(n):
        v = [int(x) for x in rng.integers(2 ** 52, 2 ** 53, terms)]
        # the sum just above an odd last place: the case a tie would be made of
        ulp = 2 ** max(0, sum(v).bit_length() - 53)
        v[0] -= (sum(v) % (2 * ulp)) - ulp
        v[0] += 2 * ulp * (v[0] < 2 ** 52) - 2 * ulp * (v[0] >= 2 ** 53)
        B[:terms, j] = v
    A = np.ones((2, terms + 1))
    A[0, terms] = 2.0 ** -t
    A[1] = -A[0]
    h = zb.Handle(0)
    try:
        C = zb.zolo_dgemm(h, dev(A), dev(B), prec=zb.ZOLO_SPLIT_FP8).cpu().numpy()
    finally:
        h.close()
    for j in range(n):
        exact = sum(fractions.Fraction(a) * fractions.Fraction(b) for a, b in zip(A[0], B[:, j]))
        assert C[0, j] == float(exact) and C[1, j] == -float(exact)
