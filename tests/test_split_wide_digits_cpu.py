"""CPU model of the split product's 8-bit digits (no GPU).

The 16-bit forms hold an operand as balanced base-256 digits; the exact level sums
are added up to a top level.  Against exact products the 34 pairs (levels 2..9,
seven digits) must be no worse than nine 6-bit digits with levels 2..11, the 28
pairs (levels 2..8) no worse than eight 7-bit digits with levels 2..9, and six
digits with levels 2..8 no worse than eight 6-bit digits with levels 2..10; and no
level of a 192-term chunk up to 6 may exceed what FP32 holds exactly."""
import numpy as np
import pytest


def digits(X, b, S):
    """Balanced base-2^b digits of the rows of X, scaled to below 1/2 by powers of two."""
    e = np.frexp(np.max(np.abs(X), axis=1))[1] + 1
    N = np.rint(np.ldexp(X.astype(np.longdouble), (b * S - e)[:, None])).astype(np.int64)
    out = [None] * S
    for s in range(S - 1, 0, -1):
        r = N & ((1 << b) - 1)
        r = np.where(r >= (1 << (b - 1)), r - (1 << b), r)
        out[s] = r.astype(np.float64)
        N = (N - r.astype(np.int64)) >> b
    out[0] = N.astype(np.float64)
    return out, e


def error(A, B, b, S, top):
    da, ea = digits(A, b, S)
    db, eb = digits(np.ascontiguousarray(B.T), b, S)
    tot = np.zeros((A.shape[0], B.shape[1]), np.longdouble)
    for s in range(1, S + 1):
        for t in range(1, min(S, top - s) + 1):
            tot += np.ldexp((da[s - 1] @ db[t - 1].T).astype(np.longdouble), -b * (s + t))
    ref = A.astype(np.longdouble) @ B.astype(np.longdouble)
    P = np.ldexp(tot, ea[:, None] + eb[None, :])
    scale = np.abs(A).max(1)[:, None] * np.abs(B).max(0)[None, :]
    return float(np.sqrt(np.mean(((P - ref) / scale) ** 2)))


def operands(kind, K):
    rng = np.random.default_rng(K)
    A, B = rng.standard_normal((40, K)), rng.standard_normal((K, 40))
    if kind == "gram":
        B = A.T.copy()
    elif kind == "graded":
        A *= 10.0 ** rng.uniform(-8, 0, (1, K))
        B *= 10.0 ** rng.uniform(-8, 0, (K, 1))
    return A, B


@pytest.mark.parametrize("kind", ["normal", "gram", "graded"])
@pytest.mark.parametrize("K", [64, 512])
def test_eight_bit_digits_lose_nothing(kind, K):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("needs an extended long double")
    A, B = operands(kind, K)
    # the rms of 1600 samples: 10% of sampling noise
    assert error(A, B, 8, 7, 9) <= 1.1 * error(A, B, 6, 9, 11)
    assert error(A, B, 8, 7, 8) <= 1.1 * error(A, B, 7, 8, 9)
    assert error(A, B, 8, 6, 8) <= 1.1 * error(A, B, 6, 8, 10)


def test_leading_levels_of_a_chunk_are_exact_in_fp32():
    for level in range(2, 7):
        pairs = level - 1
        assert pairs * 192 * 128 * 128 <= 2 ** 24
    # an int64 in units of 2^-48 holds the leading levels of 28 * 4096 terms
    per_term = sum((L - 1) * 2 ** 14 * 2.0 ** (48 - 8 * L) for L in range(2, 7))
    assert per_term * 28 * 4096 < 2 ** 63
    # one 192-term chunk also fits in units of 2^-56
    assert per_term * 192 * 2 ** 8 < 2 ** 62
