"""The fixed-point scheme of the tall-skinny products A^T B on the tensor cores, restated in exact
integer arithmetic and checked on the CPU: column bounds of one bit more than the entries need,
7 balanced base-256 digits, the digit planes of A stacked in bands of an M = 128 operand, B's
along N, accumulators read out every 256 rows, the bands shifted and added.  It pins the scheme
as the kernel uses it (which digit pairs meet in which accumulator, that FP32 holds their sums
exactly, the error of the result), not the kernel itself; that is held to the FP64 parity bound
by the GPU tests."""
import math
from fractions import Fraction

import numpy as np
import pytest

NDIG = 7
ROWS = 256          # rows between two read-outs
MASK64 = (1 << 64) - 1
WIDTHS = [16, 32, 48, 64]          # column counts padded to 16


def digits(x, e):
    """T = trunc(x 2^(56 - e)) as balanced digits, T = sum d_s 2^(48 - 8 s)."""
    T = math.trunc(Fraction(float(x)) * Fraction(2) ** (56 - e))
    V = (T + 0x808080808080) & MASK64
    d = [0] * NDIG
    for s in range(1, NDIG):
        d[s] = ((V >> (48 - 8 * s)) & 0xFF) - 128
    v = V - (1 << 64) if V >> 63 else V
    d[0] = v >> 48
    return d


def pairs(P):
    """{(band u, block g): digit pairs (s, t)} of a padded width P: the MMA at plane s1 of A
    (0, h, 2 h, ..: h planes fit in 128 lanes) covers the planes s1 + u, u < h, and the planes
    t = 0 .. 6 - s1 of B, into the blocks g = s1 + t."""
    h = 128 // P
    out = {}
    for s1 in range(0, NDIG, h):
        for u in range(min(h, NDIG)):
            for t in range(NDIG - s1):
                out.setdefault((u, s1 + t), []).append((s1 + u, t))
    # read out: orders past the last are dropped (planes past the last of A are among them)
    return {(u, g): p for (u, g), p in out.items() if g + u < NDIG}


@pytest.mark.parametrize("P", WIDTHS)
def test_every_pair_meets_once(P):
    seen = [p for ps in pairs(P).values() for p in ps]
    assert sorted(seen) == sorted((s, t) for s in range(NDIG) for t in range(NDIG - s))
    for (u, g), ps in pairs(P).items():
        assert all(s + t == g + u for s, t in ps)


def test_digits_with_the_bound_one_bit_higher():
    """Every digit, the leading one included, within [-128, 128]: at most 8 significant bits."""
    rng = np.random.default_rng(3)
    xs = np.concatenate([rng.standard_normal(2000) * 2.0 ** rng.integers(-70, 70, 2000),
                         [np.nextafter(1.0, 0.0), -np.nextafter(1.0, 0.0), 1.0, -1.0, 0.0]])
    for x in xs:
        c = math.frexp(x)[1] if x else 0
        d = digits(x, c + 1)
        assert all(-128 <= v <= 128 for v in d)
        assert all(-128 <= v <= 127 for v in d[1:])


@pytest.mark.parametrize("P", WIDTHS)
def test_fp32_sums_are_exact_over_a_read_out(P):
    """|D| <= 2^24 for every accumulator, <= 2^22 for blocks 0 and 1, whose integers are taken
    from the low bits of D + 1.5 2^23; the combined sums stay below 2^63."""
    for (u, g), ps in pairs(P).items():
        worst = ROWS * len(ps) * 128 * 128
        assert worst <= 2 ** 24
        if g <= 1:
            assert worst <= 2 ** 22
    for u in range(min(128 // P, NDIG)):
        top = sum(ROWS * len(ps) * 2 ** 14 * 2 ** (40 - 8 * g)
                  for (v, g), ps in pairs(P).items() if v == u)
        assert top < 2 ** 63
    for d in (-2 ** 22, -2 ** 22 + 1, -1, 0, 1, 2 ** 22 - 1, 2 ** 22):
        assert int((np.float32(d) + np.float32(12582912.0)).view(np.int32)) - 0x4B400000 == d


def product(A, B, P):
    """A^T B (at most 256 rows) by the scheme; the column exponents."""
    ca = [max((math.frexp(v)[1] for v in col if v), default=0) for col in A.T]
    cb = [max((math.frexp(v)[1] for v in col if v), default=0) for col in B.T]
    da = np.array([[digits(x, ca[i] + 1) for x in A[:, i]] for i in range(A.shape[1])])
    db = np.array([[digits(x, cb[j] + 1) for x in B[:, j]] for j in range(B.shape[1])])
    out = np.zeros((A.shape[1], B.shape[1]))
    for i in range(A.shape[1]):
        for j in range(B.shape[1]):
            D = {}
            for (u, g), ps in pairs(P).items():
                D[u, g] = sum(int(da[i, :, s] @ db[j, :, t]) for s, t in ps)
                assert abs(D[u, g]) <= 2 ** 24
            J = 0
            for u in range(min(128 // P, NDIG)):
                d = [D.get((u, g), 0) for g in range(NDIG)]
                J += (sum(d[g] << (40 - 8 * g) for g in range(NDIG - 1)) + (d[6] >> 8)) >> (8 * u)
            out[i, j] = float(Fraction(J) * Fraction(2) ** (ca[i] + cb[j] + 2 - 56))
    return out, ca, cb


def columns(kind, rng, rows, n):
    x = rng.standard_normal((rows, n))
    if kind == "graded":               # within a column, entries over 30 binary orders
        x *= 2.0 ** -rng.integers(0, 30, size=(rows, n))
    elif kind == "spike":              # one entry far above the others
        x[rng.integers(rows, size=n), np.arange(n)] *= 2.0 ** 25
    elif kind == "scaled":             # columns of very different size
        x *= 2.0 ** rng.integers(-300, 300, size=n)
    return x


@pytest.mark.parametrize("P", WIDTHS)
@pytest.mark.parametrize("kind", ["plain", "graded", "spike", "scaled"])
def test_error_of_the_product(P, kind):
    """In units of 2^-54 of the product of the two columns' bounds 2^c: per row 1 for the values'
    truncation (each below 2^-55 of its bound) and 1.5 for the dropped orders (six pairs of order 7,
    2^14 2^-72 each, and less); 1 for each band's shift and for the last block, at most 8; and half
    an ulp of the result."""
    rng = np.random.default_rng(P)
    for rows in (1, 31, ROWS):
        A, B = columns(kind, rng, rows, 3), columns(kind, rng, rows, 2)
        out, ca, cb = product(A, B, P)
        for i in range(3):
            for j in range(2):
                exact = sum(Fraction(float(a)) * Fraction(float(b)) for a, b in zip(A[:, i], B[:, j]))
                bound = (3 * rows + 8) * Fraction(2) ** (ca[i] + cb[j] - 54)
                ulp = Fraction(math.ulp(float(exact))) if exact else Fraction(0)
                assert abs(Fraction(out[i, j]) - exact) <= bound + ulp / 2
