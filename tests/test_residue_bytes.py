"""The residue form as the kernels store and rebuild it, restated on the CPU in exact integer
arithmetic: the plan with its 2^-9 margin, the weights on operand B, the chunk folds in FP32
and the byte of every residue, the grouped reconstruction with its offset, the nearest quotient
from the top limbs and the table of multiples of M, and the conversion of the 128-bit
magnitude to the nearest double."""
import math
from fractions import Fraction

import numpy as np
import pytest

MODULI = [256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193]
M = math.prod(MODULI)
N = [M // m for m in MODULI]
CHUNK = 1024


def sym(x, m):
    r = x % m
    return r - m if 2 * r > m else r


Y = [sym(pow(Nl % m, -1, m), m) for Nl, m in zip(N, MODULI)]


def plan_bits(Kp):
    """p of a product of at least 54 bits: all 16 moduli, 2 Kp 2^{2p} <= M (1 - 2^-9)."""
    room = (M - (M >> 9)) // (2 * Kp)
    return min((room.bit_length() - 1) // 2, 62)


def fold(x, m):
    """x - m round(x inv) with inv = 1 / m rounded to FP32 and x inv + 1.5 2^23 rounded once to
    an integer, ties to even (one unit in the last place there is 1)."""
    inv = np.int64(round(float(np.float32(1.0) / np.float32(m)) * 2.0 ** 31))  # exact: 24 bits
    t = np.asarray(x, np.int64) * inv
    q, r = t >> 31, t & (2 ** 31 - 1)
    q = q + ((r > 2 ** 30) | ((r == 2 ** 30) & (q & 1 == 1)))
    return x - q * m


def one_fold(m):
    return m == 256 or m <= 253


def stored(sums, m):
    """The value that the stored byte stands for, given the chunk sums (last axis) of an element."""
    sums = np.asarray(sums, np.int64)
    r = fold(sums, m)
    if sums.shape[-1] == 1 and one_fold(m):
        r = r[..., 0]
    else:
        r = fold(r.sum(-1), m)
    return (r + 128 & 255) - 128


@pytest.mark.parametrize("m", MODULI)
def test_the_byte_is_congruent_next_to_every_half_integer_quotient(m):
    k = np.arange(-(2 ** 24 // m) - 1, 2 ** 24 // m + 2, dtype=np.int64) * m
    x = np.concatenate([k + m // 2 + d for d in (-2, -1, 0, 1, 2)])
    x = x[np.abs(x) <= 2 ** 24]
    b = stored(x[:, None], m)
    assert np.all((x - b) % m == 0)


def test_one_fold_of_modulus_255_does_not_fit_its_byte():
    x = np.int64(-(255 * 40832 + 127))
    assert fold(x, 255) == 128 and stored(x[None], 255) == -127


@pytest.mark.parametrize("m", MODULI)
def test_several_chunks(m):
    rng = np.random.default_rng(m)
    x = rng.integers(-2 ** 24, 2 ** 24 + 1, (4000, 64))
    x[:64] = x[:64] // m * m + m // 2
    assert np.all((x.sum(1) - stored(x, m)) % m == 0)


# ---- grouped reconstruction

GROUPS = [list(range(g, min(16, g + 3))) for g in range(0, 16, 3)]
E = (-128 * sum(N)) % M
TOP = max(t for t in range(4) if M >> 32 * t)
B0 = max(0, TOP - 1)


def rebuild(t):
    """X from the values of the bytes (t + 128 in 0..255): sums of three moduli, the quotient
    nearest to S / M from three limbs in FP32, S - q M in 128 bits."""
    S = E
    for g in GROUPS:
        P = math.prod(MODULI[l] for l in g)
        v = sum((t[l] + 128) * (P // MODULI[l]) for l in g)
        assert v < 2 ** 26
        S += v * (M // P)
    assert 0 <= S < 32 * M
    a = [S >> 32 * (B0 + i) & 0xffffffff for i in range(3)]
    a[2] = S >> 32 * (B0 + 2)
    f = np.float32
    # fused multiply-adds: the products by powers of two are exact
    sf = f(float(f(a[2])) * 2.0 ** 64 + float(f(float(f(a[1])) * 2.0 ** 32 + float(f(a[0])))))
    inv = f(2.0 ** (32 * B0) / M)
    q = int(np.rint(float(sf) * float(inv)))  # |q| < 2^5: the shift by 1.5 2^23 rounds to integers
    X = S - q * M
    assert -2 ** 127 <= X < 2 ** 127
    return X


@pytest.mark.parametrize("Kp", [64, 832, 1024, 2048, 16384])
def test_saturated_and_constant_operands(Kp):
    p = plan_bits(Kp)
    assert p >= 55 and Kp * (2 ** p - 1) ** 2 <= (M - (M >> 9)) // 2
    rng = np.random.default_rng(Kp)
    top = 2 ** p - 1
    pairs = [(top, top), (top, -top), (1, 1), (0, top)]
    pairs += [(int(rng.integers(2 ** 52, 2 ** 53)) << p - 53, int(rng.integers(2 ** 52, 2 ** 53)) << p - 53)
              for _ in range(60)]
    # constant operands whose chunk sum's single fold would be 128 for modulus 255
    pairs += [(int(a * 2 ** (p - 1)), int(b * 2 ** (p - 1))) for a, b in
              [(1.31640625, 1.01171875), (1.671875, 1.9765625), (1.55078125, 1.69140625), (1.35546875, 1.203125)]]
    chunks = [min(CHUNK, Kp - c) for c in range(0, Kp, CHUNK)]
    for a, b in pairs:
        t = []
        for l, m in enumerate(MODULI):
            ab = sym(a, m) * sym(sym(b, m) * Y[l], m)
            t.append(int(stored([n * ab for n in chunks], m)))
        assert rebuild(t) == Kp * a * b


def scaled(w, neg, e):
    """The kernel's conversion of the 128-bit magnitude w times 2^e, on 32-bit words."""
    words = [w >> 32 * i & 0xffffffff for i in (3, 2, 1, 0)]
    if w == 0:
        return 0.0
    lead = next(i for i in range(4) if words[i])
    lz = 32 - words[lead].bit_length()
    v = w << (lz + 32 * lead) & (1 << 128) - 1
    h1, h0, l = v >> 96, v >> 64 & 0xffffffff, v & (1 << 64) - 1
    rest, odd = (h0 & 0x7ff) << 1 | (l != 0), h0 >> 11 & 1
    mant = (h1 >> 11 << 32 | (h1 << 32 | h0) >> 11 & 0xffffffff) + (rest + odd > 0x800)
    be = 127 - (lz + 32 * lead) + 1022
    bits = lambda b: np.array([neg << 63 | (b << 52) + mant], np.uint64).view(np.float64)[0]
    return float(bits(be + e)) if 0 <= be + e < 2046 else math.ldexp(float(bits(be)), e)


def test_conversion_rounds_to_nearest_even():
    rng = np.random.default_rng(3)
    vals = [1, 2 ** 53, 2 ** 53 + 1, 2 ** 54 + 2, 2 ** 54 + 6, 2 ** 127 - 1, 2 ** 96 - 1, (2 ** 54 - 1) << 40,
            (2 ** 53 + 1 << 11) + 1 << 60, (2 ** 53 + 1 << 60) + 1]
    vals += [int.from_bytes(rng.bytes(16), "little") >> int(rng.integers(1, 128)) for _ in range(4000)]
    for w in vals:
        for e in (0, -110, 850, -1000):
            assert scaled(w, 0, e) == float(Fraction(w) * Fraction(2) ** e)
            assert scaled(w, 1, e) == -float(Fraction(w) * Fraction(2) ** e)
