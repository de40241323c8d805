"""The arithmetic of the emulated FP64 product (Chinese remaindering) on the CPU, from the
scheme's definition with Python integers (no code shared with the CUDA path): the moduli are
coprime and large enough for the stated sizes, the accumulation bounds hold, and the 160-bit
fixed-point reconstruction returns the integer it was given."""
import math
import random

import pytest

MODULI = [255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193, 191, 181]


def needed(K, S):
    """Moduli whose product exceeds twice |Re C'| <= 2K 2^(14S-2)."""
    nm, P = 0, 1
    while P <= 2 * 2 * K * 2 ** (14 * S - 2):
        P *= MODULI[nm]
        nm += 1
    return nm


def test_moduli_and_bounds():
    for i, p in enumerate(MODULI):
        assert p % 2 == 1 and p <= 255
        assert all(math.gcd(p, q) == 1 for q in MODULI[:i])
    # a running residue plus 512 complex terms (1024 real products) stays an FP32 integer
    assert 127 * 127 * 1024 + 128 <= 2 ** 24
    # the largest order and digit count fit
    assert needed(30720, 8) <= len(MODULI)
    assert needed(2048, 8) == 16 and needed(1, 1) <= 3


@pytest.mark.parametrize("nm", [2, 5, 16, 17])
def test_reconstruction_returns_the_integer(nm):
    mods = MODULI[:nm]
    P = math.prod(mods)
    F = [(pow(P // p, -1, p) * 2 ** 160 + p // 2) // p for p in mods]
    off = -128 * sum(F) % 2 ** 160
    rnd = random.Random(nm)
    cases = [0, 1, -1, (P - 1) // 2, -((P - 1) // 2)] + [rnd.randrange(-(P // 2) + 1, P // 2) >> rnd.randrange(P.bit_length())
                                                        for _ in range(300)]
    for x in cases:
        r = [((x + p // 2) % p) - p // 2 for p in mods]
        assert all(-127 <= v <= 127 for v in r)
        s = (off + sum((v + 128) * f for v, f in zip(r, F))) % 2 ** 160
        s -= 2 ** 160 if s >> 159 else 0
        # the fraction's error, in units of x, is far below 1/2: rounding gives x
        assert abs(s * P - x * 2 ** 160) < 2 ** (160 - 15)
