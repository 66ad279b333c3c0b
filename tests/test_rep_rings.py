"""The mesh rule of VaFR_Rep that the kernels evaluate in 32 bits with one correction:
against the rule in unbounded integers, for the ring sizes that take it."""

import random

import pytest

M32 = (1 << 32) - 1


def _rule(n, n2, j, s):
    if s == 0:   # max{k : (2k+1) n < (2j+3) n2}, modulo the ring
        w = -((-(2 * j + 3) * n2) // n) - 2
        return (w // 2 if w >= 0 else -1) % n2
    q = (2 * j + 3) * n2 // n   # max{k : (2k+1) n <= (2j+3) n2}
    return ((q - 1) // 2 if q >= 1 else -1) % n2


def _kernel(n, n2, j, s):
    num = (2 * j + 3) * n2
    assert num + n - 1 <= M32
    k = (((num + n - 1) // n) - 2) >> 1 if s == 0 else ((num // n) - 1) >> 1
    if k < 0:
        k += n2
    elif k >= n2:
        k -= n2
    return k


@pytest.mark.parametrize("s", [0, 1])
def test_same_texel(s):
    rng = random.Random(5)
    rings = [1, 2, 3, 4, 7, 8, 100, 4000, 32766, 32767]
    cases = [(n, n2, j) for n in rings for n2 in rings for j in {0, 1, n // 2, n - 2, n - 1} if 0 <= j < n]
    for _ in range(20000):
        n = rng.randint(1, 32767)
        n2 = rng.choice([n, max(1, n - rng.randint(0, 40)), min(32767, n + rng.randint(0, 40)), rng.randint(1, 32767)])
        cases.append((n, n2, rng.randrange(n)))
    for n, n2, j in cases:
        k = _kernel(n, n2, j, s)
        assert 0 <= k < n2 and k == _rule(n, n2, j, s), (n, n2, j)
