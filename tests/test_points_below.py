"""The count of systematic points below a cumulative count by one 64-bit product (points_below in
dpf_resample.cuh) gives the exact rule's count, or leaves the value to the exact comparisons,
for every scale it accepts: K(c) = #{k in [0, n): (k 2^32 + u) C < c n 2^32}.

The rule is restated here in unbounded integers, with the kernel's truncations.
"""
import random


def _exact(c, n, u, C):
    # the first k with (k 2^32 + u) C >= c n 2^32
    need = -(-(c * n << 32) // C) - u
    return max(0, min(n, -(-need >> 32) if need > 0 else 0))


def _scale(n, C):
    q = C // n
    f = q.bit_length() - 2 if q else -1  # 62 - clz(q)
    if f < 8:
        return None
    f = min(f, 32)
    F = (n << (64 + f)) // C
    assert F < 1 << 64
    return F, f


def _quick(c, n, u, F, f):
    """The product's answer, or None where the kernel takes the exact comparisons."""
    d = (c * F >> 64) - (u >> (32 - f))
    if d >= 1:
        r, k = (d - 1) & ((1 << f) - 1), ((d - 1) >> f) + 1
        return min(k, n) if r + 3 <= 1 << f else None
    return 0 if d <= -2 else None


def test_exact_or_undecided():
    rng = random.Random(3)
    decided = total = 0
    for _ in range(4000):
        n = int(2 ** rng.uniform(0, 31))
        C = int(2 ** rng.uniform(0, 62)) + 1
        s = _scale(n, C)
        if s is None:
            assert C // n < 1 << 10
            continue
        us = [0, 1, (1 << 32) - 1, rng.getrandbits(32), rng.getrandbits(32)]
        for u in us:
            cs = [1, 2, C - 1, C, rng.randint(1, C)]
            k = rng.randrange(n)  # counts at and beside a point
            at = ((k << 32) + u) * C // (n << 32)
            cs += [min(max(at + e, 1), C) for e in (-1, 0, 1, 2)]
            for c in cs:
                got = _quick(c, n, u, *s)
                total += 1
                if got is not None:
                    decided += 1
                    assert got == _exact(c, n, u, C), (c, n, u, C)
    assert decided > total / 3
