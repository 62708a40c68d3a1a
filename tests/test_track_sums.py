"""CPU model of the tracker's shared warp sums: the exchange gives every lane the bits of a plain xor
butterfly per value, and every value ends in one lane."""
import numpy as np
import pytest


def sum_lane(k, n):
    lane = 0
    for m in (16, 8, 4, 2, 1):
        half = (n + 1) // 2
        if k >= half:
            lane |= m
            k -= half
        n = half
    return lane


def exchange(v):
    lanes = np.arange(32)
    t = [x.copy() for x in v]
    n = len(v)
    for m in (16, 8, 4, 2, 1):
        half = (n + 1) // 2
        up = (lanes & m) != 0
        new = list(t)
        for i in range(half):
            if i + half < n:
                keep, send = np.where(up, t[i + half], t[i]), np.where(up, t[i], t[i + half])
                new[i] = keep + send[lanes ^ m]
            else:
                new[i] = t[i] + t[i][lanes ^ m]
        t, n = new, half
    return [t[0][sum_lane(k, len(v))] for k in range(len(v))]


@pytest.mark.parametrize("n", [1, 2, 3, 5, 9, 10])
def test_exchange_equals_butterflies(n):
    rng = np.random.default_rng(n)
    v = [(rng.standard_normal(32) * 10.0 ** rng.integers(-3, 4)).astype(np.float32) for _ in range(n)]
    for got, x in zip(exchange(v), v):
        s = x.copy()
        for m in (16, 8, 4, 2, 1):
            s = s + s[np.arange(32) ^ m]
        assert (s == s[0]).all() and got.tobytes() == s[0].tobytes()
