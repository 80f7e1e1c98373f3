"""bench.py's count of the convolution's pairs: those with a weight, entry by entry over the stored
pencils, and the entries of weight 0 beside them."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    sys.path.insert(0, ROOT)
    try:
        import bench as b
    finally:
        sys.path.remove(ROOT)
    return b


@pytest.mark.parametrize("n", [8, 12])
def test_pairs_with_a_weight(bench, n):
    h = n // 2

    def held(k, m):  # zeta - xi on the mesh in every dimension
        return all(0 <= a - b + h < n for a, b in zip(k, m))

    def mirror(v):
        return tuple((n - x) % n for x in v)

    pairs = zero = 0
    for k1 in range(n):
        for k2 in range(n):
            if (k1, k2) < mirror((k1, k2)):  # of a mirror pair the pencil with the larger index
                continue
            for m1 in range(n):
                for m2 in range(n):
                    if (m1, m2) > ((k1 - m1 + h) % n, (k2 - m2 + h) % n):
                        continue
                    block = [held((k1, k2, k3), (m1, m2, m3)) or held(mirror((k1, k2, k3)), mirror((m1, m2, m3)))
                             for k3 in range(n) for m3 in range(n)]
                    if any(block):  # the kernel visits every (k3, m3) that some block holds
                        pairs += sum(block)
                        zero += sum(held((k3,), (m3,)) or held(mirror((k3,)), mirror((m3,)))
                                    for k3 in range(n) for m3 in range(n)) - sum(block)
    assert bench.conv_pairs_per_cell(n) == (pairs, zero)
