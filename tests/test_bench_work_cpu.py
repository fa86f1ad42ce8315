"""The benchmark's algorithmic bytes of a finest-level Gauss-Seidel launch, counted by brute force: a
launch updates two colours, so the second one's new neighbours never come from memory, and nothing
but what a pass needs is charged to it.
"""
import itertools

import numpy as np
import pytest

import bench


def pass_bytes(n, pair, first):
    """Distinct bytes one launch reads and writes: E once, f and u of both colours, and the u of the
    neighbours that it does not itself produce (from zero: only those an earlier launch wrote)."""
    z, y, x = np.meshgrid(*[np.arange(n)] * 3, indexing="ij")
    colour = (x & 1) + 2 * (y & 1) + 4 * (z & 1)
    read = np.zeros((n, n, n), bool)
    for c, held in ((2 * pair, None), (2 * pair + 1, 2 * pair)):
        mine = colour == c
        for d in itertools.product((-1, 0, 1), repeat=3):
            if d != (0, 0, 0):
                need = np.roll(mine, d, axis=(0, 1, 2))
                read |= need & (colour != held) if held is not None else need
    if first:
        read &= colour < 2 * pair
    own = int(((colour >> 1) == pair).sum())
    return 4 * n ** 3 + 72 * int(read.sum()) + 72 * own + 72 * own


@pytest.mark.parametrize("sweeps", [1, 2])
def test_fine_gauss_seidel_bytes(sweeps):
    n = 8
    full = sum(pass_bytes(n, q, False) for q in range(4)) / 4
    from_zero = sum(pass_bytes(n, q, True) for q in range(4)) / 4
    want = (from_zero + (2 * sweeps - 1) * full) / (2 * sweeps)
    assert bench.algorithmic_work("fine_gs", n, sweeps)[0] == pytest.approx(want, rel=1e-12)
