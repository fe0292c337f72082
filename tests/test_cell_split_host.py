"""The particle kernels split a cell index into (row, column) with one multiply-high and a shift by
host-made constants. Checked here against integer division at the places where a reciprocal goes wrong: around the
multiples of nx up to the largest cell index, for every nx up to 512 and a spread up to the largest."""
import numpy as np


def magic(nx):
    """The constants make_step_args forms: 2^s < nx <= 2^(s + 1), m = ceil(2^(32 + s) / nx)."""
    s = 0
    while (2 << s) < nx:
        s += 1
    return (2 ** (32 + s) + nx - 1) // nx, s


def test_split_is_exact_at_the_edges():
    rng = np.random.default_rng(5)
    sizes = list(range(3, 513)) + [2 ** b + d for b in range(9, 15) for d in (-1, 0, 1)] + [32766, 32767] + \
        rng.integers(513, 32767, 300).tolist()
    for nx in sizes:
        m, s = magic(nx)
        assert m < 2 ** 32
        top = min(2 ** 31 - 1, nx * 32767)
        q = np.unique(np.concatenate([np.arange(0, 40), rng.integers(0, top // nx, 200), [top // nx]])).astype(np.uint64)
        cell = np.concatenate([q * np.uint64(nx) + np.uint64(d) for d in (0, 1, nx - 1)] + [np.array([top], np.uint64)])
        cell = cell[cell <= top]
        hi = (cell * np.uint64(m)) >> np.uint64(32)          # cell < 2^31, m < 2^32: no overflow in 64 bits
        assert np.array_equal(hi >> np.uint64(s), cell // np.uint64(nx)), nx
