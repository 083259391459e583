"""The cubic nested guess (csrc/guess.cuh, k_guess2, k_guess3), replayed on the
CPU: the weights reproduce cubic polynomials at every fine node, ends of the
axis included; the window of four coarse slabs a strip carries holds the ones
its fine slab needs wherever the strip starts; and the lanes of a warp hold
the coarse columns their odd fine column takes, each fine column being made
once."""
import numpy as np
import pytest

HALO, COLS = 2, 27


def base(I, nc):
    return 0 if I == 0 else (nc - 3 if I >= nc - 1 else I - 1)


def mid(I, nc, a, b, c, d):
    if I == 0:
        w = (0.3125, 0.9375, -0.3125, 0.0625)
    elif I == nc - 1:
        w = (0.0625, -0.3125, 0.9375, 0.3125)
    else:
        w = (-0.0625, 0.5625, 0.5625, -0.0625)
    return w[0] * a + w[1] * b + w[2] * c + w[3] * d


@pytest.mark.parametrize("nc", [4, 5, 8, 32, 33])
def test_window_and_weights_reproduce_cubics(nc):
    rng = np.random.default_rng(nc)
    p = np.polynomial.Polynomial(rng.standard_normal(4))
    coarse, n = p(np.arange(nc + 1) / nc), 2 * nc
    for z0 in range(0, n + 1):
        b = base(z0 >> 1, nc)
        v = [coarse[b + k] for k in range(4)]
        for z in range(z0, n + 1):
            nb = base(z >> 1, nc)
            while b < nb:   # k_guess3 advances by one coarse slab through fine slab 2 (b + 2)
                assert base(((b + 2) * 2) >> 1, nc) == b + 1
                v = v[1:] + [coarse[b + 4]]
                b += 1
            I = z >> 1
            assert b == nb and 0 <= b <= nc - 3
            got = mid(I, nc, *v) if z & 1 else v[I - b]
            assert 0 <= I - b <= 3
            assert abs(got - p(z / n)) <= 1e-13 * (1 + abs(p(z / n)))


@pytest.mark.parametrize("nc", [4, 13, 26, 27, 28, 54, 100])
def test_lanes_hold_their_neighbours(nc):
    coarse = np.arange(nc + 1) ** 3 * 1.0 - 5.0 * np.arange(nc + 1)
    made = set()
    for strip in range((nc + COLS) // COLS):
        I0 = strip * COLS - HALO
        col = [I0 + k for k in range(32)]
        val = [coarse[c] if 0 <= c <= nc else 0.0 for c in col]
        for lane in range(HALO, HALO + COLS):
            I = col[lane]
            if not 0 <= I <= nc:
                continue
            assert 2 * I not in made
            made.add(2 * I)
            if I == nc:
                continue
            made.add(2 * I + 1)
            m2, m1, v, p1, p2, p3 = (val[lane + k] if 0 <= lane + k < 32 else None for k in range(-2, 4))
            four = (v, p1, p2, p3) if I == 0 else ((m2, m1, v, p1) if I == nc - 1 else (m1, v, p1, p2))
            b = base(I, nc)
            assert list(four) == [coarse[b + k] for k in range(4)]
            assert abs(mid(I, nc, *four) - ((I + 0.5) ** 3 - 5.0 * (I + 0.5))) <= 1e-9 * (1 + I) ** 3
    assert made == set(range(2 * nc + 1))
