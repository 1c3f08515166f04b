"""The integer stencil sums where values differ by many orders of magnitude from one
cell to the next along one axis: each sum as accurate as its own weighted terms."""
from fractions import Fraction

import numpy as np
import pytest

from helpers import make_oracle
from paper_2503_09629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

WEIGHTS = {4: (12, -90, (16, -1)), 8: (5040, -43050, (8064, -1008, 128, -9))}
# Largest error over the sum of the weighted values' magnitudes.  4th order: at most one unit
# of 2^-54 of the largest of 13 values for each, and three roundings: 16 2^-54.  8th order:
# weights of 98304 in all times 2^-58 of the largest value, which is below 2^6 of a value of
# weight 8064 or more where integers are used: 2^-48.4; FP64 chains are below that.
BOUND = {4: 2.0 ** -50, 8: 2.0 ** -48}


@pytest.fixture(scope="module")
def sc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_09629_gb300 as m
    m.build()
    return m


def _steep(rng, shape, axis, bits):
    """Random values, 2^bits larger from cell to cell along one axis (of z, y, x), 1 at the largest."""
    n = shape[axis]
    s = 2.0 ** (bits * (np.arange(n) - (n - 1.0)))
    return rng.uniform(0.5, 1.0, shape) * rng.choice([-1.0, 1.0], shape) * s.reshape([-1 if a == axis else 1 for a in range(3)])


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("bits", [0, 1, 3, 10, "mixed", "large"])
def test_laplacian_against_exact_sums(sc, order, axis, bits):
    n = 16
    h = W.Hierarchy(system=W.WAVE, boxes=[[((0, 0, 0), (n - 1,) * 3)]], ncells0=(n,) * 3, origin=(0.0,) * 3, h0=1.0 / n,
                    fd_order=order)
    rng = np.random.default_rng(5)
    if bits == "mixed":  # inside and outside of the range of the integers, cell by cell
        u = rng.uniform(-1, 1, (n,) * 3) * rng.choice([1.0, 1.0, 0.0, 1e-290, 1e-200, 1e-20], size=(n,) * 3)
    elif bits == "large":
        u = rng.uniform(-1, 1, (n,) * 3) * rng.choice([1e300, 1e290, 1.0, -0.0], size=(n,) * 3)
    else:
        u = _steep(rng, (n,) * 3, axis, bits)
    ctx = sc.Context(h)
    ctx.sc_set_field(0, 0, 0, u)
    ctx.sc_set_field(0, 0, 1, np.zeros_like(u))
    ctx.sc_advance(1)
    got = ctx.sc_debug_get_vector(0, 0, 4, 1)  # k1 of Pi
    ctx.close()
    den, w0, w = WEIGHTS[order]
    exact = np.vectorize(Fraction, otypes=[object])(u)
    lap, size = w0 * exact, -w0 * abs(exact)
    for d in range(3):
        for m, c in enumerate(w, 1):
            for s in (m, -m):
                v = np.roll(exact, s, axis=d)
                lap, size = lap + c * v, size + abs(c) * abs(v)
    scale = Fraction(n * n, den)
    worst = max(abs(Fraction(g) - a * scale) / (t * scale) for g, a, t in zip(got.flat, lap.flat, size.flat) if t)
    assert not any(g for g, t in zip(got.flat, size.flat) if not t)
    assert float(worst) <= BOUND[order]


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("steep,along", [(0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1)])
@pytest.mark.parametrize("bits", [2, 10])
def test_derivative_beside_a_steep_gradient(sc, orc, order, steep, along, bits):
    """Theta, 2^bits larger from cell to cell along one axis, advected along another by a constant
    shift in flat space without dissipation: its right-hand side is that derivative and
    4/3 Theta^2, cell by cell against the oracle, relative to Theta's size there."""
    n = (11, 10, 12)
    h = W.Hierarchy(system=W.Z4C, boxes=[[((0, 0, 0), tuple(v - 1 for v in n))]], ncells0=n, origin=(0.0,) * 3, h0=0.25,
                    bc=W.BC_RADIATIVE, fd_order=order, ko_sigma=0.0, kappa1=0.0)
    g = h.ghost
    shape = tuple(v + 2 * g for v in n[::-1])
    state = np.zeros((22,) + shape)
    for f in (0, 1, 4, 6, 18):
        state[f] = 1.0
    state[17] = theta = _steep(np.random.default_rng(9), shape, steep, bits)
    state[19 + 2 - along] = 1.0  # axes are z, y, x
    ctx = sc.Context(h)
    for f in range(22):
        ctx.sc_set_field(0, 0, f, state[f], ghosted=True)
    ctx.sc_advance(1)
    got = ctx.sc_debug_get_vector(0, 0, 4, 17)
    ctx.close()
    ref = make_oracle(orc, h).rhs_box(0, 0, state)[17]
    inner = (slice(g, -g),) * 3
    size = np.max([np.abs(np.roll(theta, m, axis=along)) for m in range(-g, g + 1)], axis=0)[inner] / h.h0
    # ten roundings of 2^-53 of terms of at most twice that size, in either evaluation
    assert np.max(np.abs(got - ref[inner]) / size) <= 40 * 2.0 ** -53
