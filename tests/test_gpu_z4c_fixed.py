"""The Z4c right-hand side in block fixed point against the CPU oracle, where it
can go wrong: blocks of zeros of either sign, blocks far below and above the
others, blocks outside the range that the fixed-point form accepts (left to the
FP64 form, cell by cell), neighbouring cells of different ranges, NaN and
infinity.  The data are rough (white noise), so every term counts."""
import numpy as np
import pytest

from helpers import make_oracle
from paper_2503_09629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# The terms of a right-hand side are sums of a few hundred products; with 1e-16
# per operation and at most 1e3 times the result's largest value among them, a
# correct evaluation stays two orders below this.
TOL = 1e-11


@pytest.fixture(scope="module")
def sc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_09629_gb300 as m
    m.build()
    return m


def _hierarchy(order):
    n = (13, 9, 11)
    return W.Hierarchy(system=W.Z4C, boxes=[[((0, 0, 0), tuple(v - 1 for v in n))]], ncells0=n, origin=(-1.7, -1.2, -1.4),
                       h0=0.25, bc=W.BC_RADIATIVE, fd_order=order)


def _state(h):
    rng = np.random.default_rng(7)
    g = h.ghost
    s = 0.1 * rng.uniform(-1, 1, (22,) + tuple(n + 2 * g for n in h.ncells0[::-1]))
    for f in (0, 1, 4, 6, 18):
        s[f] += 1.0
    return s


def _k1(sc, h, state):
    ctx = sc.Context(h)
    for f in range(22):
        ctx.sc_set_field(0, 0, f, state[f], ghosted=True)
    ctx.sc_advance(1)
    k = np.stack([ctx.sc_debug_get_vector(0, 0, 4, f) for f in range(22)])
    ctx.close()
    return k


def _oracle(orc, h, state):
    g = h.ghost
    return make_oracle(orc, h).rhs_box(0, 0, state)[:, g:-g, g:-g, g:-g]


SCALED = {"matter": [7] + list(range(8, 14)) + [17], "shift": list(range(14, 17)) + list(range(19, 22))}


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("which", sorted(SCALED))
@pytest.mark.parametrize("scale", [1.0, 0.0, -0.0, 1e-30, 1e-200, 1e-280, 1e30, 1e50, "mixed"])
def test_rhs_matches_oracle(sc, orc, order, which, scale):
    h = _hierarchy(order)
    state = _state(h)
    if scale == "mixed":
        scale = np.random.default_rng(3).choice([1.0, 0.0, 1e-290, 1e-60, 1e20, 1e48], size=state.shape[1:])
    for f in SCALED[which]:
        state[f] *= scale
    got, ref = _k1(sc, h, state), _oracle(orc, h, state)
    for f in range(22):
        m = np.abs(ref[f]).max()
        assert np.abs(got[f] - ref[f]).max() <= TOL * m, (f, np.abs(got[f] - ref[f]).max(), m)


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_non_finite_values_stay_local(sc, orc, value):
    """A non-finite value reaches the right-hand side of its field within the
    dissipation stencil, and nothing outside the widest stencil."""
    h = _hierarchy(4)
    state = _state(h)
    g = h.ghost
    z, y, x = 5, 4, 6
    ref = _oracle(orc, h, state)
    for f in (0, 3, 9, 20):
        bad = state.copy()
        bad[f, g + z, g + y, g + x] = value
        got = _k1(sc, h, bad)
        for d in range(-3, 4):
            assert not np.isfinite(got[f, z, y, x + d])
        far = np.ones(got.shape[1:], dtype=bool)
        far[z - 3:z + 4, y - 3:y + 4, x - 3:x + 4] = False
        for q in range(22):
            assert np.abs(got[q] - ref[q])[far].max() <= TOL * np.abs(ref[q]).max(), (f, q)
