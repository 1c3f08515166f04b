"""Z4c states whose tensor components differ by many orders of magnitude, against
the CPU oracle: every field's right-hand side and every constraint, relative to
that field's or constraint's own size."""
import numpy as np
import pytest

from helpers import make_oracle
from paper_2503_09629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# FP64 sums of a few hundred products of rough data, each relative to its own
# field's largest value: the tolerance of the ungraded states.
TOL = 1e-11

GT, AT, GAM, BETA = 1, 8, 14, 19
SYM = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]


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


def _state(h, kind, size):
    rng = np.random.default_rng(17)
    g = h.ghost
    s = 0.1 * rng.uniform(-1, 1, (22,) + tuple(n + 2 * g for n in h.ncells0[::-1]))
    if kind == "plane":  # data that vary along x only; 20 bits, so that the oracle's sums along y and z vanish exactly
        s = np.broadcast_to(np.round(s[:, :1, :1, :] * 2.0 ** 20) / 2.0 ** 20, s.shape).copy()
    for f in (0, 1, 4, 6, 18):
        s[f] += 1.0
    for c, (i, j) in enumerate(SYM):
        for t in (GT, AT):
            if kind.startswith("stretch"):
                axis = "xyz".index(kind[-1])
                s[t + c] *= size ** (((i == axis) + (j == axis)) / 2)
            elif kind == "offdiag" and i != j:
                s[t + c] *= size
            elif kind == "plane" and i != j:
                s[t + c] *= size if (i, j) == (1, 2) else 0.0
    if kind == "offdiag":
        s[BETA:BETA + 3] = 0.0
    if kind == "shift":
        s[BETA + 1:BETA + 3] *= size
    return s


STATES = ([("stretch_" + a, r) for a in "xyz" for r in (100.0, 1e6)] + [("offdiag", e) for e in (1e-4, 1e-8, 1e-12)] +
          [("shift", e) for e in (1e-4, 1e-8)] + [("plane", e) for e in (2.0 ** -13, 2.0 ** -26, 2.0 ** -40)])


def _load(ctx, state):
    setf = ctx.sc_set_field if hasattr(ctx, "sc_set_field") else ctx.set_field
    for f in range(22):
        setf(0, 0, f, state[f], ghosted=True)


def _close(got, ref, tol):
    for q in range(len(ref)):
        m = np.abs(ref[q]).max()
        # (subnormal results: a few hundred roundings at half of the last place, 2^-1075)
        assert np.abs(got[q] - ref[q]).max() <= tol * m + 256 * 2.0 ** -1074, (q, np.abs(got[q] - ref[q]).max(), m)


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("kind,size", STATES)
def test_rhs_of_graded_states(sc, orc, order, kind, size):
    h = _hierarchy(order)
    state = _state(h, kind, size)
    ctx = sc.Context(h)
    _load(ctx, state)
    ctx.sc_advance(1)
    got = np.stack([ctx.sc_debug_get_vector(0, 0, 4, f) for f in range(22)])  # k1
    ctx.close()
    g = h.ghost
    _close(got, make_oracle(orc, h).rhs_box(0, 0, state)[:, g:-g, g:-g, g:-g], TOL)


def _noalloc(sc, h, state):
    import torch
    n = h.ncells0
    dev = torch.from_numpy(state).cuda()
    out = torch.empty((7,) + n[::-1], dtype=torch.float64, device="cuda")
    sc.sc_z4c_constraints_noalloc(dev.data_ptr(), out.data_ptr(), n, h.h0, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("kind,size", STATES)
def test_constraints_of_graded_states(sc, orc, kind, size):
    h = _hierarchy(4)
    state = _state(h, kind, size)
    o = make_oracle(orc, h)
    _load(o, state)
    ref = o.constraints(0, 0)
    _close(_noalloc(sc, h, state), ref, TOL)
    ctx = sc.Context(h)
    _load(ctx, state)
    _close(ctx.sc_get_constraints(0, 0), ref, TOL)
    ctx.close()


@pytest.mark.parametrize("scale", [0.0, -0.0, 1e-30, 1e-200, 1e-320, 1e30, "mixed"])
def test_constraints_over_ranges(sc, orc, scale):
    """K, Theta, At, Gamt and the off-diagonal metric scaled together, or cell by cell."""
    h = _hierarchy(4)
    state = _state(h, "ranges", 1.0)
    if scale == "mixed":
        scale = np.random.default_rng(3).choice([1.0, 0.0, 1e-290, 1e-60, 1e-12], size=state.shape[1:])
    for f in [2, 3, 5, 7] + list(range(8, 18)):
        state[f] *= scale
    o = make_oracle(orc, h)
    _load(o, state)
    _close(_noalloc(sc, h, state), o.constraints(0, 0), TOL)


@pytest.mark.parametrize("field", [0, 1, 2, 6])
@pytest.mark.parametrize("value", [np.inf, np.nan, 1.5e307])
def test_constraints_not_finite_where_a_second_derivative_overflows(sc, orc, field, value):
    """Two equal neighbours of a cell: its first derivative is unchanged if they are finite,
    its second derivative leaves the range of doubles, and so does the Hamiltonian constraint."""
    h = _hierarchy(4)
    state = _state(h, "ranges", 1.0)
    z, y, x = 5, 4, 6
    state[field, 3 + z, 3 + y, 3 + x - 1] = state[field, 3 + z, 3 + y, 3 + x + 1] = value
    got = _noalloc(sc, h, state)
    assert not np.isfinite(got[0, z, y, x])
    far = np.ones(got.shape[1:], dtype=bool)
    far[z - 2:z + 3, y - 2:y + 3, x - 3:x + 4] = False
    clean = _state(h, "ranges", 1.0)
    assert np.array_equal(got[:, far], _noalloc(sc, h, clean)[:, far])
