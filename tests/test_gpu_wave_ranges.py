"""The scalar wave's integer sums (Laplacian and refinement-boundary
prolongation) against the CPU oracle where values leave the range that they
take: scaled below and above it, and cell by cell, so that one stencil mixes
both forms; and a ragged, narrow hierarchy, whose tiles are cut at every side."""
import numpy as np
import pytest

from helpers import fetch, init_arrays, load, make_oracle, max_rel_diff
from paper_2503_09629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# One coarse step of a linear scheme: a few hundred roundings of 1e-16 per value.
TOL = 1e-12


@pytest.fixture(scope="module")
def sc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_09629_gb300 as m
    m.build()
    return m


def _hierarchy(order, ragged):
    if not ragged:
        h = W.standing_wave_2level(24)
        h.fd_order = order
        return h
    return W.Hierarchy(system=W.WAVE, boxes=[[((0, 0, 0), (32, 20, 24))], [((22, 12, 14), (41, 27, 33))]],
                       ncells0=(33, 21, 25), origin=(0.0, 0.0, 0.0), h0=1.0 / 33, fd_order=order,
                       id_params=[1.0, 1.0, 1.0, 1.0])


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("scale", [1.0, 0.0, 1e-285, 1e-270, 1e270, "mixed"])
@pytest.mark.parametrize("ragged", [False, True])
def test_wave_matches_oracle(sc, orc, order, scale, ragged):
    h = _hierarchy(order, ragged)
    rng = np.random.default_rng(11)
    arrays = [[rng.uniform(-1, 1, a.shape) for a in level] for level in init_arrays(h)]
    for level in arrays:
        for a in level:
            a *= scale if scale != "mixed" else rng.choice([1.0, 0.0, 1e-290, 1e-200, 1e-20], size=a.shape)
    ctx, o = sc.Context(h), make_oracle(orc, h)
    load(ctx, h, arrays)
    load(o, h, arrays)
    ctx.sc_advance(1)
    o.advance(1)
    assert max_rel_diff(fetch(ctx, h), fetch(o, h), floor=1e-300) <= TOL
    ctx.close()
