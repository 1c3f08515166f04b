"""The autotuner times the path that a run takes, and leaves nothing behind."""
import numpy as np
import pytest

from helpers import fetch
from paper_2503_09629_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_09629_gb300 as m
    m.build()
    return m


def test_timed_stage_of_a_new_context_is_finite(sc):
    """A new context's arrays are zero, a singular metric: the stage that is timed has a regular one."""
    h = W.bl_3level(20, m1=0.41)
    h.boxes = [h.boxes[0]]
    ctx = sc.Context(h)
    _tile, ms = ctx.sc_autotune()
    assert ms > 0
    for f in range(22):
        assert np.isfinite(ctx.sc_debug_get_vector(0, 0, 5, f)).all()  # k2
        assert not ctx.sc_debug_get_vector(0, 0, 2, f).any()  # the stage buffer is as at creation
    ctx.close()


@pytest.mark.parametrize("order", [4, 8])
def test_tuned_run_is_bitwise_the_run_with_the_same_settings(sc, order):
    h = W.bl_3level(32 if order == 8 else 20, m1=0.37)
    h.fd_order = order
    out, choice = [], None
    for tune in (True, False):
        ctx = sc.Context(h)
        if not tune:
            ctx.sc_set_tuning(*choice)
        ctx.sc_set_initial_data(h.id_kind, h.id_params)
        if tune:
            ctx.sc_autotune()
            t = ctx.sc_get_tuning()
            choice = (t["tile"], t["deriv_form"], t["stage_blocks_per_sm"])
        ctx.sc_advance(1)
        if tune:
            ctx.sc_autotune()
        ctx.sc_advance(1)
        out.append(fetch(ctx, h))
        ctx.close()
    for la, lb in zip(*out):
        for a, b in zip(la, lb):
            assert np.array_equal(a, b)
