"""sc_run_op_class_pass launches the op-class build of every kernel of a Z4c stage."""
import pytest

from paper_2503_09629_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [4, 8])
def test_every_kernel_of_the_pass_is_the_op_class_build(order):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_09629_gb300 as sc
    sc.build()
    h = W.bl_3level(32)
    h.fd_order = order
    ctx = sc.Context(h)
    ctx.sc_set_initial_data(h.id_kind, h.id_params)
    ctx.sc_advance(1)
    ctx.sc_synchronize()

    def names():
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            ctx.sc_run_op_class_pass(1)
            torch.cuda.synchronize()
        return [e.name for e in prof.events() if "z4c_" in e.name]

    names()  # (the first profile of a process can miss its first launches)
    names = names()
    ctx.close()
    for kernel in ("z4c_dxy_kernel", "z4c_derivs_split_kernel", "z4c_stage_kernel"):
        assert [("PlainK" in n) for n in names if kernel in n] == [True], names
