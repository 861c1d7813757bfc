"""The FP32 operands of a dense context: built at create when asked for, and not needed by a
plan query, which a capture may contain."""
import numpy as np
import pytest

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu


def _glass(N, kind="sg"):
    inst = instances.uniform_sg(N, 5)
    inst.h = None
    if kind == "eighths":       # one BF16 slice, though not whole numbers
        inst.dense = np.sign(inst.dense) * 0.125
    return inst


def test_flag_builds_what_a_run_reads():
    """N = 2000: the slices take 25 MB, the state of one replica below 1 MB."""
    import torch

    from paper_2004_03972_gb300 import hqa
    ctx = hqa.Context.from_instance(_glass(2000), hqa.J_FP32)
    out = {k: torch.empty(1, 2000, device="cuda") for k in ("phi", "p")}
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx.run(2, 1, dt=1e-4, kernel=hqa.KERNEL_DENSE, out=out)
    ctx.sync()
    assert free - torch.cuda.mem_get_info()[0] <= 8 << 20
    ctx.close()


@pytest.mark.parametrize("kind", ["sg", "eighths"])
def test_plan_during_a_capture(kind):
    import torch

    from paper_2004_03972_gb300 import hqa
    ctx = hqa.Context.from_instance(_glass(256, kind))
    with hqa.capture(torch.cuda.Stream()) as cap:
        during = ctx.plan(2000, kernel=hqa.KERNEL_DENSE)
    cap.graph.close()
    ctx.run(2, 2000, dt=1e-4, kernel=hqa.KERNEL_DENSE, outputs=("phi",))
    ctx.sync()
    assert during == ctx.plan(2000, kernel=hqa.KERNEL_DENSE)
    ctx.close()
