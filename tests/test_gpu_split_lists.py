"""One replica per CTA of a small instance: the lists shared by the warps give the bits of a warp
per tuple, which one replica more than SMs takes, and are not slower."""
import pytest

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu


def _run(hqa, ctx, R, S, prec=0):
    return ctx.run(S, R, seed=1, dt=1e-4, precision=prec, kernel=hqa.KERNEL_SCALAR,
                   replicas_per_block=1, outputs=("phi", "p", "phibar"))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N,degree", [(16, 4), (100, 20), (200, 12), (250, 8), (256, 3), (256, 80)])
def test_same_bits(N, degree, prec):
    import torch

    from paper_2004_03972_gb300 import hqa
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctx = hqa.Context.from_instance(instances.er_mean_degree_pm1(N, degree, 1))
    shared, own = _run(hqa, ctx, sms, 120, prec), _run(hqa, ctx, sms + 1, 120, prec)
    ctx.sync()
    assert all(torch.equal(shared[k], own[k][:sms]) for k in shared)
    ctx.close()


def test_short_lists():
    """N = 250 of mean degree 8: 0.49 us a step with four chunks per warp, 0.66 with a warp per
    tuple, 0.75 with a warp per chunk."""
    import torch

    from paper_2004_03972_gb300 import hqa
    ctx = hqa.Context.from_instance(instances.er_mean_degree_pm1(250, 8, 1))
    ms = {}
    for S in (100, 2100):
        _run(hqa, ctx, 1, S)
        ms[S] = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            _run(hqa, ctx, 1, S)
            b.record()
            torch.cuda.synchronize()
            ms[S] = min(ms[S], a.elapsed_time(b))
    assert (ms[2100] - ms[100]) / 2000 <= 0.60e-3
    ctx.close()
