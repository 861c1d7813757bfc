"""The 256 x 256 units of the large-instance dense kernel: bit for bit the runs of few replicas,
which take the kernel with one CTA per row tile; odd row tiles, ragged last rows and columns,
1, 2 and 3 products, both 16-bit formats, window sums; and its bounded wait.  With a field the
two kernels may fuse 2 h |phi| into the sum in either order, one rounding of the field apart:
there the 22-bit operand is compared to 2e-6 (7 steps of 2^-24 on kB L < 2 and the operand's
2^-22, amplified by less than 1.5)."""
import pytest

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,N,R,prec_name", [
    ("sk", 4993, 1030, "PREC_FP16X2"), ("sk", 4993, 1030, "PREC_BF16"), ("sk", 5100, 1500, "PREC_FP16"),
    ("sg", 4900, 1000, "PREC_BF16X2"), ("sgh", 4900, 1000, "PREC_FP16X2"), ("sk", 5377, 770, "PREC_BF16X2")])
def test_equals_small_runs(kind, N, R, prec_name):
    import torch

    from paper_2004_03972_gb300 import hqa
    inst = instances.uniform_sg(N, 3) if kind.startswith("sg") else instances.sk_pm1(N, 3)
    if kind == "sg":
        inst.h = None
    ctx = hqa.Context.from_instance(inst)
    prec = getattr(hqa, prec_name)
    assert ctx.plan(R, precision=prec)["threads"] == 320 and ctx.plan(40, precision=prec)["threads"] == 448
    g = torch.Generator("cuda").manual_seed(N)
    phi0 = 2.0 * torch.rand(R, N, generator=g, device="cuda") - 1.0
    p0 = torch.rand(R, N, generator=g, device="cuda") - 0.5
    kw = dict(dt=1e-4, precision=prec, init=hqa.INIT_GIVEN, start_step=4000,
              sched=hqa.schedule(window=4), outputs=("phi", "p", "phibar"))
    big = ctx.run(7, R, phi0=phi0, p0=p0, **kw)
    ctx.sync()
    for r0 in (0, 250, R - 40):
        a, b = phi0[r0:r0 + 40].contiguous(), p0[r0:r0 + 40].contiguous()
        few = ctx.run(7, 40, phi0=a, p0=b, **kw)
        ctx.sync()
        for k in few:
            if kind == "sgh":
                assert (few[k] - big[k][r0:r0 + 40]).abs().max() <= 2e-6 * few[k].abs().max()
            else:
                assert torch.equal(few[k], big[k][r0:r0 + 40])
    ctx.close()


def test_wait_runs_out():
    import torch

    from paper_2004_03972_gb300 import hqa
    ctx = hqa.Context.from_instance(instances.sk_pm1(5000, 1))
    kw = dict(seed=2, dt=1e-4, precision=hqa.PREC_BF16, outputs=("phi", "p"))
    want = ctx.run(5, 1000, **kw)
    ctx.sync()
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    ctx.arm_wait_check(flag, 2, 50_000_000)
    ctx.run(5, 1000, **kw)
    with pytest.raises(hqa.HQAError) as e:
        ctx.sync()
    assert e.value.status == 8
    again = ctx.run(5, 1000, **kw)
    ctx.sync()
    assert all(torch.equal(again[k], want[k]) for k in want)
    ctx.close()
