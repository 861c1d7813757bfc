"""Window means of fluxes around the smallest normal number, in every kernel that sums them by
reductions: a table schedule with alpha = beta = 0 keeps phi, so the mean of four steps is phi
itself (four times phi is exact, and so is a quarter of it)."""
import numpy as np
import pytest

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel,prec_name,N,R", [
    ("KERNEL_DENSE", "PREC_FP32", 200, 40), ("KERNEL_DENSE", "PREC_BF16", 200, 40),
    ("KERNEL_DENSE", "PREC_FP16X2", 300, 70), ("KERNEL_DENSE", "PREC_BF16", 4993, 1030),
    ("KERNEL_DENSE", "PREC_BF16", 2500, 2200),
    ("KERNEL_STREAM", "PREC_FP32", 700, 33), ("KERNEL_STREAM", "PREC_BF16", 700, 33)])
def test_means_of_tiny_fluxes(kernel, prec_name, N, R):
    import torch

    from paper_2004_03972_gb300 import hqa
    inst = instances.er_mean_degree_pm1(N, 8, 1) if kernel == "KERNEL_STREAM" else instances.sk_pm1(N, 1)
    ctx = hqa.Context.from_instance(inst)
    g = torch.Generator("cuda").manual_seed(N)
    e = torch.randint(-146, -95, (R, N), generator=g, device="cuda").double()
    phi = (torch.where(torch.rand(R, N, generator=g, device="cuda") < 0.5, -1.0, 1.0).double()
           * torch.exp2(e)).float()
    phi[:, ::7] = -1e-40
    z = torch.zeros_like(phi)
    out = ctx.run(4, R, sched=hqa.schedule(window=4), table=(np.zeros(11), np.zeros(6)), dt=1e-4,
                  precision=getattr(hqa, prec_name), kernel=getattr(hqa, kernel), start_step=1,
                  init=hqa.INIT_GIVEN, phi0=phi, p0=z, outputs=("phi", "phibar", "spins"))
    ctx.sync()
    bits = lambda t: t.contiguous().view(torch.int32)
    assert torch.equal(bits(out["phi"]), bits(phi))
    assert torch.equal(bits(out["phibar"]), bits(phi))
    assert torch.equal(out["spins"] < 0, phi < 0)
    ctx.close()
