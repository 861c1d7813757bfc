"""Few replicas of a small instance (lists split over all warps) at the kernel's edges: one to
eight tuples of 32 rows, offsets in registers and not, empty rows, fields, both operands.
Against the FP64 oracle (tolerances of the resident sparse kernels, 1e-5 and 1e-2), and bit for
bit against the same replicas run by more CTAs than there are SMs, which the unsplit kernel takes."""
import numpy as np
import pytest

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec_name,tol", [("PREC_FP32", 1e-5), ("PREC_BF16", 1e-2)])
@pytest.mark.parametrize("kind,N,R", [("sk", 1, 1), ("sk", 2, 3), ("sk", 20, 2), ("sk", 33, 1),
                                      ("er", 90, 3), ("skh", 100, 2), ("sk", 129, 1), ("sk", 256, 1),
                                      ("er", 200, 1), ("er", 256, 3), ("torus", 36, 2), ("none", 7, 1)])
def test_against_oracle(orc, kind, N, R, prec_name, tol):
    import torch

    from paper_2004_03972_gb300 import hqa
    if kind == "er":
        inst = instances.er_pm1(N, 0.03, N)
    elif kind == "torus":
        inst = instances.torus_pm1(6, 6, 2)
    elif kind == "none":
        inst = instances.Instance("none", N, row_ptr=np.zeros(N + 1, np.int64),
                                  col=np.zeros(0, np.int32), val=np.zeros(0, np.float32))
    else:
        inst = instances.er_pm1(N, 1.0, N)
    if kind == "skh":
        inst = instances.with_integer_field(inst, 3, 1)
    ctx = hqa.Context.from_instance(inst)
    prec = getattr(hqa, prec_name)
    kw = dict(precision=prec, dt=1e-4, outputs=("phi", "p", "phibar"), kernel=hqa.KERNEL_SCALAR,
              replicas_per_block=1)
    for init in (hqa.INIT_PAPER, hqa.INIT_RANDOM_FLUX):
        out = ctx.run(100, R, seed=6, init=init, sched=hqa.schedule(window=30), **kw)
        ctx.sync()
        many = ctx.run(100, 400, seed=6, init=init, sched=hqa.schedule(window=30), **kw)
        ctx.sync()
        assert all(torch.equal(out[k], many[k][:R]) for k in out)
        pr = orc.Problem.from_instance(inst)
        for r in sorted({0, R - 1}):
            f0 = orc.initial_flux_random(6, r, N) if init == hqa.INIT_RANDOM_FLUX else None
            want = orc.md_run(pr, 100, dt=1e-4, phi0=f0, p0=orc.initial_momenta(6, r, N), window=30)
            for k, w in zip(("phi", "p", "phibar"), want):
                scale = max(np.max(np.abs(w)), 1.0 if k == "p" else 0.0)
                assert np.max(np.abs(out[k][r].cpu().numpy() - w)) <= tol * scale
    ctx.close()
