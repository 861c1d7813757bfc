"""The streaming sparse kernel at the edges of its work split."""
import numpy as np
import pytest

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec_name", ["PREC_FP32", "PREC_BF16"])
@pytest.mark.parametrize("N,R,steps", [(3, 1, 4), (40, 700, 5), (6000, 520, 3), (700, 33, 150)])
def test_cell_ranges(orc, prec_name, N, R, steps):
    """CTA ranges that start inside a row, more cells than shared memory holds, rows too
    many or too dense for the staged lists, replicas that leave a ragged vector: against the
    oracle (the tolerances of the resident kernels)."""
    import torch  # noqa: F401

    from paper_2004_03972_gb300 import hqa
    inst = instances.er_mean_degree_pm1(N, min(N - 1, 8 if N != 40 else 39), 5)
    ctx = hqa.Context.from_instance(inst)
    out = ctx.run(steps, R, seed=4, dt=1e-4, precision=getattr(hqa, prec_name),
                  kernel=hqa.KERNEL_STREAM, outputs=("phi", "p", "phibar"))
    ctx.sync()
    pr = orc.Problem.from_instance(inst)
    tol = 1e-5 if prec_name == "PREC_FP32" else 1e-2
    for r in sorted({0, R // 2, R - 1}):
        want = orc.md_run(pr, steps, dt=1e-4, p0=orc.initial_momenta(4, r, N))
        for k, w in zip(("phi", "p", "phibar"), want):
            scale = max(np.max(np.abs(w)), 1.0 if k == "p" else 0.0)
            assert np.max(np.abs(out[k][r].cpu().numpy() - w)) <= tol * scale
    ctx.close()
