"""Few replicas of a small complete graph (all couplings of a row in registers or
bytes) at the kernel's edges, against the list kernel and the FP64 oracle."""
import numpy as np
import pytest
import torch

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu

PRECS = [("PREC_FP32", 1e-5), ("PREC_BF16", 1e-2)]


@pytest.mark.parametrize("prec_name,tol", PRECS)
@pytest.mark.parametrize("N,R", [(2, 1), (3, 3), (20, 2), (33, 3), (64, 1), (65, 2), (100, 1), (127, 3),
                                 (128, 1), (129, 2), (191, 1), (192, 3), (193, 1), (255, 2), (256, 1),
                                 (32, 9), (97, 40), (130, 152)])
def test_complete_graph(N, R, prec_name, tol):
    """One step from whole-number fluxes (every sum exact) equals the list kernel's
    bit by bit; 101 steps stay within the sparse kernels' bounds of the oracle, and a
    run split at step 31 (window in the second part) has the same bits."""
    from oracle import oracle as orc
    from paper_2004_03972_gb300 import hqa
    inst = instances.sk_pm1(N, N)
    if N % 2:
        inst = instances.with_integer_field(inst, 3, 1)
    ctx = hqa.Context.from_instance(inst)
    if prec_name == "PREC_FP32":   # (a dense context's BF16 runs are the tensor-core GEMM's)
        plan = ctx.plan(R)
        assert (plan["kernel"], plan["blocks"], plan["balance"]) == (hqa.KERNEL_SCALAR, R, 1.0)
    g = torch.Generator("cuda").manual_seed(N)
    phi = torch.randint(-8, 9, (R, N), generator=g, device="cuda").float()
    p0 = torch.rand(R, N, generator=g, device="cuda") - 0.5
    base = dict(precision=getattr(hqa, prec_name), outputs=("phi", "p", "phibar"), dt=1e-4)
    one = dict(init=hqa.INIT_GIVEN, phi0=phi, p0=p0, start_step=50, **base)
    a = ctx.run(1, R, **one)
    b = ctx.run(1, R, kernel=hqa.KERNEL_SCALAR, replicas_per_block=1, **one)
    assert all(torch.equal(a[k], b[k]) for k in a)
    kw = dict(seed=6, init=hqa.INIT_RANDOM_FLUX, sched=hqa.schedule(window=30), **base)
    out = ctx.run(101, R, **kw)
    head = ctx.run(31, R, **kw)
    tail = ctx.run(70, R, **dict(kw, init=hqa.INIT_GIVEN, phi0=head["phi"], p0=head["p"], start_step=31))
    ctx.sync()
    assert all(torch.equal(out[k], tail[k]) for k in out)
    pr = orc.Problem.from_instance(inst)
    for r in sorted({0, R - 1}):
        want = orc.md_run(pr, 101, dt=1e-4, phi0=orc.initial_flux_random(6, r, N),
                          p0=orc.initial_momenta(6, r, N), window=30)
        for k, w in zip(("phi", "p", "phibar"), want):
            scale = max(np.max(np.abs(w)), 1.0 if k == "p" else 0.0)
            assert np.max(np.abs(out[k][r].cpu().numpy() - w)) <= tol * scale, (k, r)
    ctx.close()


@pytest.mark.parametrize("N,R", [(20, 2), (64, 9), (65, 1), (100, 3), (129, 2), (161, 1), (256, 4)])
def test_bf16_operand_of_sparse_context(N, R):
    """The BF16 form, which complete graphs given in CSR take: one exact step equals the
    list kernel's, 100 steps stay within 1e-2 of the oracle."""
    from oracle import oracle as orc
    from paper_2004_03972_gb300 import hqa
    inst = instances.er_pm1(N, 1.0, N)
    ctx = hqa.Context.from_instance(inst)
    plan = ctx.plan(R, precision=hqa.PREC_BF16)
    assert (plan["kernel"], plan["blocks"], plan["balance"]) == (hqa.KERNEL_SCALAR, R, 1.0)
    g = torch.Generator("cuda").manual_seed(N)
    phi = torch.randint(-8, 9, (R, N), generator=g, device="cuda").float()
    p0 = torch.rand(R, N, generator=g, device="cuda") - 0.5
    kw = dict(precision=hqa.PREC_BF16, outputs=("phi", "p", "phibar"), dt=1e-4)
    one = dict(init=hqa.INIT_GIVEN, phi0=phi, p0=p0, start_step=50, **kw)
    a = ctx.run(1, R, **one)
    b = ctx.run(1, R, kernel=hqa.KERNEL_SCALAR, replicas_per_block=1, **one)
    out = ctx.run(100, R, seed=6, **kw)
    ctx.sync()
    assert all(torch.equal(a[k], b[k]) for k in a)
    pr = orc.Problem.from_instance(inst)
    for r in sorted({0, R - 1}):
        want = orc.md_run(pr, 100, dt=1e-4, p0=orc.initial_momenta(6, r, N))
        for k, w in zip(("phi", "p"), want):
            scale = max(np.max(np.abs(w)), 1.0 if k == "p" else 0.0)
            assert np.max(np.abs(out[k][r].cpu().numpy() - w)) <= 1e-2 * scale, (k, r)
    ctx.close()


def test_neighbouring_routes():
    """A missing coupling, one spin more and a stated blocking keep the list kernels."""
    from paper_2004_03972_gb300 import hqa
    J = instances.sk_pm1(100, 3).to_dense()
    J[4, 9] = J[9, 4] = 0.0
    for inst in (instances.Instance("gap", 100, dense=J), instances.sk_pm1(257, 1)):
        ctx = hqa.Context.from_instance(inst)
        kw = dict(seed=2, dt=1e-3, outputs=("phi", "p", "phibar"))
        a = ctx.run(40, 2, **kw)
        b = ctx.run(40, 2, kernel=hqa.KERNEL_SCALAR, replicas_per_block=1, **kw)
        ctx.sync()
        assert all(torch.equal(a[k], b[k]) for k in a)
        ctx.close()
