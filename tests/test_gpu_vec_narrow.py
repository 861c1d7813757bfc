"""The 8-byte form of the vectorised sparse kernel (few replicas, open blocking)
against 64-bit fields, the scalar kernel and the FP64 oracle."""
import numpy as np
import pytest
import torch

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu

PRECS = [("fp32", 4), ("bf16", 8)]


@pytest.fixture(scope="module")
def hqa():
    from paper_2004_03972_gb300 import hqa as h
    return h


@pytest.fixture(scope="module")
def orc():
    from oracle import oracle
    return oracle


def _prec(hqa, name):
    return hqa.PREC_BF16 if name == "bf16" else hqa.PREC_FP32


@pytest.mark.parametrize("name,V", PRECS)
def test_dispatch_edges(hqa, name, V):
    """Half a vector per block while every block has an SM (152 on GB300), from one
    vector of replicas on and up to N = 2048; a stated blocking is left alone."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for N, R, want in [(300, V, V // 2), (300, V // 2 * sms, V // 2), (300, V // 2 * sms + 1, V),
                       (2048, 40, V // 2)]:
        ctx = hqa.Context.from_instance(instances.er_mean_degree_pm1(N, 8, 1))
        assert ctx.plan(R, precision=_prec(hqa, name))["replicas_per_block"] == want, (N, R)
        if N == 300:
            wide = ctx.plan(R, precision=_prec(hqa, name), replicas_per_block=V, kernel=hqa.KERNEL_VECTOR)
            assert wide["replicas_per_block"] == V
        with pytest.raises(hqa.HQAError):
            ctx.plan(R, precision=_prec(hqa, name), replicas_per_block=V // 2, kernel=hqa.KERNEL_VECTOR)
    ctx = hqa.Context.from_instance(instances.er_mean_degree_pm1(2049, 4, 1))
    assert ctx.plan(40, precision=_prec(hqa, name))["replicas_per_block"] != V // 2


@pytest.mark.parametrize("name,V", PRECS)
@pytest.mark.parametrize("N,R", [(9, 8), (33, 11), (497, 129), (800, 303), (1023, 64), (2048, 31)])
def test_exact_field_and_one_step(hqa, name, V, N, R):
    """Whole-number fluxes up to 8: every sum is exact, so the field equals the 64-bit
    one and one step the scalar kernel's, bit by bit (a field h among them)."""
    inst = instances.er_pm1(N, 0.06, N) if N == 497 else instances.er_mean_degree_pm1(N, min(8, N // 2), N)
    inst = instances.with_integer_field(inst, 3, 5) if N % 2 else inst
    ctx = hqa.Context.from_instance(inst)
    g = torch.Generator("cuda").manual_seed(N)
    phi = torch.randint(-8, 9, (R, N), generator=g, device="cuda").float()
    p0 = torch.rand(R, N, generator=g, device="cuda") - 0.5
    prec = _prec(hqa, name)
    L = ctx.local_field(phi, precision=prec)
    J = torch.from_numpy(inst.to_dense()).double().cuda()
    want = phi.double() @ J
    if inst.h is not None:
        want = want + 2.0 * torch.from_numpy(inst.h).double().cuda() * phi.double().abs()
    assert torch.equal(L.double(), want)
    kw = dict(dt=1 / 500, precision=prec, init=hqa.INIT_GIVEN, phi0=phi, p0=p0, start_step=100,
              outputs=("phi", "p", "phibar"))
    a = ctx.run(1, R, **kw)
    b = ctx.run(1, R, kernel=hqa.KERNEL_SCALAR, replicas_per_block=1, **kw)
    ctx.sync()
    for key in a:
        assert torch.equal(a[key], b[key]), key


@pytest.mark.parametrize("name,V", PRECS)
def test_anneal(hqa, orc, name, V):
    """150 steps against the oracle at the sparse kernels' bounds (FP32 1e-5, BF16
    operand 1e-2), and the run split at step 40 (window in the second call) bitwise."""
    inst = instances.with_integer_field(instances.er_pm1(129, 0.1, 3), 1, 4)
    ctx = hqa.Context.from_instance(inst)
    R, S, seed, dt = 13, 150, 21, 1 / 500
    kw = dict(seed=seed, dt=dt, precision=_prec(hqa, name), outputs=("phi", "p", "phibar"))
    assert ctx.plan(R, precision=_prec(hqa, name))["replicas_per_block"] == V // 2
    out = ctx.run(S, R, **kw)
    a = ctx.run(40, R, **kw)
    b = ctx.run(S - 40, R, init=hqa.INIT_GIVEN, phi0=a["phi"], p0=a["p"], start_step=40, **kw)
    ctx.sync()
    for key in out:
        assert torch.equal(out[key], b[key]), key
    tol = 1e-2 if name == "bf16" else 1e-5
    pr = orc.Problem.from_instance(inst)
    for r in (0, R - 1):
        ophi, op, obar = orc.md_run(pr, S, dt=dt, p0=orc.initial_momenta(seed, r, inst.N))
        for key, want, scale in (("phi", ophi, np.max(np.abs(ophi))), ("p", op, max(1.0, np.max(np.abs(op)))),
                                 ("phibar", obar, np.max(np.abs(ophi)))):
            got = out[key][r].cpu().numpy().astype(np.float64)
            assert np.max(np.abs(got - want)) <= tol * scale, (key, r)
