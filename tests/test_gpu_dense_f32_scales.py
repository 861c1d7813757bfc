"""FP32 dense MD: every replica at its own scale, whatever shares its launch, and bitwise splits.

A table schedule with alpha = 0 and beta = 1 turns one step into the field: p - L.  Tolerance of
the field against 64 bits (2-norm over the spins of one replica), derived: the operands are held
to 2^-25 of their group's and row's largest, times at most (max / rms)^2 = 3 for uniform values,
0.9e-7; three sums, the row's power of two and the kick round by at most 2^-24 each, 1.8e-7 and
less in the mean; truncation in the second accumulator, N / 16 times 2^-31, 0.3e-7: 4e-7.
"""
import numpy as np
import pytest

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu

# replicas of one launch, dealt in turn: ordinary, small, just above powers of two, large
SCALES = [1.0, 1e-2, 1e-4, 2.0 ** -6 * 1.01, 1.0, 1e-6, 2.0 ** -10 * 1.01, 30.0, 1e-3, 2.0 ** -40]


def _instance(kind, N):
    if kind == "sk":
        return instances.sk_pm1(N, 3 + N)
    inst = instances.uniform_sg(N, 3 + N)
    inst.h = None
    if kind == "whole":         # any whole numbers up to 127
        J = np.rint(127 * inst.dense / np.abs(inst.dense).max())
        inst.dense = J.astype(inst.dense.dtype)
    elif kind == "halves":
        inst.dense = np.sign(inst.dense) * (1.0 + 2.0 ** -10)
    return inst


def _fluxes(N, R, scales):
    rng = np.random.default_rng(N + R)
    x = rng.uniform(-1.5, 1.5, (R, N)) * np.resize(scales, R)[:, None]
    return x.astype(np.float32)


def _field(hqa, torch, ctx, phi):
    """-p after one step with kA = 0, kB = 1, from p = 0."""
    z = torch.zeros_like(phi)
    out = ctx.run(1, phi.shape[0], table=(np.zeros(5), np.ones(3)), dt=1e-4, start_step=1,
                  kernel=hqa.KERNEL_DENSE, init=hqa.INIT_GIVEN, phi0=phi, p0=z, outputs=("p",))
    ctx.sync()
    return -out["p"]


def _norm_errors(got, want):
    return np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)


@pytest.mark.parametrize("kind,N,R", [
    ("sk", 64, 20), ("sk", 300, 70), ("sk", 1000, 700), ("sk", 2000, 1024), ("whole", 200, 33),
    ("whole", 1000, 64), ("sg", 100, 20), ("sg", 500, 200), ("sg", 1000, 512), ("halves", 300, 40)])
def test_field_of_every_scale(kind, N, R):
    import torch

    from paper_2004_03972_gb300 import hqa
    inst = _instance(kind, N)
    ctx = hqa.Context.from_instance(inst)
    phi = _fluxes(N, R, SCALES)
    got = _field(hqa, torch, ctx, torch.from_numpy(phi).cuda()).double().cpu().numpy()
    want = phi.astype(np.float64) @ np.asarray(inst.dense, np.float32).astype(np.float64)
    assert _norm_errors(got, want).max() <= 4e-7
    ctx.close()


def test_field_beside_one_large_flux():
    """One flux 2^20 times the others: the sums are the large one's, and what is truncated
    against it stays below N / 16 units of the last place, 7.5e-6."""
    import torch

    from paper_2004_03972_gb300 import hqa
    inst = _instance("sk", 1000)
    ctx = hqa.Context.from_instance(inst)
    phi = _fluxes(1000, 40, [2.0 ** -20])
    phi[:, 5] = 1.0
    got = _field(hqa, torch, ctx, torch.from_numpy(phi).cuda()).double().cpu().numpy()
    want = phi.astype(np.float64) @ np.asarray(inst.dense, np.float64)
    assert _norm_errors(got, want).max() <= 7.5e-6
    ctx.close()


@pytest.mark.parametrize("kind,N,R", [("sk", 200, 33), ("sk", 300, 2433), ("sg", 200, 70), ("sg", 257, 1300)])
def test_replica_alone(kind, N, R):
    """A replica has the bits that it has in a run of its own."""
    import torch

    from paper_2004_03972_gb300 import hqa
    inst = _instance(kind, N)
    ctx = hqa.Context.from_instance(inst)
    phi = torch.from_numpy(_fluxes(N, R, SCALES[:7])).cuda()
    kw = dict(dt=1e-3, start_step=300, kernel=hqa.KERNEL_DENSE, init=hqa.INIT_GIVEN,
              outputs=("phi", "p", "phibar"))
    full = ctx.run(6, R, phi0=phi, p0=0.1 * phi, **kw)
    for r in (1, 2, 5, R - 1):
        own = phi[r:r + 1].contiguous()
        one = ctx.run(6, 1, phi0=own, p0=0.1 * own, **kw)
        ctx.sync()
        assert all(torch.equal(one[k][0], full[k][r]) for k in one)
    ctx.close()


@pytest.mark.parametrize("kind", ["sk", "sg"])
@pytest.mark.parametrize("hstep", [0.25, 1.0])
def test_split_run_is_bitwise(kind, hstep):
    import torch

    from paper_2004_03972_gb300 import hqa
    ctx = hqa.Context.from_instance(_instance(kind, 200))
    R, S = 40, 9
    kw = dict(dt=1e-3, sched=hqa.schedule(hstep=hstep), kernel=hqa.KERNEL_DENSE, outputs=("phi", "p"))
    full = ctx.run(S, R, seed=3, **kw)
    for m in (1, 2, 3, 5):
        a = ctx.run(m, R, seed=3, **kw)
        b = ctx.run(S - m, R, init=hqa.INIT_GIVEN, phi0=a["phi"], p0=a["p"], start_step=m, **kw)
        ctx.sync()
        assert torch.equal(full["phi"], b["phi"]) and torch.equal(full["p"], b["p"]), m
    _, phi, p = ctx.trace(S, R, 2, seed=3, dt=1e-3, sched=hqa.schedule(hstep=hstep),
                          kernel=hqa.KERNEL_DENSE)
    ctx.sync()
    assert torch.equal(full["phi"], phi) and torch.equal(full["p"], p)
    ctx.close()
