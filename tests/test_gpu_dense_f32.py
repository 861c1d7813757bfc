"""FP32 dense MD on the tensor cores (fixed-point slices) against the FP64 oracle, at the edges
of its tiles: 128-row tiles, 16 / 32 / 64 / 2 x 64 replica columns, 1 to 3 coupling slices,
pairs of row tiles, more replicas than one launch holds, and states far below 1.

Tolerance, derived: five steps round p and phi about four times each by 2^-24, 1.2e-6 of their
scale, and the steps amplify by less than 1.5; the slices' own error (2^-24 of the largest flux
or less, times sqrt(N) kB) is below that: 2e-6.
"""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu

STEPS, DT, TOL = 5, 1e-4, 2e-6


def _instance(kind, N):
    if kind == "sk":
        return instances.sk_pm1(N, 31 + N)
    if kind == "skh":
        return instances.with_integer_field(instances.sk_pm1(N, 31 + N), 3, 5)
    inst = instances.uniform_sg(N, 31 + N)
    if kind == "halves":        # couplings of two slices: 1 + 2^-10 times a sign
        inst.dense = np.sign(inst.dense) * (1.0 + 2.0 ** -10)
    elif kind == "rows":        # row scales far apart: one pair coupled a million times stronger
        inst.dense[:2, 2:] = inst.dense[2:, :2] = 0.0
        inst.dense[2:, 2:] *= 2.0 ** -20
        inst.h = None
    return inst


@pytest.mark.parametrize("kind,N,R,scale", [
    ("sk", 1, 1, 1.0), ("sk", 127, 16, 1.0), ("sk", 128, 17, 1.0), ("skh", 129, 33, 1.0),
    ("sk", 256, 2433, 1.0), ("skh", 384, 700, 1.0), ("sg", 200, 5, 1.0), ("sg", 257, 1300, 1.0),
    ("halves", 130, 70, 1.0), ("rows", 140, 40, 1.0), ("sk", 200, 40, 2.0 ** -21),
    ("sg", 200, 40, 2.0 ** -33), ("sk", 300, 64, 40.0)])
def test_against_oracle(kind, N, R, scale):
    import torch

    from paper_2004_03972_gb300 import hqa
    inst = _instance(kind, N)
    M = 2 if scale > 1 else 6   # the harmonic potential takes fluxes beyond the slices' units
    rng = np.random.default_rng(N + R)
    phi0 = (scale * rng.uniform(-0.4, 0.4, (R, N))).astype(np.float32)
    p0 = (scale * rng.uniform(-1.0, 1.0, (R, N))).astype(np.float32)
    ctx = hqa.Context.from_instance(inst)
    out = ctx.run(STEPS, R, sched=hqa.schedule(window=3, M=M), dt=DT, kernel=hqa.KERNEL_DENSE,
                  init=hqa.INIT_GIVEN, phi0=torch.from_numpy(phi0).cuda(),
                  p0=torch.from_numpy(p0).cuda(), outputs=("phi", "p", "phibar"))
    ctx.sync()
    assert ctx.plan(R, kernel=hqa.KERNEL_DENSE)["threads"] == 320
    got = [out[k].double().cpu().numpy() for k in ("phi", "p", "phibar")]
    pr = orc.Problem.from_instance(inst)
    some = sorted({0, R // 2, R - 1})
    want = [orc.md_run(pr, STEPS, dt=DT, phi0=phi0[r], p0=p0[r], window=3, M=M) for r in some]
    for g, k in zip(got, range(3)):
        w = np.stack([x[k] for x in want])
        ref = max(np.max(np.abs(w)), np.max(np.abs(p0[some])) if k == 1 else 0.0)
        assert np.max(np.abs(g[some] - w)) <= TOL * ref
    ctx.close()
