"""The register-resident form of the low-degree batch kernel at the edges of its
units per thread, against the one-replica form (RB = 1) bit by bit."""
import pytest
import torch

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hqa():
    from paper_2004_03972_gb300 import hqa as h
    return h


def _edge_members():
    # 2 replicas: 1 to 5 spins a thread, the last one full, one short, one over
    sizes = (36, 256, 1020, 1026, 1280, 2048, 2050, 2500, 3072, 4098, 5000, 5120)
    return [instances.regular3_pm1(n, 7 + n) if k % 2 else instances.torus_for_n(n, 7 + n)
            for k, n in enumerate(sizes)]


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("S,W", [(1, 100), (7, 3), (24, 24)])
def test_register_form_bits(hqa, prec, S, W):
    """Blocking 2 and an open blocking (small members at 4 and 8) give the bits of
    blocking 1; 131 replicas leave every block size a ragged last block."""
    R = 131
    batch = hqa.Context.batch([hqa.Context.from_instance(i) for i in _edge_members()])
    g = torch.Generator("cuda").manual_seed(S)
    phi0 = 3.0 * torch.rand(R, batch.N, generator=g, device="cuda") - 1.5
    p0 = torch.rand(R, batch.N, generator=g, device="cuda") - 0.5
    kw = dict(sched=hqa.schedule(window=W), dt=1 / 500, kernel=hqa.KERNEL_LOWDEG,
              precision=hqa.PREC_BF16 if prec == "bf16" else hqa.PREC_FP32,
              outputs=("phi", "p", "phibar"))
    for init in (dict(init=hqa.INIT_GIVEN, phi0=phi0, p0=p0, start_step=200),
                 dict(init=hqa.INIT_RANDOM_FLUX, seed=5)):
        want = batch.run(S, R, replicas_per_block=1, **kw, **init)
        for rb in (2, 0):
            got = batch.run(S, R, replicas_per_block=rb, **kw, **init)
            for key in want:
                assert torch.equal(got[key], want[key]), (rb, key)
    batch.sync()


def test_blocking_of_mixed_launches(hqa):
    """Few replicas, another M and a member beyond the register form (N = 5121 at
    two replicas): the same bits at blockings 1, 2 and open."""
    small = [hqa.Context.from_instance(instances.torus_for_n(n, n)) for n in (36, 400, 900)]
    large = small + [hqa.Context.from_instance(instances.regular3_pm1(5122, 3))]
    for ctxs, M in ((small, 6), (small, 4), (large, 6)):
        batch = hqa.Context.batch(ctxs)
        for R in (1, 3, 9):
            kw = dict(sched=hqa.schedule(M=M, window=4), dt=1 / 500, kernel=hqa.KERNEL_LOWDEG,
                      seed=11, outputs=("phi", "p", "phibar"))
            want = batch.run(12, R, replicas_per_block=1, **kw)
            for rb in (2, 0):
                got = batch.run(12, R, replicas_per_block=rb, **kw)
                for key in want:
                    assert torch.equal(got[key], want[key]), (M, R, rb, key)
        batch.sync()
