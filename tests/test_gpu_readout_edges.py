"""Readout and bit-mask energy at the edges of their work split: ties that only the index
decides, zeros of both signs, replica counts on both sides of the replicas-per-block steps,
sizes around the 32-spin words.  Everything is exact.
"""
import numpy as np
import pytest

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 255, 257, 2049, 5000])
@pytest.mark.parametrize("values", ["spread", "ties", "one", "tiny", "wide"])
def test_split_is_the_rank_split(N, values):
    import torch

    from paper_2004_03972_gb300 import hqa
    rng = np.random.default_rng(N)
    R = 9
    x = {"spread": rng.normal(size=(R, N)),
         "ties": rng.choice([0.0, -0.0, 0.5, -0.5, 0.5000001], size=(R, N)),
         "one": np.full((R, N), -0.75),
         "tiny": rng.integers(-9, 10, size=(R, N)) * 1e-42,
         "wide": np.exp(rng.uniform(-80, 80, size=(R, N)))}[values].astype(np.float32)
    ctx = hqa.Context.from_csr(N, np.zeros(N + 1, np.int64), np.zeros(0, np.int32), np.zeros(0))
    xt = torch.from_numpy(x).cuda()
    for n in sorted({0, 1, N // 3, N - 1, N, N + 5}):
        spins, frozen, tally = ctx.readout(xt, n)
        ctx.sync()
        k = min(n, N)
        want = np.ones((R, N), np.uint8)
        for r in range(R):
            order = np.lexsort((np.arange(N), np.abs(x[r])))
            want[r, order[:k]] = 0
        assert np.array_equal(frozen.cpu().numpy(), want)
        assert np.array_equal(spins.cpu().numpy(), np.where(x >= 0, 1, -1))
        assert np.array_equal(tally.cpu().numpy(), np.tile([N - k, k], (R, 1)))
    ctx.close()


@pytest.mark.parametrize("N,R,field", [(2, 1, True), (31, 40, False), (32, 911, True), (33, 913, True),
                                       (64, 3650, True), (97, 5001, False), (257, 1000, True),
                                       (300, 4000, True)])
def test_bit_mask_energy(N, R, field):
    import torch

    from paper_2004_03972_gb300 import hqa
    inst = instances.sk_pm1(N, N)
    inst.dense[np.random.default_rng(N).random((N, N)) < 0.15] = 0.0
    inst.dense = np.triu(inst.dense) + np.triu(inst.dense).T
    if field:
        inst = instances.with_integer_field(inst, 1000000, 3)
    ctx = hqa.Context.from_instance(inst)
    s = np.random.default_rng(R).choice([-1, 1], size=(R, N)).astype(np.int8)
    e, c = ctx.energy(torch.from_numpy(s).cuda())
    ctx.sync()
    J, h = inst.dense.astype(np.int64), 0 if inst.h is None else inst.h.astype(np.int64)
    pairs = ((s.astype(np.int64) @ J) * s).sum(axis=1)
    assert np.array_equal(e.cpu().numpy(), pairs // 2 + (s * h).sum(axis=1))
    assert np.array_equal(c.cpu().numpy(), (J.sum() - pairs) // 4)
    ctx.close()
