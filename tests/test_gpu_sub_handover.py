"""Where the sub-solve hands a component to the GPU-wide walk: cliques of c of the n open spins,
which no reduction touches, on both sides of the line."""
import numpy as np
import pytest


pytestmark = pytest.mark.gpu


def _clique(n, c, R, torch, hqa):
    rng = np.random.default_rng(n + c)
    J = np.zeros((n, n), np.float32)
    a = np.triu(rng.choice([-1.0, 1.0], size=(c, c)), 1)
    J[:c, :c] = a + a.T
    ctx = hqa.Context.from_dense(J)
    return (ctx, torch.ones(R, n, dtype=torch.int8, device="cuda"),
            torch.zeros(R, n, dtype=torch.uint8, device="cuda"))


@pytest.mark.parametrize("n,c,R", [(16, 12, 1), (18, 14, 2), (24, 16, 1), (24, 17, 1), (24, 20, 200),
                                   (26, 19, 1), (26, 22, 3)])
def test_both_sides_of_the_line(n, c, R):
    import torch

    from paper_2004_03972_gb300 import hqa
    ctx, spins, frozen = _clique(n, c, R, torch, hqa)
    got, e = ctx.solve_sub(spins, frozen, n)
    want, we = torch.empty_like(got), torch.empty_like(e)
    ctx.solve_sub_noalloc(spins, frozen, n, want, we)
    ctx.sync()
    assert torch.equal(got, want) and torch.equal(e, we)
    ctx.close()


def test_one_replica_with_a_large_component():
    """26 of 30 spins: 0.23 ms over the whole GPU, 15 ms in one CTA."""
    import torch

    from paper_2004_03972_gb300 import hqa
    ctx, spins, frozen = _clique(30, 26, 1, torch, hqa)
    ctx.solve_sub(spins, frozen, 30)
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    ctx.solve_sub(spins, frozen, 30)
    b.record()
    torch.cuda.synchronize()
    assert a.elapsed_time(b) < 4.0
    ctx.close()
