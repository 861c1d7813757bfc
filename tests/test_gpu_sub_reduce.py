"""The sub-solve's exact reduction (fields that decide, leaves, components) against the plain
Gray-code walk of the allocation-free entry point, which does not reduce: same configurations,
bit for bit, ties included, on graphs of every density.
"""
import numpy as np
import pytest

from paper_2004_03972_gb300 import instances

pytestmark = pytest.mark.gpu


def _graph(kind, N, seed):
    rng = np.random.default_rng(seed)
    i, j = np.triu_indices(N, k=1)
    if kind == "path":
        keep = j == i + 1
    elif kind == "cycle":
        keep = (j == i + 1) | ((i == 0) & (j == N - 1))
    elif kind == "star":
        keep = i == 0
    elif kind == "pairs":
        keep = (j == i + 1) & (i % 2 == 0)
    elif kind == "tree":
        parent = np.array([0] + [rng.integers(0, k) for k in range(1, N)])
        keep = parent[j] == i
    else:
        keep = rng.random(i.size) < kind
    i, j = i[keep], j[keep]
    w = rng.choice([-1.0, 1.0], size=i.size)
    rp, col, val = instances._edges_to_csr(N, i, j, w)
    return instances.Instance(f"g{kind}", N, row_ptr=rp, col=col, val=val)


@pytest.mark.parametrize("kind", ["path", "cycle", "star", "pairs", "tree", 0.0, 0.03, 0.08, 0.15,
                                  0.3, 1.0])
@pytest.mark.parametrize("n", [1, 5, 13, 19, 30])
@pytest.mark.parametrize("hmax", [0, 2, 1000000])
def test_reduction_equals_the_walk(kind, n, hmax):
    import torch

    from paper_2004_03972_gb300 import hqa
    if n == 30 and kind == 1.0:
        n = 22                      # the complete graph is walked in full
    N, R = n + 6, 5 if n > 20 else 40
    rng = np.random.default_rng(100 * n + hmax % 7)
    inst = _graph(kind, N, n)
    if hmax:
        inst = instances.with_integer_field(inst, hmax, 9)
    ctx = hqa.Context.from_instance(inst)
    spins = torch.from_numpy(rng.choice([-1, 1], size=(R, N)).astype(np.int8)).cuda()
    frozen = np.ones((R, N), np.uint8)
    for r in range(R):              # n open spins, fewer in some replicas
        frozen[r, rng.choice(N, size=n - (r % 3 if n > 2 else 0), replace=False)] = 0
    frozen = torch.from_numpy(frozen).cuda()
    got, e = ctx.solve_sub(spins, frozen, n)
    want, we = torch.empty_like(got), torch.empty_like(e)
    ctx.solve_sub_noalloc(spins, frozen, n, want, we)
    ctx.sync()
    assert torch.equal(got, want) and torch.equal(e, we)
    ctx.close()
