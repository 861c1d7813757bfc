"""The work a user of this library has it do, as cases that can be timed and checked.

Each case is one call, or one short sequence of calls, through the package's
Python binding.  Sizes come from the benchmark's workloads (SK N = 100 and
2000, ER N = 800, the uniform spin glass, the uneven batch, ER graphs of mean
degree 8) and from the tests.  An anneal is thousands of leapfrog steps; a case
runs a segment of one (a segment is what the feature prefix, a trace and a
resumed run are), so that its outputs can be compared before rounding
differences have grown.  ``exact`` restates every floating-point result in
64 bits with plain torch and numpy.
"""
import math

import numpy as np
import torch

from paper_2004_03972_gb300 import hqa, instances

PRECISIONS = {"fp32": hqa.PREC_FP32, "bf16": hqa.PREC_BF16, "bf16x2": hqa.PREC_BF16X2,
              "fp16": hqa.PREC_FP16, "fp16x2": hqa.PREC_FP16X2}
KERNELS = {"auto": hqa.KERNEL_AUTO, "dense": hqa.KERNEL_DENSE, "stream": hqa.KERNEL_STREAM}


def listed():
    return [
        # one small trajectory, the first thing a user runs: all latency
        {"name": "sk100_single", "op": "run", "graph": "sk", "N": 100, "R": 1, "steps": 150,
         "total": 1000, "sched": "linear", "prec": "fp32", "kernel": "auto", "from": "start"},
        # sparse MAX-CUT replicas in the default precision, from the start of an anneal
        {"name": "er800_fp32", "op": "run", "graph": "er48", "N": 800, "R": 1024, "steps": 200,
         "total": 5000, "sched": "paper", "prec": "fp32", "kernel": "auto", "from": "start"},
        # the same with the BF16 operand, resumed in the middle of an anneal
        {"name": "er800_bf16", "op": "run", "graph": "er48", "N": 800, "R": 1024, "steps": 100,
         "total": 5000, "sched": "paper", "prec": "bf16", "kernel": "auto", "from": "middle"},
        # large sparse graph: the streaming kernel
        {"name": "er20000_bf16", "op": "run", "graph": "er8", "N": 20000, "R": 256, "steps": 100,
         "total": 10000, "sched": "paper", "prec": "bf16", "kernel": "stream", "from": "start"},
        # many small instances of uneven size in one launch
        {"name": "uneven96_fp32", "op": "batch", "count": 96, "lo": 200, "hi": 5000, "R": 64,
         "steps": 100, "total": 5000, "sched": "paper", "prec": "fp32"},
        # K2000 MAX-CUT, the plain FP32 form
        {"name": "sk2000_fp32", "op": "run", "graph": "sk", "N": 2000, "R": 1024, "steps": 40,
         "total": 10000, "sched": "paper", "prec": "fp32", "kernel": "dense", "from": "start"},
        # K2000 MAX-CUT, the split operand at full replica count
        {"name": "sk2000_fp16x2", "op": "run", "graph": "sk", "N": 2000, "R": 4096, "steps": 40,
         "total": 10000, "sched": "paper", "prec": "fp16x2", "kernel": "dense", "from": "start"},
        # real-valued spin glass with a field, plain FP32, resumed
        {"name": "sg1000_fp32", "op": "run", "graph": "sg", "N": 1000, "R": 512, "steps": 40,
         "total": 10000, "sched": "paper", "prec": "fp32", "kernel": "dense", "from": "middle"},
        # large real-valued spin glass, split operands
        {"name": "sg10000_bf16x2", "op": "run", "graph": "sg", "N": 10000, "R": 1024, "steps": 10,
         "total": 10000, "sched": "paper", "prec": "bf16x2", "kernel": "dense", "from": "start"},
        # exact solution of the reduced problem on the ambivalent spins
        {"name": "sub24_er800", "op": "sub", "graph": "er48", "N": 800, "R": 1024, "n": 24},
        # signs, ranking and integer energies of a K2000 ensemble
        {"name": "readout_sk2000", "op": "readout", "graph": "sk", "N": 2000, "R": 4096, "n": 24},
        # surrogate gate: logits, loss and gradient of its network on one batch
        {"name": "mlp_fp32", "op": "mlp", "rows": 128000, "prec": "fp32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["single", "sparse", "sparse", "stream", "batch", "dense", "dense", "glass",
                       "sub", "readout", "mlp"])
    where = rng.choice(["start", "middle"])
    if kind == "single":
        return {"op": "run", "graph": "sk", "N": rng.randint(20, 200), "R": rng.randint(1, 4),
                "steps": rng.randint(50, 150), "total": 1000,
                "sched": rng.choice(["linear", "paper"]), "prec": "fp32", "kernel": "auto",
                "from": "start"}
    if kind == "sparse":
        prec = rng.choice(["fp32", "bf16"])
        return {"op": "run", "graph": rng.choice(["er48", "er8", "er48h"]),
                "N": rng.randint(300, 1000), "R": _log_int(rng, 30, 1024),
                "steps": rng.randint(50, 200 if prec == "fp32" and where == "start" else 100),
                "total": 5000, "sched": "paper", "prec": prec, "kernel": "auto", "from": where}
    if kind == "stream":
        return {"op": "run", "graph": "er8", "N": _log_int(rng, 8000, 20000),
                "R": _log_int(rng, 40, 256), "steps": rng.randint(30, 100), "total": 10000,
                "sched": "paper", "prec": rng.choice(["fp32", "bf16"]), "kernel": "stream",
                "from": where}
    if kind == "batch":
        return {"op": "batch", "count": rng.randint(10, 96), "lo": 200, "hi": 5000,
                "R": rng.randint(16, 64), "steps": rng.randint(30, 100), "total": 5000,
                "sched": "paper", "prec": rng.choice(["fp32", "bf16"])}
    if kind == "dense":
        return {"op": "run", "graph": rng.choice(["sk", "skh"]), "N": _log_int(rng, 300, 2000),
                "R": _log_int(rng, 64, 1024), "steps": rng.randint(10, 40), "total": 10000,
                "sched": "paper", "prec": rng.choice(["fp32", "fp32", "fp16x2", "bf16", "fp16"]),
                "kernel": "dense", "from": where}
    if kind == "glass":
        return {"op": "run", "graph": "sg", "N": _log_int(rng, 200, 4000),
                "R": _log_int(rng, 64, 512), "steps": rng.randint(5, 20), "total": 10000,
                "sched": "paper", "prec": rng.choice(["fp32", "bf16x2", "fp16x2"]),
                "kernel": "dense", "from": where}
    if kind == "sub":
        graph = rng.choice(["er48", "er8", "sk"])
        return {"op": "sub", "graph": graph, "N": rng.randint(300, 1000),
                "R": _log_int(rng, 16, 1024), "n": rng.randint(10, 24)}
    if kind == "readout":
        return {"op": "readout", "graph": rng.choice(["sk", "er48"]), "N": rng.randint(300, 2000),
                "R": _log_int(rng, 64, 4096), "n": rng.randint(0, 100)}
    return {"op": "mlp", "rows": _log_int(rng, 4096, 128000), "prec": rng.choice(["fp32", "bf16"])}


# ---- inputs -----------------------------------------------------------------

def _instance(case, seed):
    N, graph = case["N"], case["graph"]
    if graph.startswith("sk"):
        inst = instances.sk_pm1(N, seed)
    elif graph.startswith("er48"):
        inst = instances.er_pm1(N, 48.0 / 800, seed)
    elif graph.startswith("er8"):
        inst = instances.er_mean_degree_pm1(N, 8, seed)
    else:
        inst = instances.uniform_sg(N, seed)
    return instances.with_integer_field(inst, 3, seed + 1) if graph.endswith("h") else inst


def _members(case, seed):
    """Half random 3-regular, half tori; the sizes go with the case, the graphs with the seed."""
    sizes = np.random.default_rng(case["count"]).integers(case["lo"], case["hi"] + 1, case["count"])
    return [instances.regular3_pm1(int(n), 1000 * seed + k) if k % 2 == 0 else
            instances.torus_for_n(int(n), 1000 * seed + k) for k, n in enumerate(sizes)]


def _state(case, seed, N):
    """phi0 and p0 of a run: the method's start, or a spread like the one in mid-anneal."""
    g = torch.Generator("cuda").manual_seed(seed + 2)
    R = case["R"]
    if case.get("from", "start") == "middle":
        phi = 3.0 * torch.rand(R, N, generator=g, device="cuda") - 1.5
        return phi, torch.rand(R, N, generator=g, device="cuda") - 0.5
    p = 2.0 * torch.randint(0, 2, (R, N), generator=g, device="cuda") - 1.0
    return torch.zeros(R, N, device="cuda"), p


def _start_step(case):
    return case["total"] // 2 if case.get("from", "start") == "middle" else 0


def _phibar(case, seed, N):
    """Window means as an anneal leaves them: two-sided, a few near zero."""
    g = torch.Generator("cuda").manual_seed(seed + 3)
    x = torch.randn(case["R"], N, generator=g, device="cuda")
    return 1.5 * x / (0.3 + x.abs())


def _local_minimum(case, seed, inst):
    """Spins near a local minimum, as an anneal leaves them; the n with the weakest field open."""
    g = torch.Generator("cuda").manual_seed(seed + 5)
    J = torch.from_numpy(inst.to_dense()).float().cuda()
    s = 2.0 * torch.randint(0, 2, (case["R"], inst.N), generator=g, device="cuda") - 1.0
    for _ in range(40):
        field = s @ J
        turn = (field * s > 0) & (torch.rand(s.shape, generator=g, device="cuda") < 0.3)
        s = torch.where(turn, -s, s)
    weak = (s @ J).abs() + 0.5 * torch.rand(s.shape, generator=g, device="cuda")
    frozen = torch.ones(s.shape, dtype=torch.uint8, device="cuda")
    frozen.scatter_(1, weak.argsort(dim=1, stable=True)[:, :case["n"]], 0)
    return s.to(torch.int8), frozen


def _rows(case, seed):
    g = torch.Generator("cuda").manual_seed(seed + 4)
    x = torch.randn(case["rows"], hqa.MLP_IN, generator=g, device="cuda")
    y = (torch.rand(case["rows"], hqa.MLP_OUT, generator=g, device="cuda") < 0.5).float()
    return x, y


def _schedule(case):
    s = hqa.schedule()
    if case["sched"] == "linear":
        s.kind = hqa.SCHED_LINEAR_GAMMA
    return s


def prepare(case, seed):
    op = case["op"]
    if op == "mlp":
        x, y = _rows(case, seed)
        return {"op": op, "net": hqa.MLP(hqa.MLP.init_params(seed)), "x": x, "y": y,
                "prec": PRECISIONS[case["prec"]]}
    if op == "batch":
        parts = [hqa.Context.from_instance(i) for i in _members(case, seed)]
        ctx = hqa.Context.batch(parts)
    else:
        flags = hqa.J_FP16 if case.get("prec", "").startswith("fp16") else 0
        inst = _instance(case, seed)
        ctx = hqa.Context.from_instance(inst, flags)
    if op in ("run", "batch"):
        phi, p = _state(case, seed, ctx.N)
        s = {"op": op, "ctx": ctx, "phi0": phi, "p0": p, "case": case, "sched": _schedule(case)}
        if op == "run":
            ctx.plan(case["R"], precision=PRECISIONS[case["prec"]], kernel=KERNELS[case["kernel"]])
        return s
    if op == "sub":
        spins, frozen = _local_minimum(case, seed, inst)
        return {"op": op, "ctx": ctx, "n": case["n"], "spins": spins, "frozen": frozen}
    return {"op": op, "ctx": ctx, "n": case["n"], "phibar": _phibar(case, seed, ctx.N)}


def run(state):
    op = state["op"]
    if op == "mlp":
        z = state["net"].forward(state["x"], precision=state["prec"])
        g, loss = state["net"].grad(state["x"], state["y"], precision=state["prec"])
        return {"logits": z, "grad": g, "loss": loss}
    ctx = state["ctx"]
    if op == "sub":
        spins, energy = ctx.solve_sub(state["spins"], state["frozen"], state["n"])
        return {"spins": spins, "energy": energy}
    if op == "readout":
        spins, frozen, tally = ctx.readout(state["phibar"], state["n"])
        energy, cut = ctx.energy(spins)
        return {"spins": spins, "frozen": frozen, "tally": tally, "energy": energy, "cut": cut}
    case = state["case"]
    kernel = KERNELS[case["kernel"]] if op == "run" else hqa.KERNEL_AUTO
    return ctx.run(case["steps"], case["R"], sched=state["sched"], dt=1.0 / case["total"],
                   precision=PRECISIONS[case["prec"]], kernel=kernel, init=hqa.INIT_GIVEN,
                   phi0=state["phi0"], p0=state["p0"], start_step=_start_step(case),
                   outputs=("phi", "p", "phibar"))


# ---- what a pass cannot do without ------------------------------------------

def _nnz(case):
    N = case["N"]
    if case["graph"].startswith("er48"):
        return int(N * (N - 1) * 48.0 / 800)
    if case["graph"].startswith("er8"):
        return 8 * N
    return N * (N - 1)


def work(case):
    op = case["op"]
    if op == "mlp":
        macs = hqa.MLP_IN * hqa.MLP_HIDDEN + hqa.MLP_HIDDEN ** 2 + hqa.MLP_HIDDEN * hqa.MLP_OUT
        rows = case["rows"]
        # two forward passes, and the products of the backward one
        back = macs + hqa.MLP_HIDDEN ** 2 + hqa.MLP_HIDDEN * hqa.MLP_OUT
        return {"bytes": 4 * rows * (2 * hqa.MLP_IN + 2 * hqa.MLP_OUT) + 8 * hqa.MLP_PARAMS,
                "flops": 2 * rows * (2 * macs + back)}
    if op == "batch":
        N = case["count"] * (case["lo"] + case["hi"]) // 2
        nnz, jbytes = int(3.5 * N), int(3.5 * N * 5)
    else:
        N, nnz = case["N"], _nnz(case)
        jbytes = nnz * (2 if case["graph"].startswith(("sk", "sg")) else 5)
    R = case["R"]
    if op in ("run", "batch"):
        # two state arrays in, three out; the field, kick, drift and window of every step
        return {"bytes": jbytes + 20 * R * N, "flops": case["steps"] * R * (2 * nnz + 12 * N)}
    if op == "sub":
        # one update per replica and configuration, as if no graph allowed less
        return {"bytes": jbytes + 3 * R * N + 8 * R, "flops": R * 2.0 ** case["n"]}
    return {"bytes": jbytes + R * (6 * N + 24), "flops": R * (2 * nnz + 4 * N)}


# ---- the same in 64 bits ----------------------------------------------------

def _alpha_beta(case, tau):
    beta = 0.12 * (tau + 0.05 * (1.0 - tau) + tau * (tau - 1.0))
    if case["sched"] == "linear":
        return 0.032 * (1.0 - tau), beta
    return 0.008 * (tau + 4.0 * (1.0 - tau) + 3.0 * tau * (tau - 1.0)), beta


def _leapfrog(case, field, phi, p):
    """Kick and drift of arXiv:2004.03972, Methods; phi and p are (spins, replicas), h = 1."""
    m0, S, dt, window = _start_step(case), case["steps"], 1.0 / case["total"], 100
    w = torch.zeros_like(phi)
    for m in range(m0, m0 + S):
        a, b = _alpha_beta(case, m * dt)
        half, _ = _alpha_beta(case, (m + 0.5) * dt)
        c = 0.5 if m == 0 else 1.0
        p = p - c * (6.0 * a * phi ** 5 + b * field(phi))
        phi = phi + half * p
        if m >= m0 + S - window:
            w += phi
    return phi, p, w / min(S, window)


def _csr64(inst):
    rp, col, val = inst.to_csr()
    return torch.sparse_csr_tensor(torch.from_numpy(np.asarray(rp)), torch.from_numpy(col.astype(np.int64)),
                                   torch.from_numpy(val.astype(np.float64)),
                                   size=(inst.N, inst.N)).cuda()


def _exact_mlp(case, seed):
    x, y = (t.double() for t in _rows(case, seed))
    w = torch.from_numpy(hqa.MLP.init_params(seed)).double().cuda().requires_grad_(True)
    I, H, O = hqa.MLP_IN, hqa.MLP_HIDDEN, hqa.MLP_OUT
    w1, b1, w2, b2, w3, b3 = torch.split(w, [H * I, H, H * H, H, O * H, O])
    a = torch.relu(x @ w1.view(H, I).T + b1)
    a = torch.relu(a @ w2.view(H, H).T + b2)
    z = a @ w3.view(O, H).T + b3
    # summed over the two outputs, mean over the rows
    loss = 2.0 * torch.nn.functional.binary_cross_entropy_with_logits(z, y)
    loss.backward()
    return {"logits": z.detach(), "grad": w.grad, "loss": loss.detach().reshape(1)}


def exact(case, seed):
    op = case["op"]
    if op == "mlp":
        return _exact_mlp(case, seed)
    if op not in ("run", "batch"):
        return None                     # whole numbers only
    if op == "run":
        inst = _instance(case, seed)
        if inst.dense is not None:
            J = torch.from_numpy(inst.dense).cuda()
        else:
            J = _csr64(inst)
        h = 0.0 if inst.h is None else torch.from_numpy(inst.h).cuda()[:, None]
        phi, p = (t.double().T.contiguous() for t in _state(case, seed, inst.N))
        out = _leapfrog(case, lambda f: J @ f + 2.0 * h * f.abs(), phi, p)
        return {k: v.T.contiguous() for k, v in zip(("phi", "p", "phibar"), out)}
    members, R = _members(case, seed), case["R"]
    total = sum(i.N for i in members)
    phi, p = _state(case, seed, total)
    parts, at = [], 0
    for inst in members:                # blocks [R][N_k] back to back
        J = _csr64(inst)
        f, q = (t.reshape(-1)[R * at:R * (at + inst.N)].view(R, inst.N).double().T.contiguous()
                for t in (phi, p))
        out = _leapfrog(case, lambda v, J=J: J @ v, f, q)
        parts.append([v.T.contiguous().reshape(-1) for v in out])
        at += inst.N
    return {k: torch.cat([q[i] for q in parts]).view(R, total)
            for i, k in enumerate(("phi", "p", "phibar"))}
