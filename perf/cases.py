"""What a user of this package has it do, as measurable cases.

A case is one call (or the few calls that belong together) through the public
entry points of ``paper_2501_19221_gb300.binding``: whole solves on the
topologies of the benchmark, integration steps that a caller drives itself,
batches of uneven instances, the gradient of the unrolled integrator, exact
energies, and the end-to-end cycle from host arrays to the best vector.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2501_19221_gb300 import binding as B
from paper_2501_19221_gb300 import instances as I

PREC = {"fp32": B.VELOXQ_PREC_FP32, "bf16": B.VELOXQ_PREC_BF16, "fp8": B.VELOXQ_PREC_FP8,
        "fp8_one_term": B.VELOXQ_PREC_FP8_ONE_TERM}
METHOD = {"bsb": B.VELOXQ_METHOD_BSB, "asb": B.VELOXQ_METHOD_ASB, "pa": B.VELOXQ_METHOD_PA}
VTYPE = {"int8": np.int8, "int32": np.int32, "float32": np.float32, "float64": np.float64}

# Schedule constants of the cases that are checked against 64 bits: the
# library's defaults, and c0 near 2 / rho of the instance (rho of a Gaussian
# +-1/sqrt(n) matrix is 2, of the +-J cubic lattice about 5), given so that
# the check does not depend on the estimate made at creation.
DT, A0, SIGMA0, ALPHA = 0.5, 1.0, 0.1, 0.9
C0 = {"sk": 1.0, "lattice": 0.4}


def listed():
    return [
        # the smallest call: an exactly solvable 20-variable QUBO, a solve that is all latency
        {"name": "solve_dense_n20", "op": "solve_dense", "n": 20, "R": 128, "steps": 500, "method": "bsb"},
        # one annealer-sized graph (2048 qubits) with the replicas that fill the GPU, state on chip
        {"name": "solve_chimera_c16", "op": "solve_sparse", "graph": "chimera", "m": 16, "R": 1024, "steps": 500,
         "method": "bsb"},
        # today's annealer graph (5640 qubits, float couplings, irregular rows of up to 15)
        {"name": "solve_pegasus_p16", "op": "solve_sparse", "graph": "pegasus", "m": 16, "R": 1024, "steps": 100,
         "method": "bsb"},
        # the planted 3-XORSAT benchmark after its reduction: 2e5 spins on a random graph, state past L2
        {"name": "solve_xorsat_1e5", "op": "solve_sparse", "graph": "xorsat", "m": 100000, "R": 256, "steps": 100,
         "method": "bsb"},
        # the 3-D lattice of 1e6 spins, a caller that drives the integration itself and keeps its state
        {"name": "steps_lattice_l100", "op": "steps_sparse", "m": 100, "R": 256, "steps": 10, "method": "bsb"},
        # the dense benchmark instance in the default precision
        {"name": "steps_sk_n8192_fp32", "op": "steps_dense", "n": 8192, "R": 1024, "steps": 4, "prec": "fp32",
         "method": "bsb"},
        # an ordinary dense instance at ragged sizes, default precision
        {"name": "steps_sk_n1001_fp32", "op": "steps_dense", "n": 1001, "R": 100, "steps": 20, "prec": "fp32",
         "method": "bsb"},
        # the dense benchmark instance with the field on 8-bit operands
        {"name": "steps_sk_n8192_fp8", "op": "steps_dense", "n": 8192, "R": 1024, "steps": 20, "prec": "fp8",
         "method": "bsb"},
        # hundreds of uneven Wishart instances in one call
        {"name": "batch_wishart_256", "op": "batch", "count": 256, "nmin": 100, "nmax": 2000, "R": 64, "steps": 50,
         "prec": "bf16", "method": "bsb"},
        # the gradient that tunes dt, kappa and the schedule: forward, recomputation and reverse sweep
        {"name": "grad_lattice_l50", "op": "grad", "m": 50, "R": 64, "steps": 40, "ckpt": 10},
        # exact energies of a batch of candidate vectors on the device (post-processing, checking)
        {"name": "energy_dense_n2048", "op": "energy_dense", "n": 2048, "batch": 1024, "vtype": "int32"},
        # from host arrays to the best vector and back to nothing: creation, solve, results, destruction
        {"name": "end_to_end_sk_n4096", "op": "end_to_end", "n": 4096, "R": 256, "steps": 100, "prec": "fp8"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["solve_dense", "solve_sparse", "solve_sparse", "steps_sparse", "steps_dense", "steps_dense",
                     "batch", "grad", "energy_dense", "energy_sparse", "end_to_end"])
    method = rng.choice(["bsb", "bsb", "pa", "asb"])
    if op == "solve_dense":
        return {"op": op, "n": _log(rng, 8, 512), "R": _log(rng, 8, 256), "steps": _log(rng, 50, 500),
                "method": method}
    if op in ("solve_sparse", "energy_sparse"):
        graph = rng.choice(["chimera", "pegasus", "zephyr", "xorsat", "tile", "chain"])
        m = {"chimera": (2, 16), "pegasus": (3, 30), "zephyr": (2, 24), "xorsat": (1000, 100000), "tile": (16, 300),
             "chain": (1000, 300000)}[graph]
        m = _log(rng, *m)
        if graph == "tile":
            m += m % 2
        n = {"chimera": 8 * m * m, "pegasus": 24 * m * (m - 1), "zephyr": 16 * m * (2 * m + 1), "xorsat": 2 * m,
             "tile": m * m, "chain": 2 * m}[graph]
        if op == "energy_sparse":
            batch = max(1, min(_log(rng, 1, 4096), 200_000_000 // n))
            return {"op": op, "graph": graph, "m": m, "batch": batch}
        R = max(1, min(_log(rng, 8, 1024), 50_000_000 // n))
        steps = max(10, min(_log(rng, 20, 500), 2_500_000_000 // (n * R)))
        return {"op": op, "graph": graph, "m": m, "R": R, "steps": steps, "method": method}
    if op == "steps_sparse":
        m = _log(rng, 8, 100)
        R = max(1, min(_log(rng, 8, 512), 250_000_000 // m ** 3))
        return {"op": op, "m": m, "R": R, "steps": rng.randint(1, 10), "method": method}
    if op == "steps_dense":
        prec = rng.choice(["fp32", "fp32", "bf16", "fp8", "fp8_one_term"])
        if prec.startswith("fp8") and method == "asb":
            method = "bsb"
        n, R = _log(rng, 600, 8192), _log(rng, 16, 1024)
        if prec == "fp32" and rng.random() < 0.3:
            n = 8 * (n // 8)
        most = int(2.7e11 // (n * n * R)) if prec == "fp32" else 20
        if method == "pa" and prec == "fp32":
            most = 1        # the operand sign(s) makes later steps jump on the last bit of s
        return {"op": op, "n": n, "R": R, "steps": max(1, min(rng.randint(1, 20), most)), "prec": prec,
                "method": method}
    if op == "batch":
        count = _log(rng, 4, 256)
        return {"op": op, "count": count, "nmin": 100, "nmax": _log(rng, 300, 2000), "R": 16 * rng.randint(1, 8),
                "steps": rng.randint(5, 25 if count > 100 else 50), "prec": rng.choice(["bf16", "fp8"]),
                "method": rng.choice(["bsb", "pa"])}
    if op == "grad":
        m = _log(rng, 6, 50)
        return {"op": op, "m": m, "R": _log(rng, 8, 64), "steps": rng.randint(8, 40), "ckpt": rng.randint(4, 12)}
    if op == "energy_dense":
        return {"op": op, "n": _log(rng, 32, 2500), "batch": _log(rng, 1, 1024),
                "vtype": rng.choice(["int8", "int32", "float32", "float64"])}
    return {"op": op, "n": _log(rng, 100, 4096), "R": 16 * rng.randint(1, 16), "steps": rng.randint(20, 100),
            "prec": rng.choice(["bf16", "fp8"])}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _sk(n, seed):
    """Gaussian couplings J_ij ~ N(0, 1)/sqrt(n), symmetric, zero diagonal (CUDA, float32)."""
    J = torch.randn(n, n, generator=_gen(seed), device="cuda", dtype=torch.float32).triu_(1)
    J = J + J.T
    return J.mul_(1.0 / math.sqrt(n))


def _int_qubo(n, seed, vtype):
    """Symmetric QUBO matrix with entries in [-8, 8], whole numbers for the integer types (CUDA, float64)."""
    g = _gen(seed)
    if vtype.startswith("int"):
        U = torch.randint(-8, 9, (n, n), generator=g, device="cuda").double()
    else:
        U = torch.rand(n, n, generator=g, device="cuda", dtype=torch.float64) * 16.0 - 8.0
        if vtype == "float32":
            U = U.float().double()
    return U.triu() + U.triu(1).T


def _graph(case, seed):
    """(sparse couplings, whether they are an Ising model) of a case's graph."""
    g, m = case["graph"], case["m"]
    if g == "chimera":
        return I.chimera_ising(m, m, 4, seed=seed), True
    if g == "pegasus":
        return I.pegasus_qubo(m, seed=seed), False
    if g == "zephyr":
        return I.zephyr_qubo(m, seed=seed), False
    if g == "tile":
        return I.tile_planted_ising(m, seed=seed).sp, True
    h = I.xorsat_3r3x(m, seed=seed).hubo if g == "xorsat" else I.hubo_chain_3body(m, seed=seed)
    r = B.veloxq_hubo3_reduce(h.n, h.h, h.pairs, h.triples, local=g == "chain")
    return I.SparseCoupling(r["n"], r["rowptr"], r["col"], r["val"], r["lin"]), True


def _sparse_ctx(sp, ising):
    make = B.veloxq_create_ising_csr if ising else B.veloxq_create_csr
    return make(sp.n, sp.rowptr, sp.col, sp.val, sp.lin)


def _start_state(R, n, seed):
    """Positions and momenta as a run starts with them: uniform in [-sigma0, sigma0)."""
    g = _gen(seed + 7919)
    S = torch.rand(R, n, generator=g, device="cuda").mul_(2 * SIGMA0).sub_(SIGMA0)
    Y = torch.rand(R, n, generator=g, device="cuda").mul_(2 * SIGMA0).sub_(SIGMA0)
    return S, Y


def _schedule(case, c0=None):
    kw = {"method": METHOD[case.get("method", "bsb")], "prec": PREC[case.get("prec", "fp32")]}
    if c0 is not None:
        kw["c0"] = c0
    if case["op"] == "batch" or case["op"] == "end_to_end":
        kw["readout_every"] = 0
    if case["op"] == "grad":
        kw.update(readout_every=0, knots=[0.0, 0.5, 1.0])
    return B.make_schedule(**kw)


def _wishart(case, seed):
    """The batch's Ising couplings -J~ (host float32), drawn as the Wishart ensemble's: planted t, W of alpha n
    columns orthogonal to it."""
    g = _gen(seed)
    out = []
    for n in I.wishart_sizes(case["count"], case["nmin"], case["nmax"], seed=0):
        n = int(n)
        t = torch.randint(0, 2, (n, 1), generator=g, device="cuda").float().mul_(2).sub_(1)
        z = torch.randn(n, max(1, round(0.75 * n)), generator=g, device="cuda")
        W = math.sqrt(n / (n - 1.0)) * (z - t @ (t.T @ z) / n)
        J = (W @ W.T) / n
        J = 0.5 * (J + J.T)
        J.fill_diagonal_(0.0)
        out.append(J.cpu().numpy())
    return out


def prepare(case, seed):
    op, st = case["op"], {"case": case, "seed": int(seed) % 1_000_003}
    s = st["seed"]
    if op == "solve_dense":
        Q = _int_qubo(case["n"], s, "int32").to(torch.int32).cpu().numpy()
        st["ctx"] = B.veloxq_create_dense(Q)
        st["sched"] = _schedule(case)
    elif op == "solve_sparse":
        st["ctx"] = _sparse_ctx(*_graph(case, s))
        st["sched"] = _schedule(case)
    elif op == "steps_sparse":
        sp = I.cubic_lattice_ising(case["m"], seed=s)
        st["ctx"] = _sparse_ctx(sp, True)
        st["sched"] = _schedule(case, C0["lattice"])
        st["S0"], st["Y0"] = _start_state(case["R"], sp.n, s)
        st["S"], st["Y"], st["F"] = (torch.empty_like(st["S0"]) for _ in range(3))
    elif op == "steps_dense":
        st["ctx"] = B.veloxq_create_ising_dense(_sk(case["n"], s).cpu().numpy())
        st["sched"] = _schedule(case, C0["sk"])
        st["S0"], st["Y0"] = _start_state(case["R"], case["n"], s)
        st["S"], st["Y"], st["F"] = (torch.empty_like(st["S0"]) for _ in range(3))
    elif op == "batch":
        st["ctxs"] = [B.veloxq_create_ising_dense(J) for J in _wishart(case, s)]
        st["sched"] = _schedule(case)
    elif op == "grad":
        st["ctx"] = _sparse_ctx(I.cubic_lattice_ising(case["m"], seed=s), True)
        st["sched"] = _schedule(case, C0["lattice"])
    elif op in ("energy_dense", "energy_sparse"):
        if op == "energy_dense":
            Q = _int_qubo(case["n"], s, case["vtype"]).cpu().numpy().astype(VTYPE[case["vtype"]])
            st["ctx"] = B.veloxq_create_dense(Q)
        else:
            st["ctx"] = _sparse_ctx(*_graph(case, s))
        n, b = st["ctx"].info.n, case["batch"]
        st["X"] = torch.randint(0, 2, (b, n), generator=_gen(s + 1), device="cuda", dtype=torch.uint8)
        st["E"] = torch.zeros(b, device="cuda", dtype=torch.float64)
        st["E_int"] = torch.zeros(b, device="cuda", dtype=torch.int64) if st["ctx"].info.is_integer else None
    elif op == "end_to_end":
        J = _sk(case["n"], s).cpu().numpy()
        st["Q"] = torch.from_numpy(J).pin_memory().numpy()
        st["sched"] = _schedule(case)
    else:
        raise ValueError(op)
    torch.cuda.synchronize()
    return st


def run(state):
    case, op = state["case"], state["case"]["op"]
    if op in ("solve_dense", "solve_sparse"):
        return B.veloxq_solve(state["ctx"], case["R"], case["steps"], state["sched"], seed=state["seed"])
    if op in ("steps_sparse", "steps_dense"):
        # the caller keeps its start state and advances a copy of it
        S, Y, F = state["S"], state["Y"], state["F"]
        S.copy_(state["S0"])
        Y.copy_(state["Y0"])
        B.veloxq_steps_dev(state["ctx"], case["R"], 0, case["steps"], 200, state["sched"], S, Y, F)
        return {"S": S, "Y": Y, "F": F}
    if op == "batch":
        out = B.veloxq_solve_batch(state["ctxs"], case["R"], case["steps"], state["sched"], seed=state["seed"])
        return {"E": out["E"], "x": np.concatenate(out["x"])}
    if op == "grad":
        return B.veloxq_grad(state["ctx"], case["R"], case["steps"], state["sched"], seed=state["seed"],
                             ckpt_every=case["ckpt"])
    if op in ("energy_dense", "energy_sparse"):
        B.veloxq_energy_dev(state["ctx"], state["X"], state["E"], state["E_int"])
        return {"E": state["E"], "E_int": state["E_int"]}
    ctx = B.veloxq_create_dense(state["Q"])
    out = B.veloxq_solve(ctx, case["R"], case["steps"], state["sched"], seed=state["seed"])
    ctx.destroy()
    return out


# ---------------------------------------------------------------- what a pass cannot do without
_DEGREE = {"chimera": 5.75, "pegasus": 14.4, "zephyr": 19.3, "xorsat": 6.0, "tile": 4.0, "chain": 7.0}


def _sparse_size(case):
    g, m = case["graph"], case["m"]
    n = {"chimera": 8 * m * m, "pegasus": 24 * m * (m - 1), "zephyr": 16 * m * (2 * m + 1), "xorsat": 2 * m,
         "tile": m * m, "chain": 2 * m}[g]
    per = 5 if g in ("chimera", "tile") else 8      # column and weight of a coupling
    return n, n * _DEGREE[g], per


def work(case):
    op = case["op"]
    if op == "solve_dense":
        n, R, K = case["n"], case["R"], case["steps"]
        return {"bytes": 4 * n * n + 8 * R + n, "flops": 2.0 * n * n * R * K}
    if op == "solve_sparse":
        n, nnz, per = _sparse_size(case)
        R, K = case["R"], case["steps"]
        return {"bytes": per * nnz + 8 * n + 8 * R + n, "flops": (2.0 * nnz + 8 * n) * R * K}
    if op == "steps_sparse":
        n, R, K = case["m"] ** 3, case["R"], case["steps"]
        return {"bytes": 30 * n + 20 * n * R, "flops": (12.0 + 8) * n * R * K}
    if op == "steps_dense":
        n, R, K = case["n"], case["R"], case["steps"]
        terms = 2 if case["prec"] == "fp8" else 1
        return {"bytes": 4 * n * n + 20 * n * R, "flops": 2.0 * terms * n * n * R * K}
    if op == "batch":
        nmin, nmax = case["nmin"], case["nmax"]
        n2 = case["count"] * (nmax ** 3 - nmin ** 3) / (3.0 * (nmax - nmin))     # sum of n^2, n uniform
        b = 2 if case["prec"] == "bf16" else 1
        return {"bytes": b * n2, "flops": 2.0 * n2 * case["R"] * case["steps"]}
    if op == "grad":
        n, R, K = case["m"] ** 3, case["R"], case["steps"]
        return {"bytes": 30 * n, "flops": 3.0 * (12.0 + 8) * n * R * K}
    if op == "energy_dense":
        n, b = case["n"], case["batch"]
        return {"bytes": np.dtype(VTYPE[case["vtype"]]).itemsize * n * n + n * b + 8 * b, "flops": 2.0 * n * n * b}
    if op == "energy_sparse":
        n, nnz, per = _sparse_size(case)
        return {"bytes": per * nnz + 8 * n + n * case["batch"] + 8 * case["batch"], "flops": nnz * case["batch"]}
    n, R, K = case["n"], case["R"], case["steps"]
    return {"bytes": 4 * n * n + n + 8 * R, "flops": 2.0 * n * n * R * K}


# ---------------------------------------------------------------- 64 bits
def _advance(field, S, Y, steps, K, method, c0, a=None, dt=DT, b=0.0):
    """`steps` steps of the integrator in the type of S; returns the state and the last field. With `a` (values
    of a(t) per step) instead of the default ramp over K steps."""
    F = None
    for k in range(steps):
        ak = a[k] if a is not None else A0 * k / (K - 1)
        op = torch.where(S > 0, 1.0, -1.0).to(S.dtype) if method == "pa" else S
        F = field(op)
        phi = -0.5 * (F + b)
        if method == "pa":
            Y = ALPHA * Y - dt * ((A0 - ak) / A0 * S - c0 * phi)
            S = (S + Y).clamp(-1.0, 1.0)
        elif method == "asb":
            Y = Y + dt * (-(S * S + A0 - ak) * S + c0 * phi)
            S = S + dt * A0 * Y
        else:
            Y = Y + dt * (-(A0 - ak) * S + c0 * phi)
            S = S + dt * A0 * Y
            hit = S.abs() > 1.0
            Y = torch.where(hit, torch.zeros_like(Y), Y)
            S = torch.where(hit, torch.sign(S.detach()), S)
    return S, Y, F


def _philox_state(R, n, seed):
    """The Philox4x32-10 start state (Salmon et al., SC'11) of a run, variable-major: counter (i, 0, r, 0), key the
    seed; words 0 and 1 as 24-bit uniforms give s and y."""
    i, r = np.meshgrid(np.arange(n, dtype=np.uint64), np.arange(R, dtype=np.uint64), indexing="ij")
    m32 = np.uint64(0xFFFFFFFF)
    c = [i.ravel(), np.zeros(n * R, np.uint64), r.ravel(), np.zeros(n * R, np.uint64)]
    k = [np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)]
    for _ in range(10):
        p, q = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(q >> np.uint64(32)) ^ c[1] ^ k[0], q & m32, (p >> np.uint64(32)) ^ c[3] ^ k[1], p & m32]
        k = [(k[0] + np.uint64(0x9E3779B9)) & m32, (k[1] + np.uint64(0xBB67AE85)) & m32]
    u = [(w >> np.uint64(8)).astype(np.float64) * 2.0 ** -24 for w in c[:2]]
    return tuple(torch.from_numpy((SIGMA0 * (2 * v - 1)).astype(np.float32)).cuda().double().view(n, R) for v in u)


def _lattice_field(sp):
    """The field of a lattice whose rows hold six couplings, on variable-major states [n][R]."""
    col = torch.from_numpy(sp.col.astype(np.int64).reshape(sp.n, 6)).cuda()
    val = torch.from_numpy(sp.val.reshape(sp.n, 6)).cuda().double()

    def field(S):
        F = torch.zeros_like(S)
        for d in range(6):
            F = F + S[col[:, d]] * val[:, d:d + 1]
        return F
    return field


def exact(case, seed):
    op, s = case["op"], int(seed) % 1_000_003
    if op == "steps_dense":
        Q = _sk(case["n"], s).double()
        S, Y = _start_state(case["R"], case["n"], s)
        S, Y, F = _advance(lambda o: o @ Q, S.double(), Y.double(), case["steps"], 200, case["method"], C0["sk"])
        return {"S": S, "Y": Y, "F": F}
    if op == "steps_sparse":
        sp = I.cubic_lattice_ising(case["m"], seed=s)
        S, Y = _start_state(case["R"], sp.n, s)
        S, Y, F = _advance(_lattice_field(sp), S.double().T.contiguous(), Y.double().T.contiguous(), case["steps"],
                           200, case["method"], C0["lattice"])
        return {"S": S.T.contiguous(), "Y": Y.T.contiguous(), "F": F.T.contiguous()}
    if op == "energy_dense":
        Q, whole = _int_qubo(case["n"], s, case["vtype"]), case["vtype"].startswith("int")
        X = torch.randint(0, 2, (case["batch"], case["n"]), generator=_gen(s + 1), device="cuda", dtype=torch.uint8)
        E = ((X.double() @ Q) * X.double()).sum(1)
        return {"E": E, "E_int": E.round().to(torch.int64) if whole else None}
    if op == "grad":
        sp, K, R = I.cubic_lattice_ising(case["m"], seed=s), case["steps"], case["R"]
        field = _lattice_field(sp)
        S, Y = _philox_state(R, sp.n, s)
        dt, c0, knots = (torch.tensor(v, device="cuda", dtype=torch.float64, requires_grad=True)
                         for v in (DT, C0["lattice"], [0.0, 0.5, 1.0]))
        t = torch.arange(K, device="cuda", dtype=torch.float64) * (2.0 / max(K - 1, 1))
        j = t.floor().clamp(max=1).long()
        a = knots[j] * (1 - (t - j)) + knots[j + 1] * (t - j)
        S, Y, _ = _advance(field, S, Y, K, K, "bsb", c0.float().double(), a, dt)
        loss = 0.25 * (S * field(S)).sum() / R - 0.25 * float(sp.val.astype(np.float64).sum())
        loss.backward()
        return {"loss": loss.detach(), "d_dt": dt.grad, "d_kappa": c0.grad, "d_knots": knots.grad}
    return None
