"""The library's work as its users have it done: what a timing run measures.

A case is one call sequence through the public binding at one size.  The
operations are those of an imaginary-time run and of the measurements along it:

  environment   the exact environment of one bond: the gated composite of the
                current state, a fixed number of warm-started CTM sweeps, the
                bond's metric, and from it the bond's two-spin density matrix
                (its components in the basis of Pauli products)
  gate          one gate layer (eefu_apply_gate): environment, ALS bond update,
                gauge; the updated site tensors come back
  step          one whole Trotter step and the observables after it
  observables   the three mappings' environments, side by side, and <H>, <S>
  batch         trajectories at one or several couplings advanced one Trotter
                step together, with their observables (eefu_evolve_batch)
  gradient      the bond cost's gradient for trial factors (the backward
                direction of the bond update), the environment in hand
  site          the two-layer site contraction alone

A state is a purification with its spins partly aligned, as a bias field
leaves them, plus normal noise of 5 % per entry at D <= 4, as the library's
benchmark and tests start from, and of the same norm at larger D.  Every pass starts again from the same site tensors; the
environments stay in the context from pass to pass and are converged before
the first one, as along a trajectory.  The number of CTM sweeps is fixed
(tolerance < 0), as in the benchmark.

Environment tensors are fixed only up to a rotation of their bonds and a scale,
so the quantities returned are those that both leave alone: the gauge-fixed
site tensors, expectation values, density matrices.  Contexts of a
single-precision kind hold values of that precision, which the C interface
hands out widened to FP64; they come back as the FP32 values that they are.
"""
import math

import numpy as np
import torch

import paper_1906_02220_gb300 as g

DEV = "cuda:0"
GAMMAS = ("x", "y", "z")
ANGLE = 0.3 * math.pi                      # coupling angle of the mixed Kitaev-Heisenberg runs
DBETA = 0.01
SWEEPS, OBS_SWEEPS, START_SWEEPS = 4, 2, 8   # per gate layer, per observables mapping, before the first pass
# the Pauli products on the two spins of a composite (sA, aA, sB, aB) that a real density matrix can hold
PAULI = dict(I=np.eye(2), X=np.array([[0.0, 1.0], [1.0, 0.0]]), Y=np.array([[0.0, -1.0], [1.0, 0.0]]),
             Z=np.diag([1.0, -1.0]))
PAIRS = np.stack([np.kron(np.kron(PAULI[a], np.eye(2)), np.kron(PAULI[b], np.eye(2)))
                  for a, b in ("IX", "IZ", "XI", "XX", "XZ", "YY", "ZI", "ZX", "ZZ")])
ROW = ("E_site", "Hx", "Hy", "Hz", "Ax", "Az", "Bx", "Bz")


def listed():
    return [
        # the small FP64 runs of the duality and closed-form studies: latency only
        dict(name="step D2 chi16 fp64", op="step", D=2, chi=16, prec="fp64"),
        # an FP64 environment beyond the dense projector limit (n = 288, k = 48)
        dict(name="environment D3 chi32 fp64", op="environment", D=3, chi=32, prec="fp64", gamma="x"),
        # a gate layer at a ragged size: chi and n = chi D^2 = 441 odd
        dict(name="gate D3 chi49", op="gate", D=3, chi=49, prec="tf32x3", gamma="y"),
        # the headline run, D = 4 and chi = 64: one step of its trajectory, ...
        dict(name="trajectory D4 chi64", op="batch", D=4, chi=64, prec="tf32x3", problems=1),
        # ... the environment of one of its layers, ...
        dict(name="environment D4 chi64", op="environment", D=4, chi=64, prec="tf32x3", gamma="z"),
        # ... its measurement (three mappings side by side) ...
        dict(name="observables D4 chi64", op="observables", D=4, chi=64, prec="tf32x3"),
        # ... and a scan over couplings, several problems on the GPU at once
        dict(name="batch D4 chi64 x4", op="batch", D=4, chi=64, prec="tf32x3", problems=4),
        # gradient-based bond optimisation: the smallest call
        dict(name="gradient D4 chi64", op="gradient", D=4, chi=64, prec="tf32x3", gamma="y"),
        # the middle size of the batched scans, in BF16
        dict(name="environment D5 chi100 bf16", op="environment", D=5, chi=100, prec="bf16", gamma="z"),
        # the large size of the batched scans
        dict(name="environment D6 chi144", op="environment", D=6, chi=144, prec="tf32x3", gamma="z"),
        # the largest bond dimension
        dict(name="environment D8 chi144", op="environment", D=8, chi=144, prec="tf32x3", gamma="x"),
        # the site contraction of a wide bond
        dict(name="site D6 chi144", op="site", D=6, chi=144, prec="tf32x3", kind=0, frame=1),
    ]


def draw(rng):
    """One case of the same ranges: FP64 at D = 2, 3 and chi = 8..40, single
    precision at D = 3..8 and chi = 24..144 (log-uniform, odd ones among them)."""
    op = rng.choice(("environment",) * 6 + ("gate",) * 3 + ("observables",) * 2 + ("step", "batch", "gradient", "site"))
    if op == "step" or (op in ("environment", "gate") and rng.random() < 0.3):
        c = dict(op=op, D=2 if op == "step" else rng.choice((2, 3)), prec="fp64")
        lo, hi = (8, 40) if op != "step" else (8, 24)
    else:
        bonds = dict(environment=(3, 4, 5, 6, 7, 8), gate=(3,), observables=(3, 4, 5, 6), batch=(3, 4), gradient=(3, 4, 5),
                     site=(3, 4, 5, 6, 7, 8))[op]
        c = dict(op=op, D=rng.choice(bonds), prec=rng.choice(("tf32x3",) * 3 + ("bf16",)))
        if op == "gradient":
            c["prec"] = "tf32x3"
        elif op in ("environment", "gate") and c["D"] <= 4 and rng.random() < 0.2:
            c["prec"] = "fp32"
        lo, hi = (24, 144) if op != "batch" else (24, 80)
    c["chi"] = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if op == "site":
        c.update(kind=rng.randrange(2), frame=rng.randrange(4))
    elif op == "batch":
        c["problems"] = rng.choice((1, 2, 3, 4))
    elif op in ("environment", "gate", "gradient"):
        c["gamma"] = rng.choice(GAMMAS)
    return c


def site_tensors(D, seed):
    """A, B: spin and ancilla entangled at virtual index 0, the up spin the
    likelier one, plus normal noise, unit Frobenius norm (FP64)."""
    rng = np.random.default_rng(seed)
    eps = 0.05 * min(1.0, (4.0 / D) ** 1.5)
    out = []
    for _ in range(2):
        X = eps * rng.standard_normal((2, 2, D, D, D))
        X[0, 0, 0, 0, 0] += 1.0
        X[1, 1, 0, 0, 0] += 0.6
        out.append(torch.as_tensor(X / np.linalg.norm(X), device=DEV))
    return out


def site_operands(case, seed):
    """The site tensor T[p][l][u][r][d] (p = 16) and the blocks Y[b][ib][ik]
    that the enlarged corners of chi^2 blocks hand to the site contraction."""
    D, chi = case["D"], case["chi"]
    rng = np.random.default_rng(seed)
    T = rng.standard_normal((16, D, D, D, D))
    T = torch.as_tensor(T / np.linalg.norm(T), device=DEV)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    Y = torch.randn((chi * chi, D * D, D * D), dtype=torch.float64, device=DEV, generator=gen)
    return T, Y / (chi * D * D)


def context(case):
    return g.Context(case["D"], case["chi"], case["prec"], **({} if case["prec"] == "fp64" else {"proj_fp64": 1}))


def bonds(J, K):
    return [g.bond_hamiltonian(i, J, K[i]) for i in range(3)]


def prepare(case, seed):
    op = case["op"]
    if op == "site":
        T, Y = site_operands(case, seed)
        return dict(case=case, T=T, Y=Y)
    A, B = site_tensors(case["D"], seed)
    s = dict(case=case, A=A, B=B)
    if op == "batch":
        n = case["problems"]
        s["ctx"] = [context(case) for _ in range(n)]
        s["J"] = [math.cos(2 * math.pi * (i + 0.5) / n) for i in range(n)]
        s["K"] = [(2 * math.sin(2 * math.pi * (i + 0.5) / n),) * 3 for i in range(n)]
        run(s)                                       # environments
        return s
    ctx = s["ctx"] = context(case)
    ctx.set_state(A, B)
    J, K = math.cos(ANGLE), (2 * math.sin(ANGLE),) * 3
    s.update(J=J, K=K, H=bonds(J, K))
    if "gamma" in case:
        i = s["slot"] = GAMMAS.index(case["gamma"])
        s["gate"] = g.gate(s["H"][i], DBETA / 2 if i == 2 else DBETA / 4)
        ctx.ctm_build_composite(i, i, s["gate"])
        ctx.ctm_sweep(i, START_SWEEPS)
    if op == "gradient":
        rng = np.random.default_rng(seed + 1)
        shape = (2, 2) + (case["D"],) * 3
        s["trial"] = [torch.as_tensor(0.3 * rng.standard_normal(shape), device=DEV) for _ in range(2)]
    if op in ("observables", "step"):
        ctx.observables(s["H"], ctm_max_sweeps=START_SWEEPS, ctm_tol=-1.0)
    if op == "step":
        run(s)                                       # the gate layers' environments
    return s


def run(s):
    case = s["case"]
    op, single = case["op"], case["prec"] != "fp64"
    if op == "site":
        return g.selftest_site_layered(s["T"], s["Y"], case["kind"], case["frame"],
                                       16 if case["prec"] == "bf16" else 3).float()

    def held(t):
        return t.float() if single else t

    def numbers(v):
        return np.asarray(v, dtype=np.float32 if single else np.float64)

    ctx = s["ctx"]
    if op == "batch":
        for c in ctx:
            c.set_state(s["A"], s["B"])
        rows = g.evolve_batch(ctx, s["J"], s["K"], DBETA, 1, ctm_max_sweeps=SWEEPS, ctm_tol=-1.0,
                              obs_max_sweeps=OBS_SWEEPS, obs_tol=-1.0)
        return numbers([[r[0][k] for k in ROW] for r in rows])
    ctx.set_state(s["A"], s["B"])
    if op == "gradient":
        gA, gB, cost, norm = ctx.cost_gradient(s["slot"], s["gate"], s["trial"][0], s["trial"][1], ctm_max_sweeps=0)
        return [held(gA), held(gB), numbers([cost, norm])]
    if op == "environment":
        ctx.ctm_build_composite(s["slot"], s["slot"], s["gate"])
        ctx.ctm_sweep(s["slot"], SWEEPS)
        return numbers(ctx.ctm_expval(s["slot"], PAIRS))
    if op == "gate":
        ctx.eefu_apply_gate(s["slot"], s["gate"], ctm_max_sweeps=SWEEPS, ctm_tol=-1.0)
        return [held(t) for t in ctx.get_state()]
    out = []
    if op == "step":
        ctx.eefu_trotter_step(s["J"], s["K"], DBETA, ctm_max_sweeps=SWEEPS, ctm_tol=-1.0)
        out = [held(t) for t in ctx.get_state()]
    o = ctx.observables(s["H"], ctm_max_sweeps=OBS_SWEEPS, ctm_tol=-1.0)
    return out + [numbers([o[k] for k in ROW])]


def work(case):
    """Flops of the contractions (ket and bra layers applied in turn, p = 16),
    of the top-chi projection of each move's half-system matrix (one pass over
    it from each side) and of the projectors; bytes of the site tensors, the
    environment (read and written once) and the results."""
    D, chi, op = case["D"], case["chi"], case["op"]
    d2, p, n = D * D, 16, chi * D * D
    word = 8.0 if case["prec"] == "fp64" else 4
    site = 4.0 * p * chi**2 * d2**3
    if op == "site":
        return {"bytes": 8.0 * (2 * chi**2 * d2**2 + p * d2**2), "flops": site}
    corner = 2.0 * chi**3 * d2 + 2.0 * chi**3 * d2**2 + site
    move = 2 * corner + 2.0 * n**3 + 8.0 * n * n * chi + 6.0 * chi**3 * d2 + 4.0 * chi**3 * d2**2 + site
    env = word * 4.0 * chi**2 * (1 + d2)
    metric = 8.0 * chi**3 * d2 + 4.0 * chi**3 * d2**2 + 2.0 * chi**2 * d2**4
    update = 8.0 * d2**3 * d2 + 8.0 * D**9        # one sweep's normal equations
    tensors = 8.0 * 8 * D**3
    if op == "environment":
        return {"bytes": 2 * env + tensors, "flops": 4 * SWEEPS * move + metric}
    if op == "gate":
        return {"bytes": 2 * env + 2 * tensors, "flops": 4 * SWEEPS * move + metric + update}
    if op == "gradient":
        return {"bytes": env + 3 * tensors, "flops": metric + update}
    measured = 3 * (4 * OBS_SWEEPS * move + metric)
    if op == "observables":
        return {"bytes": 6 * env + tensors, "flops": measured}
    step = 5 * (4 * SWEEPS * move + metric + update) + measured
    k = case.get("problems", 1)
    return {"bytes": k * (12 * env + 2 * tensors), "flops": k * step}


def exact(case, seed):
    """The site contraction has a value in 64 bits: out[b][ok][ob] = sum over p,
    ik, ib of TL[ik][p][ok] Y[b][ib][ik] TL[ib][p][ob].  An environment after a
    given number of sweeps of a truncated iteration has none."""
    if case["op"] != "site":
        return None
    T, Y = site_operands(case, seed)
    D = case["D"]
    for _ in range(case["frame"]):
        T = T.permute(0, 2, 3, 4, 1)
    TL = T.permute(1, 2, 0, 3, 4) if case["kind"] == 0 else T.permute(1, 4, 0, 2, 3)
    TL = TL.reshape(D * D, 16, D * D)
    out = torch.empty_like(Y)
    per = max(1, (1 << 27) // (16 * D**4))           # blocks at a time: 1 GB of intermediate
    for b in range(0, Y.shape[0], per):
        Z = torch.einsum("bji,ipo->bjpo", Y[b:b + per], TL)
        out[b:b + per] = torch.einsum("bjpo,jpq->boq", Z, TL)
    return out
