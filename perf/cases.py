"""The work that a user of the solver has it do, as measurable cases.

A case is one pass of a program that solves root-coupled branch-MPC systems
(an interior-point or ADMM loop, a batch of independent problems, a serving
loop) through the public entry points of ``paper_2609_29977_gb300``. The
kinds:

* ``fp64``: BranchKKTSolver in FP64: factor + solve of one system;
* ``ir``: the same with FP32 tails and refinement at the default tolerance;
* ``host``: factor_solve_host, page-locked host buffers in and out;
* ``qp``: bm_assemble_reduced of a branch-MPC QP, then factor + solve;
* ``batch``: BranchKKTBatch over systems of uneven sizes: factor + solve;
* ``serve``: BranchKKTServer: requests of several right-hand sides each,
  submitted together and drained.

Inputs are the seeded MPC-shaped systems of ``bmgen``. ``exact`` solves the
same systems in natural order with plain torch in 64 bits.
"""
import random

import torch

import bmgen
import paper_2609_29977_gb300 as bm

# stage block sizes: those with compiled tail kernels, and others (the
# generic kernels), with nr at most nb
COMPILED_NB = (2, 3, 4, 6, 8, 12, 16, 24, 32, 48)
OTHER_NB = (5, 7, 10, 14, 20)
BATCH_NB = (6, 12, 24, 48)


def listed():
    return [
        # the smallest system of the test and benchmark configurations: every
        # launch and dependent chain shows
        {"name": "fp64_s4_n16_nb4", "kind": "fp64", "S": 4, "N": 16, "nb": 4, "nr": 2, "barrier": 0.0},
        # the medium workload: one interior-point step of a mid-sized problem
        {"name": "fp64_s64_n64_nb12", "kind": "fp64", "S": 64, "N": 64, "nb": 12, "nr": 4, "barrier": 4.0},
        # the largest horizon of the paper's sweep (12 states + 4 inputs, 100 scenarios)
        {"name": "fp64_s100_n160_nb16", "kind": "fp64", "S": 100, "N": 160, "nb": 16, "nr": 16, "barrier": 0.0},
        # the default benchmark workload's sizes in FP64, with the barrier range
        # of the medium, batched, serving and large workloads: at 10^+-6 the
        # 64-bit solution itself is determined to 4e-9 only (measured against
        # exact()), less than what two correct FP64 solvers are compared to
        {"name": "fp64_s512_n128_nb24", "kind": "fp64", "S": 512, "N": 128, "nb": 24, "nr": 8, "barrier": 4.0},
        # a block size without compiled tail kernels, ragged sizes
        {"name": "fp64_s37_n50_nb10", "kind": "fp64", "S": 37, "N": 50, "nb": 10, "nr": 7, "barrier": 2.0},
        # FP32 tails with refinement: the medium workload, the default
        # benchmark workload (its 10^+-6 barrier makes the library refine the
        # coupling columns), and the large request's block size and horizon
        {"name": "ir_s64_n64_nb12", "kind": "ir", "S": 64, "N": 64, "nb": 12, "nr": 4, "barrier": 4.0},
        {"name": "ir_s512_n128_nb24", "kind": "ir", "S": 512, "N": 128, "nb": 24, "nr": 8, "barrier": 6.0},
        {"name": "ir_s512_n256_nb48", "kind": "ir", "S": 512, "N": 256, "nb": 48, "nr": 16, "barrier": 4.0},
        # host buffers end to end: the benchmark's end-to-end measure
        {"name": "host_s512_n128_nb24", "kind": "host", "S": 512, "N": 128, "nb": 24, "nr": 8, "barrier": 4.0},
        # QP data to solution with the paper's quadrotor sizes (12 states, 4 inputs)
        {"name": "qp_s100_n160_nb16", "kind": "qp", "S": 100, "N": 160, "nb": 16, "nr": 4},
        # uneven systems in one batch (the batched workload's draw, fewer and smaller systems)
        {"name": "batch_16", "kind": "batch", "count": 16, "Smax": 128, "Nmax": 128, "shape_seed": 4000},
        # requests that arrive together, four right-hand sides each (the serving workload's draw)
        {"name": "serve_8", "kind": "serve", "count": 8, "Smax": 64, "Nmax": 96, "shape_seed": 5000},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choices(("fp64", "ir", "host", "qp", "batch", "serve"), (4, 4, 1, 1, 1, 1))[0]
    if kind in ("batch", "serve"):
        few = kind == "serve"
        return {"kind": kind, "count": rng.randint(2, 8 if few else 16), "Smax": _log_int(rng, 8, 64 if few else 128),
                "Nmax": _log_int(rng, 16, 96 if few else 128), "shape_seed": rng.randrange(1 << 20)}
    # no drawn system does more work than the largest listed one of its kind
    most = 512 * 256 * 48 ** 3 if kind == "ir" else 512 * 128 * 24 ** 3
    while True:
        S, N = _log_int(rng, 2, 512), _log_int(rng, 4, 256)
        if kind == "qp":
            nx, nu = rng.choice(((4, 2), (6, 2), (12, 4), (16, 8), (18, 6), (24, 8)))
            nb, nr = nx + nu, nu
        else:
            nb = rng.choice(COMPILED_NB[2:]) if kind != "fp64" or rng.random() < 0.8 else rng.choice(OTHER_NB)
            nr = rng.choice((-(-nb // 3), rng.randint(1, nb)))
        if S * N * nb ** 3 <= most:
            break
    case = {"kind": kind, "S": S, "N": N, "nb": nb, "nr": nr}
    if kind != "qp":
        case["barrier"] = rng.choice((0.0, 2.0, 4.0))
    return case


# ---- inputs --------------------------------------------------------------------

def _shapes(case):
    """Sizes of the systems of a batch or of a run of requests."""
    rng = random.Random(case["shape_seed"])
    out = []
    for _ in range(case["count"]):
        S, N = rng.randint(8, max(8, case["Smax"])), rng.randint(16, max(16, case["Nmax"]))
        nb = rng.choice(BATCH_NB)
        out.append((S, N, nb, -(-nb // 3)))
    return out


def _system(S, N, nb, nr, barrier, seed, rhs=1):
    w = bmgen.Workload("case", S, N, nb, nr, barrier=(-barrier, barrier) if barrier else None, shared_A=True)
    d = bmgen.generate(w, seed=seed, device="cuda", with_rhs=False)
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    d["r"] = torch.randn((rhs, S * N * nb + nr), generator=g, device="cuda", dtype=torch.float64)
    return d


def _inputs(case, seed):
    """The systems of a case: a list of dicts D, E, C, R, r."""
    if case["kind"] in ("batch", "serve"):
        rhs = 4 if case["kind"] == "serve" else 1
        return [_system(S, N, nb, nr, 4.0, 7919 * seed + 2 * j, rhs) for j, (S, N, nb, nr) in enumerate(_shapes(case))]
    return [_system(case["S"], case["N"], case["nb"], case["nr"], case["barrier"], 7919 * seed)]


def _qp(case, seed):
    S, N, nb, nr = case["S"], case["N"], case["nb"], case["nr"]
    qp = bmgen.generate_qp(S, N, nb - nr, nr, seed=seed, device="cuda", delta=1e-2)
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    r = torch.randn(S * N * nb + nr, generator=g, device="cuda", dtype=torch.float64)
    return qp, r


def prepare(case, seed):
    kind = case["kind"]
    if kind == "qp":
        qp, r = _qp(case, seed)
        solver = bm.BranchKKTSolver(case["S"], case["N"], case["nb"], case["nr"])
        return {"kind": kind, "qp": qp, "r": r, "x": torch.empty_like(r), "solver": solver}
    systems = _inputs(case, seed)
    if kind == "batch":
        return {"kind": kind, "systems": systems, "rs": [d["r"][0] for d in systems],
                "xs": [torch.empty_like(d["r"][0]) for d in systems], "batch": bm.BranchKKTBatch(_shapes(case))}
    if kind == "serve":
        return {"kind": kind, "systems": systems, "xs": [torch.empty_like(d["r"]) for d in systems],
                "server": bm.BranchKKTServer(8 << 30, slots=8)}
    d = systems[0]
    solver = bm.BranchKKTSolver(case["S"], case["N"], case["nb"], case["nr"],
                                precision=bm.BM_PREC_FP32_IR if kind == "ir" else bm.BM_PREC_FP64)
    if kind == "host":
        host = {k: torch.empty(d[k].shape, dtype=torch.float64, pin_memory=True).copy_(d[k])
                for k in ("D", "E", "C", "R")}
        host["r"] = torch.empty(d["r"].shape[1], dtype=torch.float64, pin_memory=True).copy_(d["r"][0])
        x = torch.empty(d["r"].shape[1], dtype=torch.float64, pin_memory=True)
        return {"kind": kind, "host": host, "x": x, "solver": solver}
    return {"kind": kind, "d": d, "r": d["r"][0], "x": torch.empty_like(d["r"][0]), "solver": solver}


def run(state):
    kind = state["kind"]
    if kind == "host":
        h = state["host"]
        x, code = state["solver"].factor_solve_host(h["D"], h["E"], h["C"], h["R"], h["r"], state["x"])
        return {"x": x, "status": code}
    if kind == "batch":
        ds = state["systems"]
        state["batch"].factor([d["D"] for d in ds], [d["E"] for d in ds], [d["C"] for d in ds], [d["R"] for d in ds])
        return {"x": state["batch"].solve(state["rs"], state["xs"])}
    if kind == "serve":
        server = state["server"]
        for j, (d, x) in enumerate(zip(state["systems"], state["xs"])):
            server.submit(j, d["S"], d["N"], d["nb"], d["nr"], d["D"], d["E"], d["C"], d["R"], d["r"], x)
        done = server.drain()
        return {"x": state["xs"], "status": [c["status"] for c in sorted(done, key=lambda c: c["id"])]}
    d = bm.bm_assemble_reduced(state["qp"]) if kind == "qp" else state["d"]
    state["solver"].factor(d["D"], d["E"], d["C"], d["R"])
    return {"x": state["solver"].solve(state["r"], state["x"])}


# ---- what a pass cannot do without -----------------------------------------------

def work(case):
    """Inputs read once and solutions written once; the flops of a factor in
    natural order (7/3 nb^3 per stage) and of two triangular solves."""
    kind = case["kind"]
    shapes = _shapes(case) if kind in ("batch", "serve") else [(case["S"], case["N"], case["nb"], case["nr"])]
    rhs = 4 if kind == "serve" else 1
    nbytes = flops = 0.0
    for S, N, nb, nr in shapes:
        n = S * N * nb + nr
        flops += bmgen.natural_flops(S, N, nb, nr) + rhs * 6.0 * S * N * nb * nb
        nbytes += 8.0 * 2 * rhs * n
        if kind == "qp":
            nx = nb - nr
            nbytes += 8.0 * S * N * (nx * nx + nx * nr + 2 * nb)
            flops += 1.0 * S * N * nx * nb * (nb + 1)
        else:
            nbytes += 8.0 * S * (N * nb * (nb + 1) / 2 + (N - 1) * nb * nb + nr * nb) + 8.0 * nr * (nr + 1) / 2
    return {"bytes": nbytes, "flops": flops}


# ---- the same results from plain torch in 64 bits ---------------------------------

def _natural_solve(D, E, C, R, rs):
    """K x = r in natural order: every tail is eliminated from its last
    stage to its first, the root Schur complement is solved, and the stages
    follow from first to last. rs: [nrhs, n]."""
    S, N, nb, nr = D.shape[0], D.shape[1], D.shape[2], R.shape[0]
    m = rs.shape[0]
    z = rs[:, :S * N * nb].reshape(m, S, N, nb).permute(1, 2, 3, 0).clone()   # [S, N, nb, m]
    Ls = [None] * N
    for k in range(N - 1, -1, -1):
        Sk = D[:, k]
        if k < N - 1:
            G = torch.cholesky_solve(torch.cat((E[:, k], z[:, k + 1]), 2), Ls[k + 1])
            upd = E[:, k].transpose(1, 2) @ G
            Sk = Sk - upd[:, :, :nb]
            z[:, k] -= upd[:, :, nb:]
        Sk = torch.tril(Sk) + torch.tril(Sk, -1).transpose(1, 2)
        Ls[k] = torch.linalg.cholesky(Sk)
    Ct = C.transpose(1, 2)
    Y = torch.cholesky_solve(torch.cat((Ct, z[:, 0]), 2), Ls[0])
    T = (C @ Y).sum(0)
    root = R - T[:, :nr]
    root = torch.tril(root) + torch.tril(root, -1).T
    x0 = torch.cholesky_solve(rs[:, S * N * nb:].T - T[:, nr:], torch.linalg.cholesky(root))
    x = torch.empty_like(z)
    x[:, 0] = torch.cholesky_solve(z[:, 0] - Ct @ x0, Ls[0])
    for k in range(1, N):
        x[:, k] = torch.cholesky_solve(z[:, k] - E[:, k - 1] @ x[:, k - 1], Ls[k])
    return torch.cat((x.permute(3, 0, 1, 2).reshape(m, -1), x0.T), 1)


def _reduced(qp):
    """The reduced matrix of a branch-MPC QP, K = P + tau I + A^T A / delta
    + (W + delta I)^-1, in blocks."""
    S, N, nx, nu = qp["S"], qp["N"], qp["nx"], qp["nu"]
    nb, delta = nx + nu, qp["delta"]
    diag = torch.cat((qp["q"], qp["rw"]), 2) + qp["tau"] + 1.0 / (qp["w"] + delta)
    AB = torch.cat((qp["A"], qp["B"]), 3)   # x_{k+1} = [A_k B_k] z_k at index k
    D = torch.diag_embed(diag)
    D[:, :, :nx, :nx] += torch.eye(nx, dtype=D.dtype, device=D.device) / delta
    E = torch.zeros((S, N - 1, nb, nb), dtype=D.dtype, device=D.device)
    if N > 1:
        D[:, :N - 1] += AB[:, 1:].transpose(2, 3) @ AB[:, 1:] / delta
        E[:, :, :nx] = -AB[:, 1:] / delta
    B0 = qp["B"][:, 0]
    C = torch.zeros((S, nu, nb), dtype=D.dtype, device=D.device)
    C[:, :, :nx] = -B0.transpose(1, 2) / delta
    R = torch.diag(qp["r0w"] + qp["tau"] + 1.0 / (qp["w0"] + delta)) + (B0.transpose(1, 2) @ B0).sum(0) / delta
    return D, E, C, R


def exact(case, seed):
    if case["kind"] == "qp":
        qp, r = _qp(case, seed)
        return {"x": _natural_solve(*_reduced(qp), r[None])[0]}
    xs = [_natural_solve(d["D"], d["E"], d["C"], d["R"], d["r"]) for d in _inputs(case, seed)]
    if case["kind"] == "batch":
        return {"x": [x[0] for x in xs]}
    if case["kind"] == "serve":
        return {"x": xs, "status": [None] * len(xs)}
    if case["kind"] == "host":
        return {"x": xs[0][0], "status": None}
    return {"x": xs[0][0]}
