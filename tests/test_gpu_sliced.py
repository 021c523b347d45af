"""Backward error of the tail factor in extended precision: FP64 with sliced
tensor-core products (nb >= 16, csrc/bm_sliced.cuh; plain FMAs below), and the FP32 tails of the
mixed path (csrc/bm_tail_rows.cuh), whose blocks move through shared memory;
and the properties that the digits must not break.

Bound of the backward error: the blocks of L satisfy, entry by entry,
|K - L L^T|_ij <= gamma sqrt(K_ii K_jj) for a backward-stable Cholesky with
gamma = (m + 1) u, u = 2^-53 and m the longest sum behind an entry (Demmel,
"On floating point errors in Cholesky", 1989). An entry of a chain position
gathers two nb-term products per level and the nb terms of its own block:
m = nb (2 levels + 1). The same bound holds for FP64 FMAs; the sliced
products, with one rounding per product, have to meet it as well. FP32 tails:
u = 2^-24, and one more rounding for the inputs (m + 2).
"""
import numpy as np
import pytest
import torch

import bmgen

pytestmark = pytest.mark.gpu

# every compiled block size from 12 up; N at powers of two and beside them
SHAPES = [(2, 9, 12, 4), (1, 17, 16, 16), (2, 6, 16, 5), (2, 13, 24, 8), (1, 2, 24, 8), (1, 8, 32, 11), (1, 5, 48, 16)]


def _bm():
    import paper_2609_29977_gb300 as bm
    return bm


def _gen(S, N, nb, nr, seed=3):
    return bmgen.generate(bmgen.Workload("t", S, N, nb, nr, barrier=(-4.0, 4.0), shared_A=True), seed=seed)


def _run(d, flags=0, precision=0):
    bm = _bm()
    g = {k: (v.cuda() if isinstance(v, torch.Tensor) else v) for k, v in d.items()}
    s = bm.BranchKKTSolver(d["S"], d["N"], d["nb"], d["nr"], precision=precision, flags=flags)
    s.factor(g["D"], g["E"], g["C"], g["R"])
    x = s.solve(g["r"]).cpu().numpy()
    fac = {k: v.cpu().numpy() for k, v in s.export_factor().items()}
    info = s.query()
    s.close()
    return x, fac, info


def _check_backward_error(d, fac, terms, u):
    S, N, nb = d["S"], d["N"], d["nb"]
    D, E = d["D"].numpy(), d["E"].numpy()
    levels = (N - 1).bit_length()
    gamma = (nb * (2 * levels + 1) + terms) * u
    for s in range(S):
        # rows of the tail by chain position p = N + 1 - k; column p of L has
        # the blocks (p, p), (left neighbour, p), (right neighbour, p)
        n = N * nb
        K = np.zeros((n, n), dtype=np.longdouble)
        L = np.zeros((n, n), dtype=np.longdouble)
        at = lambda p: slice((p - 1) * nb, p * nb)  # noqa: E731
        for p in range(1, N + 1):
            k = N - p                                # natural stage index
            K[at(p), at(p)] = np.tril(D[s, k]) + np.tril(D[s, k], -1).T
            if p < N:                                # (stage k+1, stage k) = E[k-1]
                K[at(p), at(p + 1)] = E[s, k - 1]
                K[at(p + 1), at(p)] = E[s, k - 1].T
            L[at(p), at(p)] = np.tril(fac["Ld"][s, k])
            if p < N:
                h = p & -p
                right = p + h if p + h <= N - 1 else N
                L[at(right), at(p)] = fac["Lr"][s, k]
                if p > h:
                    L[at(p - h), at(p)] = fac["Ll"][s, k]
        err = np.abs(K - L @ L.T)
        scale = np.sqrt(np.outer(np.diag(K), np.diag(K)))
        assert float((err / scale).max()) <= gamma, float((err / scale).max()) / gamma


@pytest.mark.parametrize("S,N,nb,nr", SHAPES)
def test_backward_error_of_the_tail_factor(S, N, nb, nr):
    d = _gen(S, N, nb, nr)
    _, fac, info = _run(d)
    assert info["status"] == 0
    _check_backward_error(d, fac, 1, 2.0 ** -53)


# every block size of the staged FP32 tasks, the plain ones (3, 6) beside them
@pytest.mark.parametrize("S,N,nb,nr", [(3, 9, 3, 2), (9, 16, 4, 2), (2, 12, 6, 2), (5, 17, 8, 3), (3, 13, 12, 4),
                                       (3, 7, 16, 5), (2, 21, 24, 8), (1, 6, 32, 11), (2, 11, 48, 16), (1, 2, 48, 3)])
def test_backward_error_of_the_fp32_tail_factor(S, N, nb, nr):
    bm = _bm()
    d = _gen(S, N, nb, nr)
    d["D"], d["E"] = d["D"].float().double(), d["E"].float().double()   # the factor's own inputs
    _, fac, _ = _run(d, precision=bm.BM_PREC_FP32_IR)
    _check_backward_error(d, fac, 2, 2.0 ** -24)


@pytest.mark.parametrize("S,N,nb,nr", [(2, 13, 24, 8), (2, 9, 12, 4)])
def test_scaling_by_powers_of_two_is_exact(S, N, nb, nr):
    """K scaled by an even power of two scales L and x exactly: the digits
    are taken relative to each row's exponent."""
    d = _gen(S, N, nb, nr)
    x, fac, _ = _run(d)
    for k in (600, -600):
        f = 2.0 ** k
        e = dict(d, D=d["D"] * f, E=d["E"] * f, C=d["C"] * f, R=d["R"] * f)
        xs, fs, info = _run(e)
        assert info["status"] == 0
        assert np.array_equal(xs * f, x)
        assert np.array_equal(fs["Lr"] * 2.0 ** (-k // 2), fac["Lr"])


@pytest.mark.parametrize("S,N,nb,nr", [(3, 37, 24, 8), (3, 37, 16, 4), (2, 11, 48, 16)])
def test_team_sizes_and_top_levels_give_the_same_bits(S, N, nb, nr, tmp_path, monkeypatch):
    """Schedules of the cache file, of every compiled team size and two top
    levels, against the default rule."""
    import json
    bm = _bm()
    d = _gen(S, N, nb, nr)
    ref, fac, _ = _run(d, flags=bm.BM_FLAG_NO_TUNE)
    monkeypatch.setenv("BM_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    _run(d)                                          # writes the entry
    path = tmp_path / "tune.json"
    key = next(k for k in json.loads(path.read_text()) if "fp64-schedule" in k)
    for team in (32, 64, 128):
        for top in (2, 3):
            path.write_text(json.dumps({key: [top] + [team] * top}))
            x, f, _ = _run(d)
            assert np.array_equal(x, ref) and all(np.array_equal(f[k], fac[k]) for k in fac), (team, top)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("nb", [12, 24])
def test_non_finite_coupling_is_reported(nb, bad):
    d = _gen(2, 9, nb, 4)
    d["E"] = d["E"].clone()
    d["E"][1, 3, nb - 1, 2] = bad
    _, _, info = _run(d)
    assert info["name"] == "BM_ERR_NOT_SPD" and info["fail_scenario"] == 1


def _units(N, nb, spread, order, seed=8):
    """Exponents of power-of-two units, one per variable of every stage, that
    span 0..spread within each group of eight columns."""
    i = np.arange(nb) % 8
    if order == "alternating":
        e = np.where(i % 2, spread, 0)
    else:
        e = np.round(spread * i / 7.0).astype(int)
        if order == "descending":
            e = spread - e
    e = np.tile(e, (N, 1))
    if order == "shuffled":
        rng = np.random.default_rng(seed)
        for k in range(N):
            for c in range(0, nb, 8):
                rng.shuffle(e[k, c:c + 8])
    return e


def _in_units(d, e):
    """The system of d in variables scaled by s = 2^e: S K S x' = S r, x = S x'."""
    N = d["N"]
    s = torch.from_numpy(2.0 ** e)
    f = dict(d, D=s[:, :, None] * d["D"] * s[:, None, :], C=d["C"] * s[0])
    if N > 1:
        f["E"] = s[1:, :, None] * d["E"] * s[:-1, None, :]
    r = d["r"].clone()
    n0 = d["S"] * N * d["nb"]
    r[:n0] = (r[:n0].reshape(d["S"], N, d["nb"]) * s).reshape(-1)
    f["r"] = r
    return f


@pytest.mark.parametrize("order", ["alternating", "ascending", "descending", "shuffled"])
@pytest.mark.parametrize("spread", [0, 20, 60])
@pytest.mark.parametrize("S,N,nb,nr", [(2, 6, 12, 4), (2, 6, 16, 5), (1, 7, 24, 8), (1, 5, 32, 11), (1, 5, 48, 16)])
def test_variables_of_different_units(S, N, nb, nr, spread, order):
    """The bounds are those of a Cholesky solve whatever the units are: the
    factor's as above, and for x, with two substitutions of the same sums and
    |L| |L^T| <= sqrt(K_ii K_jj), |r - K x|_i <= 3 M u sum_j sqrt(K_ii K_jj) |x_j|
    with M the longest sum of the whole factor (the root's rows gather the
    nb terms of every tail besides); both sides carry s_i, which divides out."""
    from oracle import dense
    d = _gen(S, N, nb, nr)
    e = _units(N, nb, spread, order)
    f = _in_units(d, e)
    x, fac, info = _run(f)
    assert info["status"] == 0
    _check_backward_error(f, fac, 1, 2.0 ** -53)
    n0 = S * N * nb
    xs = x.astype(np.longdouble)
    xs[:n0] *= np.tile(2.0 ** e.reshape(-1), S)          # the solution in d's own variables
    K = dense.assemble_system(d["D"], d["E"], d["C"], d["R"]).astype(np.longdouble)
    r = d["r"].numpy().astype(np.longdouble)
    g = np.sqrt(np.diag(K))
    M = nb * (2 * (N - 1).bit_length() + 1) + S * nb + nr + 1
    bound = 3 * M * 2.0 ** -53 * g * (g * np.abs(xs)).sum()
    ratio = float((np.abs(r - K @ xs) / bound).max())
    assert ratio <= 1.0, ratio


def _check_backward_error_at_the_edge(d, fac):
    """As _check_backward_error (barrier-free systems, u = 2^-53), with the
    subnormal range's absolute rounding: half of 2^-1074 for each of an
    entry's nb (2 levels + 1) operations."""
    S, N, nb = d["S"], d["N"], d["nb"]
    m = nb * (2 * (N - 1).bit_length() + 1)
    for s in range(S):
        from oracle import dense
        K = dense.assemble_tail(d["D"][s], d["E"][s]).astype(np.longdouble)
        L = np.zeros_like(K)
        at = lambda p: slice((N - p) * nb, (N - p + 1) * nb)  # noqa: E731  (stage N + 1 - p)
        for p in range(1, N + 1):
            k = N - p
            L[at(p), at(p)] = np.tril(fac["Ld"][s, k])
            if p < N:
                h = p & -p
                L[at(p + h if p + h <= N - 1 else N), at(p)] = fac["Lr"][s, k]
                if p > h:
                    L[at(p - h), at(p)] = fac["Ll"][s, k]
        g = np.sqrt(np.diag(K))
        bound = (m + 1) * (np.longdouble(2.0) ** -53 * np.outer(g, g) + np.longdouble(2.0) ** -1075)
        ratio = float((np.abs(K - L @ L.T) / bound).max())
        assert ratio <= 1.0, ratio


@pytest.mark.parametrize("S,N,nb,nr", [(2, 6, 12, 4), (2, 6, 16, 5), (1, 7, 24, 8), (1, 5, 32, 11), (1, 5, 48, 16)])
@pytest.mark.parametrize("end", ["subnormal", "largest"])
def test_scales_at_the_ends_of_the_range(S, N, nb, nr, end):
    """K scaled so far down that its entries and pivots are subnormal (below
    2^-1024, where 1/d overflows), or so far up that the largest lie in the
    last binade."""
    w = bmgen.Workload("t", S, N, nb, nr, shared_A=True)
    d = bmgen.generate(w, seed=4)
    top = max(float(d[k].abs().max()) for k in "DECR")
    k = -1033 - int(np.ceil(np.log2(top))) if end == "subnormal" else 1024 - int(np.floor(np.log2(top))) - 1
    # in two steps, so that no factor is itself out of range; r as it is: the
    # solution scales by 2^-k, out of range at the lower end, so r goes along
    f = lambda t: t * 2.0 ** (k // 2) * 2.0 ** (k - k // 2)  # noqa: E731
    e = dict(d, D=f(d["D"]), E=f(d["E"]), C=f(d["C"]), R=f(d["R"]), r=f(d["r"]))
    x, fac, info = _run(e)
    assert info["status"] == 0
    _check_backward_error_at_the_edge(e, fac)
    assert np.isfinite(x).all()


@pytest.mark.parametrize("nb", [12, 16, 24, 32, 48])
@pytest.mark.parametrize("col", [0, 5, -1])
def test_decoupled_variable_with_a_subnormal_pivot(nb, col):
    """A variable that nothing couples to, with a diagonal entry whose
    reciprocal overflows: its factor entry is the square root, the others
    are those of the system without it, and x_c = r_c / d."""
    S, N, nr, s, k = 2, 6, 3, 1, 2
    d = _gen(S, N, nb, nr)
    d = {q: (v.clone() if isinstance(v, torch.Tensor) else v) for q, v in d.items()}
    D, E = d["D"], d["E"]
    D[s, k, col, :] = 0.0
    D[s, k, :, col] = 0.0
    D[s, k, col, col] = 2.0 ** -1030
    E[s, k - 1, col, :] = 0.0
    E[s, k, :, col] = 0.0
    d["r"][((s * N + k) * nb) + col % nb] = 3.0 * 2.0 ** -1030
    x, fac, info = _run(d)
    assert info["status"] == 0
    _check_backward_error(d, fac, 1, 2.0 ** -53)
    assert fac["Ld"][s, k, col, col] == 2.0 ** -515
    assert x[((s * N + k) * nb) + col % nb] == 3.0


@pytest.mark.parametrize("S,N,nb,nr", [(153, 3, 24, 5), (153, 6, 32, 6), (153, 3, 48, 16), (305, 5, 16, 7),
                                       (305, 2, 12, 12), (161, 2, 24, 24)])
def test_top_levels_of_many_tails_give_the_same_factor(S, N, nb, nr):
    """The top kernel's forms for more tails than SMs, and the root's sums a
    warp per entry or 32 entries at a time, against the same tails alone; the
    root against the sum of their U in 64 bits."""
    bm = _bm()
    d = _gen(S, N, nb, nr)
    _, fac, info = _run(d, flags=bm.BM_FLAG_NO_TUNE)
    assert info["status"] == 0
    keep = torch.tensor([0, 1, S - 2, S - 1])
    few = dict(d, S=4, **{k: d[k][keep].contiguous() for k in ("D", "E", "C")})
    few["r"] = torch.ones(4 * N * nb + nr, dtype=torch.float64)
    _, ref, _ = _run(few, flags=bm.BM_FLAG_NO_TUNE)
    for k in ("Ld", "Ll", "Lr", "F"):
        assert np.array_equal(fac[k][keep.numpy()], ref[k]), k
    F = fac["F"].astype(np.longdouble).reshape(S, nr, nb)
    U = np.einsum("sik,sjk->ij", F, F)
    R = np.tril(d["R"].numpy())
    R = R + np.tril(R, -1).T
    L = np.tril(fac["LR"]).astype(np.longdouble)
    # S nb-term sums and nr terms of the Cholesky, each rounded
    g = np.sqrt(np.diag(R).astype(np.longdouble))
    assert float((np.abs(R - U - L @ L.T) / np.outer(g, g)).max()) <= (S + nb + nr + 2) * 2.0 ** -53
