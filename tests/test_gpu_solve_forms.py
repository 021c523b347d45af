"""The substitutions of few tails (one CTA per tail, vectors in shared memory)
against the cluster kernels, bit for bit.

FP64: a system of the largest S that takes the first form, and the same system
with one more tail, whose coupling block is zero, which takes the second. That
tail adds exact zeros to the root, so every other component of x has to be
the same. Mixed precision: the batched form, whose substitutions are those of
the cluster kernels (another tail would move the root's residual terms to
other partial sums).
"""
import pytest
import torch

import bmgen

pytestmark = pytest.mark.gpu


def _solve(bm, d, S):
    solver = bm.BranchKKTSolver(S, d["N"], d["nb"], d["nr"])
    solver.factor(d["D"], d["E"], d["C"], d["R"])
    x = solver.solve(d["r"])
    torch.cuda.synchronize()
    assert solver.query()["status"] == 0
    solver.close()
    return x


def _system(S, N, nb):
    w = bmgen.Workload("f", S, N, nb, max(1, nb // 3), workload_id=95, barrier=(-2.0, 2.0), shared_A=True)
    return bmgen.generate(w, seed=11, device="cuda")


# S the last of the few-tails form; N = 1, at and beside powers of two, and
# more positions than one round of a CTA's teams
@pytest.mark.parametrize("S,N,nb", [(304, 1, 4), (304, 9, 4), (304, 6, 3), (304, 40, 12), (304, 33, 16), (152, 17, 24),
                                    (152, 50, 24)])
def test_few_tails_form_gives_the_cluster_kernels_bits(S, N, nb):
    import paper_2609_29977_gb300 as bm
    d = _system(S, N, nb)
    n, nr = S * N * nb, d["nr"]
    more = {k: torch.cat([d[k], d[k][:1]]) for k in ("D", "E", "C")}
    more["C"][S:] = 0.0
    more.update(R=d["R"], N=N, nb=nb, nr=nr, r=torch.cat([d["r"][:n], d["r"][:N * nb], d["r"][n:]]))
    a, b = _solve(bm, d, S), _solve(bm, more, S + 1)
    assert torch.equal(a[:n], b[:n]) and torch.equal(a[n:], b[-nr:])


# few tails in one CTA each; blocks of 48 with a warp per position, over
# clusters and one CTA per tail; the batch's staged FP64 residual where the
# tail's rows are not a multiple of 32
@pytest.mark.parametrize("S,N,nb", [(304, 1, 4), (304, 2, 4), (304, 8, 6), (304, 33, 12), (304, 40, 24), (152, 13, 48),
                                    (160, 1, 48), (160, 9, 48), (3, 64, 48), (2, 45, 48), (3, 3, 24), (5, 7, 24)])
def test_substitutions_and_residuals_give_the_batched_forms_bits(S, N, nb, tmp_path, monkeypatch):
    import paper_2609_29977_gb300 as bm
    monkeypatch.setenv("BM_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    d = _system(S, N, nb)
    tol = 1e-12   # FP64 residuals, as in the batched form
    solver = bm.BranchKKTSolver(S, N, nb, d["nr"], precision=bm.BM_PREC_FP32_IR, tol=tol)
    solver.factor(d["D"], d["E"], d["C"], d["R"])
    x, info = solver.solve(d["r"]), solver.query()
    solver.close()
    batch = bm.BranchKKTBatch([(S, N, nb, d["nr"])], tol=tol)
    batch.factor([d["D"]], [d["E"]], [d["C"]], [d["R"]])
    (xb,), (ib,) = batch.solve([d["r"]]), batch.query()
    batch.close()
    assert info["status"] == ib["status"] == 0 and info["iters"] == ib["iters"] >= 1
    assert torch.equal(x, xb)


# the root's sums: fewer tails than threads per component and more, components
# that do and do not divide the threads
@pytest.mark.parametrize("S,nr", [(1, 1), (1, 64), (5, 33), (7, 64), (130, 3), (513, 1), (600, 7), (90, 48)])
def test_root_solve_over_sizes(S, nr):
    import paper_2609_29977_gb300 as bm
    from oracle import natural
    w = bmgen.Workload("f", S, 2, 6, nr, workload_id=96, barrier=(-2.0, 2.0), shared_A=True)
    d = bmgen.generate(w, seed=12)
    x = _solve(bm, {k: (v.cuda() if isinstance(v, torch.Tensor) else v) for k, v in d.items()}, S).cpu().numpy()
    assert natural.residual(d["D"], d["E"], d["C"], d["R"], x, d["r"])["eta"] <= 1e-12


# five CTAs per SM where that saves a wave, four beside it
@pytest.mark.parametrize("S,N,nb", [(608, 3, 4), (609, 3, 4), (760, 9, 6), (761, 2, 12), (700, 5, 24), (1217, 2, 6)])
def test_substitutions_with_more_ctas_give_the_batched_forms_bits(S, N, nb, tmp_path, monkeypatch):
    test_substitutions_and_residuals_give_the_batched_forms_bits(S, N, nb, tmp_path, monkeypatch)


# the batched residual with four CTAs per SM (457 to 608 tails), three beside it
@pytest.mark.parametrize("S,N,nb", [(456, 3, 6), (457, 5, 24), (608, 3, 48), (609, 3, 24), (457, 2, 12)])
def test_batched_residual_with_more_ctas_gives_the_same_bits(S, N, nb, tmp_path, monkeypatch):
    test_substitutions_and_residuals_give_the_batched_forms_bits(S, N, nb, tmp_path, monkeypatch)


# nb = 32, which the batch does not take: one CTA per SM and per tail, two, and
# the cluster kernels. The tails beyond the first 152 do not couple to the root,
# and the tolerance stops after the first solve, before any sum over all rows.
@pytest.mark.parametrize("N", [1, 2, 9, 33])
def test_forms_for_few_tails_of_wide_blocks_give_the_same_bits(N):
    import paper_2609_29977_gb300 as bm
    S, nb = 152, 32
    d = _system(S, N, nb)
    n, nr = S * N * nb, d["nr"]
    out = []
    for q in (S, S + 1, 2 * S, 2 * S + 1):
        m = torch.arange(q, device="cuda") % S
        D, E, C = (d[k][m].contiguous() for k in ("D", "E", "C"))
        C[S:] = 0.0
        r = torch.cat([d["r"][:n].reshape(S, -1)[m].reshape(-1), d["r"][n:]])
        solver = bm.BranchKKTSolver(q, N, nb, nr, precision=bm.BM_PREC_FP32_IR, tol=1e-2, flags=bm.BM_FLAG_COUPLING_FP32)
        solver.factor(D, E, C, d["R"])
        x, info = solver.solve(r), solver.query()
        solver.close()
        assert info["status"] == 0 and info["iters"] == 0
        out.append(torch.cat([x[:n], x[-nr:]]))
    assert all(torch.equal(o, out[0]) for o in out)


# the top levels' CTAs have fewer teams from three and from five tails per SM
# on: the first and last tails of a system against the same tails alone
@pytest.mark.parametrize("nb", [24, 32])
@pytest.mark.parametrize("S,N", [(305, 2), (305, 5), (608, 9), (609, 4), (609, 7)])
def test_top_levels_with_fewer_teams_give_the_same_factor(S, N, nb):
    import paper_2609_29977_gb300 as bm
    d = _system(S, N, nb)
    keep = torch.tensor([0, 1, S - 2, S - 1], device="cuda")
    few = {k: d[k][keep].contiguous() for k in ("D", "E", "C")}
    out = []
    for q, D, E, C in ((S, d["D"], d["E"], d["C"]), (4, few["D"], few["E"], few["C"])):
        solver = bm.BranchKKTSolver(q, N, nb, d["nr"], precision=bm.BM_PREC_FP32_IR)
        solver.factor(D, E, C, d["R"])
        assert solver.query()["status"] == 0
        out.append(solver.export_factor())
        solver.close()
    for k in ("Ld", "Ll", "Lr", "F"):
        assert torch.equal(out[0][k][keep], out[1][k]), k


# arrays eight bytes off a 16-byte boundary, which a batch has always taken
@pytest.mark.parametrize("nb", [4, 6, 24, 48])
def test_batch_takes_arrays_eight_bytes_off(nb, tmp_path, monkeypatch):
    import paper_2609_29977_gb300 as bm
    monkeypatch.setenv("BM_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    S, N = 3, 6
    d = _system(S, N, nb)

    def off(t):
        buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
        v = buf[1:].view(t.shape)
        v.copy_(t)
        assert v.data_ptr() % 16 == 8
        return v

    xs = []
    for f in (lambda t: t, off):
        batch = bm.BranchKKTBatch([(S, N, nb, d["nr"])])
        batch.factor([f(d["D"])], [f(d["E"])], [f(d["C"])], [f(d["R"])])
        (x,) = batch.solve([f(d["r"])])
        assert batch.query()[0]["status"] == 0
        batch.close()
        xs.append(x)
    assert torch.equal(*xs)
