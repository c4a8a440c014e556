"""The two-cyclic solves (CG on the explicit Schur rows of a two-coloured
graph) and the resident loop on all cells: at the edges of their forms, on
permuted numberings, from warm starts, at the iteration bound, on input that
is not finite, and from several host threads at once.

Tolerances: two solves to relative residual 1e-12 differ by at most their
errors, within 1e-9 as in the parity tests; a claimed residual is checked with
the exported matrix to a factor of two (rounding of the check itself)."""
import dataclasses
import threading

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

cps = pytest.importorskip("paper_2309_03543_gb300")
CONVERGED = (0, cps._cps.ERR_NOT_CONVERGED)


@pytest.fixture(scope="module")
def ctx(cuda_device):
    c = cps.Context(0)
    yield c
    c.close()


def _assemble(ctx, p, kind=cps.KIND_CP2):
    m = p.mesh
    return ctx.assemble(m.xy, m.tri, m.dirichlet, p.eps, p.kinv, p.field_loc, kind, p.nu, p.dt)


def _shuffled(p, seed):
    """The same mesh with its cells in random order (colours stay, numbering
    has no locality: every block depends on most others)."""
    m = p.mesh
    order = np.random.default_rng(seed).permutation(m.nt)
    back = np.empty_like(order)
    back[order] = np.arange(m.nt)
    d = m.dirichlet
    return dataclasses.replace(p, mesh=dataclasses.replace(
        m, tri=np.ascontiguousarray(m.tri[order]),
        dirichlet=(back[d // 3] * 3 + d % 3).astype(np.int32)))


def _residual(s, b, x):
    diag, col, val = s.export_matrix()
    r = b - diag * x
    for j in range(3):
        r = r - val[j] * x[col[j].long()]
    return float(r.norm() / b.norm())


# rows of one block, one more, ragged last blocks, no rows left for some blocks
@pytest.mark.parametrize("n", [2, 3, 4, 12, 23, 24, 34, 65, 130, 201])
@pytest.mark.parametrize("pc", [cps.PC_JACOBI, cps.PC_IC0, cps.PC_REDUCED])
def test_two_cyclic_solve_matches_the_oracle(ctx, n, pc):
    p = synth.channel_block_problem(n, seed=n)
    b = synth.rhs(p.mesh, 5)
    xo, _, A = oracle.solve_problem(p, b, rtol=1e-13)
    s = _assemble(ctx, p)
    s.set_precond(pc)
    if pc != cps.PC_JACOBI:
        s.set_solver_path(cps.PATH_PERSISTENT_1RED)
    bt = torch.as_tensor(b, device="cuda")
    x, st = s.solve(bt, rtol=1e-12, check=False)
    assert st.status in CONVERGED and st.rel_res < 1e-10
    assert np.linalg.norm(x.cpu().numpy() - xo) / np.linalg.norm(xo) < 1e-9
    r = b - A.matvec(x.cpu().numpy())
    assert np.linalg.norm(r) / np.linalg.norm(b) < 2 * max(st.rel_res, 1e-13)
    _, st2 = s.solve(bt, x=x.clone(), rtol=1e-8)          # warm start: nothing to do
    assert st2.iters == 0
    _, st3 = s.solve(bt, rtol=1e-14, max_iter=1, check=False)
    assert st3.iters <= 1
    s.free()


@pytest.mark.parametrize("pc", [cps.PC_JACOBI, cps.PC_IC0, cps.PC_REDUCED])
@pytest.mark.parametrize("n", [40, 120])
def test_two_cyclic_solve_without_locality(ctx, n, pc):
    p = _shuffled(synth.ensemble_member_problem(2 * (n - 1) ** 2, seed=3), seed=9)
    b = synth.rhs(p.mesh, 6)
    xo, _, _ = oracle.solve_problem(p, b, rtol=1e-13)
    s = _assemble(ctx, p)
    s.set_precond(pc)
    if pc != cps.PC_JACOBI:
        s.set_solver_path(cps.PATH_PERSISTENT_1RED)
    x, st = s.solve(torch.as_tensor(b, device="cuda"), rtol=1e-12, check=False)
    assert st.status in CONVERGED and st.rel_res < 1e-10
    assert np.linalg.norm(x.cpu().numpy() - xo) / np.linalg.norm(xo) < 1e-9
    s.free()


# cells whose rows a block holds on chip whole, with five, four and three
# vectors, and with none (152 SMs), for the Schur rows and for all cells
@pytest.mark.parametrize("n,pc", [(520, cps.PC_REDUCED), (560, cps.PC_REDUCED),
                                  (960, cps.PC_REDUCED), (1100, cps.PC_REDUCED),
                                  (1300, cps.PC_REDUCED), (960, cps.PC_IC0),
                                  (470, cps.PC_JACOBI), (490, cps.PC_JACOBI),
                                  (700, cps.PC_JACOBI), (800, cps.PC_JACOBI),
                                  (900, cps.PC_JACOBI)])
def test_every_resident_form(ctx, n, pc):
    p = synth.centred_block_problem(n, seed=1)
    b = torch.as_tensor(synth.rhs(p.mesh, 2), device="cuda")
    s = _assemble(ctx, p)
    s.set_precond(pc)
    s.set_solver_path(cps.PATH_PERSISTENT_1RED)
    x, st = s.solve(b, rtol=1e-9)
    assert st.rel_res <= 1e-9 and _residual(s, b, x) < 2e-9
    s.free()


def test_iteration_bound_zero_and_non_finite_input(ctx):
    p = synth.channel_block_problem(40, seed=4)
    s = _assemble(ctx, p)
    b = torch.as_tensor(synth.rhs(p.mesh, 1), device="cuda")
    s.solve(b, rtol=1e-10)
    assert s.tuning()["two_cyclic"]
    for k in (0, 1, 2, 7, 8):
        _, st = s.solve(b, rtol=1e-13, max_iter=k, check=False)
        assert st.iters == k and st.status == cps._cps.ERR_NOT_CONVERGED
    x = torch.ones_like(b)
    _, st = s.solve(torch.zeros_like(b), x=x)
    assert st.iters == 0 and torch.all(x == 0)
    for bad in (float("nan"), float("inf")):
        c = b.clone()
        c[17] = bad
        for prec in (cps.FP64, cps.MIXED):
            _, st = s.solve(c, rtol=1e-10, precision=prec, check=False)
            assert st.status != 0
    x, st = s.solve(b, rtol=1e-10)                        # and the next solve is right
    assert _residual(s, b, x) < 2e-10
    s.free()


def test_cp1_systems_keep_the_loop_on_all_cells(ctx):
    p = synth.channel_block_problem(40, seed=4)
    s = _assemble(ctx, p, cps.KIND_CP1_X)
    b = torch.as_tensor(synth.rhs(p.mesh, 1), device="cuda")
    x, _ = s.solve(b, rtol=1e-11)
    assert not s.tuning()["two_cyclic"] and _residual(s, b, x) < 2e-11
    s.free()


def test_solves_on_several_threads_and_streams(ctx):
    """Systems of different sizes (other shared-memory forms of one kernel) are
    solved at the same time."""
    probs = [synth.ensemble_member_problem(c, seed=c) for c in (600, 40000, 2500, 9000, 90000, 1200)]
    systems = [_assemble(ctx, p) for p in probs]
    bs = [torch.as_tensor(synth.rhs(p.mesh, 7), device="cuda") for p in probs]
    for s, b in zip(systems, bs):
        s.solve(b, rtol=1e-6)                             # tuned and set up, one at a time
    torch.cuda.synchronize()
    res = [None] * len(probs)

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(8):
                res[i] = systems[i].solve(bs[i], rtol=1e-10, check=False,
                                          precision=cps.MIXED if i % 2 else cps.FP64)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(probs))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    for s, b, (x, st) in zip(systems, bs, res):
        assert st.status == 0 and _residual(s, b, x) < 2e-10
        s.free()
