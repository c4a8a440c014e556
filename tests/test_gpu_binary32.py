"""The binary32 iteration inside FP64 refinement where it still runs -- pinned
solves of CP2 systems, ensembles with a CP1 member, CP1 steps on meshes of more
than two colours -- and the FP64 ensemble on all cells (more colours), with the
teams' stalled waits of both.

Tolerances: 1e-9 (FP64) and 1e-8 (mixed) against the oracle, as in the parity
tests; a claimed residual is checked with the oracle's matrix to a factor of two."""
import dataclasses
import time

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

cps = pytest.importorskip("paper_2309_03543_gb300")
NOT_CONVERGED = cps._cps.ERR_NOT_CONVERGED


@pytest.fixture(scope="module")
def ctx(cuda_device):
    c = cps.Context(0)
    yield c
    c.close()


def _assemble(ctx, p, kind=cps.KIND_CP2):
    m = p.mesh
    return ctx.assemble(m.xy, m.tri, m.dirichlet, p.eps, p.kinv, p.field_loc, kind, p.nu, p.dt)


def _oracle(p, kind=oracle.CP2):
    m = p.mesh
    return oracle.assemble(m.xy, m.tri, m.dirichlet, p.eps, p.kinv, p.field_loc, kind, p.nu, p.dt)


def _walls(p):
    e, j = np.nonzero(oracle.topology(p.mesh.tri) < 0)
    return dataclasses.replace(p, mesh=dataclasses.replace(
        p.mesh, dirichlet=(e * 3 + j).astype(np.int32)))


def _rel(A, b, x):
    return np.linalg.norm(b - A.matvec(x.cpu().numpy())) / np.linalg.norm(b)


MESHES = {"lattice": lambda: synth.channel_block_problem(64, seed=5),
          "defect": lambda: synth.defect_problem(40, seed=3),
          "lattice300": lambda: synth.channel_block_problem(300, seed=8)}


@pytest.mark.parametrize("pc", [cps.PC_JACOBI, cps.PC_IC0])
@pytest.mark.parametrize("mesh", sorted(MESHES))
def test_pinned_mixed_solve(ctx, mesh, pc):
    p = MESHES[mesh]()
    b = synth.rhs(p.mesh, 7)
    A = _oracle(p)
    s = _assemble(ctx, p)
    s.set_precond(pc)
    s.set_solver_path(cps.PATH_STREAM)
    bt = torch.as_tensor(b, device="cuda")
    x, st = s.solve(bt, rtol=1e-10, precision=cps.MIXED)
    assert st.refinements > 1 and _rel(A, b, x) <= 1e-10 * 1.01
    xo, _, _ = oracle.solve_problem(p, b, rtol=1e-13)
    x, st = s.solve(bt, rtol=1e-12, precision=cps.MIXED, check=False)
    assert st.status in (0, NOT_CONVERGED) and st.rel_res < 1e-10
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-8 * np.linalg.norm(xo)
    # a tolerance below what FP64 holds: the refinement ends with its best iterate
    x, st = s.solve(bt, rtol=1e-18, precision=cps.MIXED, check=False)
    assert st.status == NOT_CONVERGED and st.refinements > 1 and st.rel_res < 1e-10
    assert _rel(A, b, x) <= 2 * st.rel_res
    s.free()


def _ensemble(ctx, kind):
    """(systems, oracle matrices, right-hand sides): teams for the first and the
    third member, a CP1 system among CP2 ones, or a mesh of more colours."""
    if kind == "cp1":
        probs = [synth.ensemble_member_problem(nt, seed=70 + i)
                 for i, nt in enumerate((30000, 600, 9000, 2500))]
        kinds = [cps.KIND_CP2, cps.KIND_CP1_X, cps.KIND_CP2, cps.KIND_CP2]
    else:
        probs = [synth.defect_problem(n, seed=5 + i) for i, n in enumerate((120, 18, 68, 36))]
        kinds = [cps.KIND_CP2] * 4
    systems = [_assemble(ctx, p, k) for p, k in zip(probs, kinds)]
    mats = [_oracle(p, oracle.CP2 if k == cps.KIND_CP2 else oracle.CP1_X)
            for p, k in zip(probs, kinds)]
    return probs, kinds, systems, mats, [synth.rhs(p.mesh, 80 + i) for i, p in enumerate(probs)]


CASES = [("cp1", cps.MIXED, 1e-8), ("cp1", cps.FP64, 1e-9), ("colours", cps.FP64, 1e-9)]


@pytest.mark.parametrize("kind,precision,tol", CASES)
def test_one_launch_ensemble_on_all_cells(ctx, kind, precision, tol):
    probs, kinds, systems, mats, bs = _ensemble(ctx, kind)
    bt = [torch.as_tensor(b, device="cuda") for b in bs]
    xs = [torch.zeros_like(b) for b in bt]
    st = cps.solve_batch(systems, bt, xs, rtol=1e-10, precision=precision)
    for A, b, x, t in zip(mats, bs, xs, st):
        assert t.status == 0 and _rel(A, b, x) <= 1e-10 * 1.01
    if precision == cps.MIXED:
        assert st[0].refinements > 1 and st[2].refinements > 1
    xs = [torch.zeros_like(b) for b in bt]
    st = cps.solve_batch(systems, bt, xs, rtol=1e-12, precision=precision, check=False)
    for p, k, b, x, t in zip(probs, kinds, bs, xs, st):
        assert t.status in (0, NOT_CONVERGED) and t.rel_res < 1e-10
        if k == cps.KIND_CP2:
            xo, _, _ = oracle.solve_problem(p, b, rtol=1e-13)
            assert np.linalg.norm(x.cpu().numpy() - xo) <= tol * np.linalg.norm(xo)
    for s in systems:
        s.free()


@pytest.mark.parametrize("kind,precision,tol", CASES)
def test_stalled_team_waits_on_all_cells(ctx, kind, precision, tol):
    probs, kinds, systems, mats, bs = _ensemble(ctx, kind)
    bt = [torch.as_tensor(b, device="cuda") for b in bs]
    xs = [torch.zeros_like(b) for b in bt]
    assert ctx.lib.cps_test_inject(systems[0].handle, 1) == 0
    t0 = time.time()
    st = cps.solve_batch(systems, bt, xs, rtol=1e-10, precision=precision, check=False)
    assert time.time() - t0 < 60
    assert st[0].status == cps._cps.ERR_TIMEOUT and st[2].status == cps._cps.ERR_TIMEOUT
    assert st[1].status == 0 and st[3].status == 0
    for x in xs:
        x.zero_()
    cps.solve_batch(systems, bt, xs, rtol=1e-10, precision=precision)
    for A, b, x in zip(mats, bs, xs):
        assert _rel(A, b, x) <= 1e-10 * 1.01
    for s in systems:
        s.free()


def test_mixed_graph_ensemble_of_pinned_systems(ctx):
    """The host threads' solves of the binary32 iteration, at the same time."""
    probs = [synth.ensemble_member_problem(nt, seed=40 + i) for i, nt in enumerate((600, 9000, 30000, 1200))]
    systems = [_assemble(ctx, p) for p in probs]
    for s in systems:
        s.set_solver_path(cps.PATH_STREAM)
    bs = [synth.rhs(p.mesh, 90 + i) for i, p in enumerate(probs)]
    bt = [torch.as_tensor(b, device="cuda") for b in bs]
    xs = [torch.zeros_like(b) for b in bt]
    ctx.set_batch_path(cps.BATCH_GRAPH)
    try:
        st = cps.solve_batch(systems, bt, xs, rtol=1e-10, precision=cps.MIXED)
    finally:
        ctx.set_batch_path(cps.BATCH_ONE_LAUNCH)
    for p, b, x, t in zip(probs, bs, xs, st):
        assert t.refinements > 1 and _rel(_oracle(p), b, x) <= 1e-10 * 1.01
    for s in systems:
        s.free()


@pytest.mark.parametrize("precision,tol", [(cps.MIXED, 1e-8), (cps.FP64, 1e-9)])
def test_one_launch_cp1_step_on_all_cells(ctx, precision, tol):
    p = _walls(synth.defect_problem(90, seed=3))
    du_b = synth.cell_vector_field(p.mesh, 19, scale=0.05)
    o = oracle.cp1_step(p, du_b, toll=1e-4, rtol=1e-13)
    sx, sy = (_assemble(ctx, p, k) for k in (cps.KIND_CP1_X, cps.KIND_CP1_Y))
    cps.cp1_setup(sx, sy, p.mesh.xy, p.mesh.tri, p.eps, p.kinv)
    for _ in range(6):                                     # also past the step that looks for rows
        du, st = cps.cp1_step(sx, sy, du_b, toll=1e-4, rtol=1e-12, precision=precision)
        assert st["outer"] == o.outer
        assert np.linalg.norm(du.cpu().numpy() - o.du) <= tol * np.linalg.norm(o.du)
    sx.free()
    sy.free()
