"""The binary32 iteration inside FP64 refinement where it still runs -- pinned
solves of CP2 systems, ensembles with a CP1 member, CP1 steps on meshes of more
than two colours -- and the FP64 ensemble on all cells (more colours), with the
teams' stalled waits of both.

Tolerances: 1e-9 (FP64) and 1e-8 (mixed) against the oracle, as in the parity
tests; a claimed residual is checked with the oracle's matrix to a factor of two."""
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
