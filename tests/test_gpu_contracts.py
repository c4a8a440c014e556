"""Calls at the edges of what the header promises: a zero right-hand side in
the middle of a team's work, iteration bounds, refused pins, unusable first
right-hand sides, and what an unconverged mixed-precision solve returns."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

cps = pytest.importorskip("paper_2309_03543_gb300")


@pytest.fixture(scope="module")
def ctx(cuda_device):
    c = cps.Context(0)
    yield c
    c.close()


def _assemble(ctx, p, kind=cps.KIND_CP2):
    m = p.mesh
    return ctx.assemble(m.xy, m.tri, m.dirichlet, p.eps, p.kinv, p.field_loc, kind, p.nu, p.dt)


def _walls(p):
    """No-slip: every boundary side holds a zero increment."""
    e, j = np.nonzero(oracle.topology(p.mesh.tri) < 0)
    return dataclasses.replace(p, mesh=dataclasses.replace(
        p.mesh, dirichlet=(e * 3 + j).astype(np.int32)))


def _cp1_pair(ctx, p):
    s = [_assemble(ctx, p, k) for k in (cps.KIND_CP1_X, cps.KIND_CP1_Y)]
    cps.cp1_setup(*s, p.mesh.xy, p.mesh.tri, p.eps, p.kinv)
    return s


@pytest.mark.parametrize("n", [20, 150])
@pytest.mark.parametrize("zero", [0, 1])
def test_cp1_step_with_one_zero_component(ctx, n, zero):
    """The component whose right-hand side is zero on every sweep comes out
    zero from any start, the other one as from the oracle (1e-9: both solve to
    1e-12)."""
    p = _walls(synth.centred_block_problem(n, seed=2))     # isotropic: not coupled
    du_b = synth.cell_vector_field(p.mesh, 3, mean=(0.02, 0.01), scale=0.05)
    du_b[zero] = 0.0
    o = oracle.cp1_step(p, du_b, toll=1e-4, rtol=1e-13)
    sx, sy = _cp1_pair(ctx, p)
    for _ in range(3):
        start = torch.full((2, p.mesh.nt), 0.5, dtype=torch.float64, device="cuda")
        du, st = cps.cp1_step(sx, sy, du_b, du=start, toll=1e-4, rtol=1e-12)
        d = du.cpu().numpy()
        assert np.all(d[zero] == 0.0)
        assert np.linalg.norm(d - o.du) <= 1e-9 * np.linalg.norm(o.du)
    sx.free()
    sy.free()
