"""The pairing of sides in the assembly where its table is crowded: vertices
with fewer, as many and more sides than a line of the table has slots, cells
without a common side (the most sides a mesh can have), a vertex numbering
without locality, and what it has to refuse.

Tolerance: a fan's k cells have angles of 2 pi / k at the hub, their
circumcentres are known to about k / 2 pi rounding errors and lie k / 2 pi
times closer together, so entries agree to a few k^2 / 40 roundings of 1.1e-16
on either side: 1e-13 + 1e-16 k^2.  Columns and counts are equal."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

cps = pytest.importorskip("paper_2309_03543_gb300")


@pytest.fixture(scope="module")
def ctx(cuda_device):
    c = cps.Context(0)
    yield c
    c.close()


def _fan(k):
    """k cells around vertex 0."""
    a = 2 * np.pi * np.arange(k) / k
    xy = np.concatenate([[[0.0, 0.0]], np.stack([np.cos(a), np.sin(a)], 1)])
    i = np.arange(k)
    tri = np.stack([np.zeros(k, int), 1 + i, 1 + (i + 1) % k], 1).astype(np.int32)
    return synth.Mesh(0, xy, tri, np.array([0], np.int32))


def _apart(k):
    """k cells without a common side, one Dirichlet side each."""
    t = np.array([[0.0, 0.0], [1.0, 0.0], [0.4, 0.8]])
    xy = (t[None] + 2.0 * np.arange(k)[:, None, None]).reshape(-1, 2)
    return synth.Mesh(0, xy, np.arange(3 * k, dtype=np.int32).reshape(k, 3),
                      (3 * np.arange(k)).astype(np.int32))


def _renumbered(mesh, seed):
    new = np.random.default_rng(seed).permutation(mesh.nv)
    xy = np.empty_like(mesh.xy)
    xy[new] = mesh.xy
    return synth.Mesh(mesh.n, xy, new[mesh.tri].astype(np.int32), mesh.dirichlet)


MESHES = {f"fan{k}": (lambda k=k: _fan(k), k) for k in (5, 7, 8, 9, 17, 1000)}
MESHES.update({f"apart{k}": (lambda k=k: _apart(k), 1) for k in (1, 2, 64, 1024)})
MESHES.update({f"lattice{n}": (lambda n=n: synth.lattice(n, seed=n), 1) for n in (2, 3, 40)})


@pytest.mark.parametrize("renumber", [False, True])
@pytest.mark.parametrize("name", sorted(MESHES))
def test_sides_pair_up_where_the_table_is_crowded(ctx, name, renumber):
    make, k = MESHES[name]
    mesh = make()
    if renumber:
        mesh = _renumbered(mesh, 5)
    eps = np.linspace(0.4, 1.0, mesh.nv)
    kinv = synth.iso_kinv(synth.kozeny_carman_kinv(eps))
    p = synth.Problem(mesh, eps, kinv, synth.PER_VERTEX)
    s = ctx.assemble(mesh.xy, mesh.tri, mesh.dirichlet, eps, kinv, p.field_loc, cps.KIND_CP2,
                     p.nu, p.dt)
    diag, col, val = (t.cpu().numpy() for t in s.export_matrix())
    nbr = oracle.topology(mesh.tri)
    own = np.arange(mesh.nt)[:, None]
    assert np.array_equal(col.T, np.where(nbr >= 0, nbr, own))
    assert s.info()["n_interior_sides"] == int((nbr >= 0).sum()) // 2
    A = oracle.assemble_problem(p).dense()
    tol = 1e-13 + 1e-16 * k * k
    assert np.all(np.abs(diag - A.diagonal()) <= tol * A.diagonal())
    want = np.where(nbr >= 0, A[own, nbr], 0.0)
    assert np.all(np.abs(val.T - want) <= tol * np.abs(want).max())
    # bitwise symmetric: a side has one coefficient, whichever cell computes it
    e, j = np.nonzero(nbr >= 0)
    back = np.argmax(nbr[nbr[e, j]] == e[:, None], 1)
    assert np.array_equal(val.T[e, j], val.T[nbr[e, j], back])
    s.free()


@pytest.mark.parametrize("k", [3, 20])
def test_a_side_of_more_than_two_cells_is_refused(ctx, k):
    # k cells on the side between vertices 0 and 1, all counter-clockwise
    xy = np.concatenate([[[0.0, 0.0], [1.0, 0.0]], [[0.5, 0.6 + 0.01 * i] for i in range(k)]])
    tri = np.array([[0, 1, 2 + i] for i in range(k)], np.int32)
    eps = np.ones(2 + k)
    with pytest.raises(cps.CpsError) as err:
        ctx.assemble(xy, tri, np.array([0], np.int32), eps, synth.iso_kinv(eps), cps.PER_VERTEX,
                     cps.KIND_CP2, 1.5e-5, 0.225)
    assert err.value.code == cps._cps.ERR_NONMANIFOLD


@pytest.mark.parametrize("kind", [cps.KIND_CP2, cps.KIND_CP1_X])
@pytest.mark.parametrize("where", [(0, 0), (50, 1), (97, 2)])
def test_vertex_ids_out_of_range_are_refused(ctx, kind, where):
    m = synth.lattice(8, seed=0)
    eps = np.ones(m.nv)
    for bad in (m.nv, 2**31 - 1, -1, -2**31):
        tri = m.tri.copy()
        tri[where] = bad
        with pytest.raises(cps.CpsError) as err:
            ctx.assemble(m.xy, tri, m.dirichlet, eps, synth.iso_kinv(eps), cps.PER_VERTEX, kind,
                         1.5e-5, 0.225)
        assert err.value.code == cps._cps.ERR_ARG
