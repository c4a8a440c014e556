"""Calls at the edges of what the header promises: a zero right-hand side in
the middle of a team's work, iteration bounds, refused pins, unusable first
right-hand sides, and what an unconverged mixed-precision solve returns."""
import dataclasses
import time

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
    for _ in range(7):                                     # on all cells, then on the Schur rows
        start = torch.full((2, p.mesh.nt), 0.5, dtype=torch.float64, device="cuda")
        du, st = cps.cp1_step(sx, sy, du_b, du=start, toll=1e-4, rtol=1e-12)
        d = du.cpu().numpy()
        assert np.all(d[zero] == 0.0)
        assert np.linalg.norm(d - o.du) <= 1e-9 * np.linalg.norm(o.du)
    sx.free()
    sy.free()


def _colours(nbr):
    """Two colours by breadth-first search from cell 0 (a connected graph)."""
    colour = np.full(nbr.shape[0], -1)
    colour[0], front = 0, [0]
    while front:
        nxt = []
        for e in front:
            for c in nbr[e]:
                if c >= 0 and colour[c] < 0:
                    colour[c] = 1 - colour[e]
                    nxt.append(c)
        front = nxt
    return colour


@pytest.mark.parametrize("n", [16, 24])
def test_step_length_of_the_schur_loop_keeps_53_bits(ctx, n):
    """One step from x = 0 on the Schur rows: alpha = (r.r) / (r.S r), read back
    from the solution (the average over its elements: their own rounding cancels)
    against extended precision.  An emulation in integers of the threads', warps',
    blocks' and the grid's sums gives 1.8e-16 to 2.2e-16 rms over these 24
    right-hand sides where a block's total is rounded once to 53 bits and added
    without further loss, and 5.8e-16 to 7.4e-16 where it is rounded per warp,
    gives its last bit away and is cut to 50 bits in the grid's sum.  The bound is
    between the two (their geometric mean)."""
    ld = np.longdouble
    p = synth.centred_block_problem(n, seed=1)
    nbr = oracle.topology(p.mesh.tri)
    black = _colours(nbr) == 1
    s = _assemble(ctx, p)
    s.set_precond(cps.PC_REDUCED)
    s.set_solver_path(cps.PATH_PERSISTENT_1RED)
    diag, col, val = (v.cpu().numpy() for v in s.export_matrix())
    sc = np.sqrt(diag.astype(ld))
    off = np.where(col == np.arange(p.mesh.nt), ld(0), val.astype(ld) / (sc * sc[col]))

    def rest(y):                                           # E y or E^T y, each colour's rows
        return (off * y[col]).sum(0)

    err = []
    for seed in range(24):
        b = synth.rhs(p.mesh, 100 + seed)
        bt = torch.as_tensor(b, device="cuda")
        x, st = s.solve(bt, rtol=0.0, max_iter=1, check=False)
        assert st.iters == 1
        bh = b.astype(ld) / sc
        r = np.where(black, bh - rest(np.where(black, ld(0), bh)), ld(0))
        sr = np.where(black, r - rest(np.where(black, ld(0), rest(r))), ld(0))
        alpha = (r * r).sum() / (r * sr).sum()
        y = np.where(black, x.cpu().numpy().astype(ld) * sc, ld(0))
        err.append(float(((y * r).sum() / (r * r).sum() - alpha) / alpha))
    rms = float(np.sqrt(np.mean(np.square(err))))
    print("rms error of alpha", rms)
    assert rms < 3.5e-16
    s.free()


def test_mixed_solve_times_no_kernels_it_does_not_run(cuda_device):
    """Above 131072 cells a mixed solve that takes the FP64 loop leaves the binary32
    kernels at their first shapes, untimed.  Shapes pinned for the binary32
    iteration make it run: it replaces residuals, the FP64 loop reports one."""
    c = cps.Context(0)                                     # remembers no size yet
    p = synth.channel_block_problem(300, seed=8)
    s = _assemble(c, p)
    b = torch.as_tensor(synth.rhs(p.mesh, 2), device="cuda")
    _, st = s.solve(b, rtol=1e-10, precision=cps.MIXED)
    tu = s.tuning(cps.MIXED)
    assert st.refinements == 1 and tu["unroll"] == [2, 2, 2] and tu["block"] == [256, 256, 256]
    assert len(set(tu["grid"])) == 1
    s.set_kernel_shapes(cps.MIXED, [1, 4, 2], [608, 152, 608], [256, 256, 256])
    _, st = s.solve(b, rtol=1e-10, precision=cps.MIXED)
    assert st.refinements > 1 and st.rel_res <= 1e-10
    assert s.tuning(cps.MIXED)["unroll"] == [1, 4, 2]
    s.free()
    c.close()


def _rises(p):
    """A right-hand side from whose start x = 0 the residual of CG rises several
    times before it falls."""
    return torch.ones(p.mesh.nt, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("pc", [cps.PC_JACOBI, cps.PC_IC0])
@pytest.mark.parametrize("mesh", ["lattice", "defect"])
@pytest.mark.parametrize("start", ["zero", "better"])
def test_unconverged_mixed_solve_returns_the_least_residual(ctx, pc, mesh, start):
    """Eight iterations, after which the residual is above the start's: the start
    comes back, with its residual, whichever loop ran; from a start better than
    any iterate of a solve that cannot reach its tolerance, no worse a one."""
    p = synth.channel_block_problem(40, seed=4) if mesh == "lattice" else synth.defect_problem(20, seed=3)
    s = _assemble(ctx, p)
    s.set_precond(pc)
    b = _rises(p)
    A = oracle.assemble_problem(p)
    bn = b.cpu().numpy()

    def rel(x):
        return np.linalg.norm(bn - A.matvec(x.cpu().numpy())) / np.linalg.norm(bn)

    if start == "zero":
        x, st = s.solve(b, rtol=1e-13, max_iter=8, precision=cps.MIXED, check=False)
        assert st.status == cps._cps.ERR_NOT_CONVERGED
        assert st.rel_res <= 1.0 + 1e-12 and abs(rel(x) - st.rel_res) <= 1e-9
    else:
        x0, _ = s.solve(b, rtol=1e-10)
        _, st0 = s.solve(b, x=x0.clone(), rtol=1e-10)     # its residual, as the solver forms it
        for k in (2, 4, 40):
            x, st = s.solve(b, x=x0.clone(), rtol=0.0, max_iter=k, precision=cps.MIXED, check=False)
            assert st.status == cps._cps.ERR_NOT_CONVERGED
            assert st.rel_res <= st0.rel_res * (1 + 1e-6) and rel(x) <= 1.05 * st0.rel_res
    s.free()


@pytest.mark.parametrize("mesh", ["lattice", "defect"])
def test_unconverged_mixed_ensemble_returns_the_least_residual(ctx, mesh):
    """Members solved by single blocks and by teams, after eight iterations."""
    sizes = [30000, 600, 9000]
    if mesh == "lattice":
        probs = [synth.ensemble_member_problem(nt, seed=70 + i) for i, nt in enumerate(sizes)]
    else:
        probs = [synth.defect_problem(n, seed=5 + i) for i, n in enumerate((120, 18, 60))]
    systems = [_assemble(ctx, p) for p in probs]
    bs = [_rises(p) for p in probs]
    xs = [torch.zeros_like(b) for b in bs]
    st = cps.solve_batch(systems, bs, xs, rtol=1e-10, max_iter=8, precision=cps.MIXED, check=False)
    for s, b, x, t in zip(systems, bs, xs, st):
        assert t.status == cps._cps.ERR_NOT_CONVERGED and t.iters <= 8
        r = float((b - s.matvec(x)).norm() / b.norm())
        assert t.rel_res <= 1.0 + 1e-12 and abs(r - t.rel_res) <= 1e-9
    # and in FP64 the last iterate, as before
    st = cps.solve_batch(systems, bs, xs, rtol=1e-10, max_iter=8, check=False)
    assert all(t.rel_res > 1.0 for t in st)
    for s in systems:
        s.free()


@pytest.mark.parametrize("pc", [cps.PC_JACOBI, cps.PC_IC0, cps.PC_REDUCED])
@pytest.mark.parametrize("first", ["nan", "inf", "zero"])
def test_the_first_right_hand_side_does_not_choose_the_loop(cuda_device, pc, first):
    """A first solve that cannot iterate leaves the choice that any other one
    does, to its own system and to the next one of its size."""
    c = cps.Context(0)                                     # remembers no size yet
    p = synth.channel_block_problem(60, seed=4)
    good = torch.as_tensor(synth.rhs(p.mesh, 1), device="cuda")
    bad = good.clone() if first != "zero" else torch.zeros_like(good)
    if first != "zero":
        bad[17] = float(first)
    for rhs in (bad, good):
        s = _assemble(c, p)
        s.set_precond(pc)
        s.solve(rhs, rtol=1e-10, check=False)
        x, st = s.solve(good, rtol=1e-10)
        assert st.rel_res <= 1e-10
        tu = s.tuning()
        probe = tu["probe_us_per_iter"]
        # the loop on the Schur rows ran when it was timed, and was the faster one
        if pc == cps.PC_JACOBI:
            assert tu["two_cyclic"] and 1.0 < tu["two_cyclic_us_per_iter"] < 100.0
        elif pc == cps.PC_IC0:
            assert tu["ic0_persistent"] and 1.0 < probe["ic0_persistent"] < 100.0
        else:
            assert tu["reduced_single_reduction"] and 1.0 < probe["reduced_persistent_1red"] < 100.0
        s.free()
    c.close()


def test_max_iter_bounds_the_iterations_made(ctx):
    """On a system whose Jacobi solves count two iterations a step: none leaves x
    as it is, one is the steepest descent step, an odd bound makes one more than
    the even one below and not as many as the next (the energy norm of the error
    falls with every iteration made)."""
    p = synth.channel_block_problem(40, seed=4)
    s = _assemble(ctx, p)
    A = oracle.assemble_problem(p)
    b = torch.as_tensor(synth.rhs(p.mesh, 1), device="cuda")
    s.solve(b, rtol=1e-10)
    assert s.tuning()["two_cyclic"]
    xs, _ = s.solve(b, rtol=1e-12, check=False)
    x0 = xs + 1e-3 * xs.norm() / np.sqrt(p.mesh.nt) * torch.sin(torch.arange(p.mesh.nt, device="cuda").double())

    def energy(x):
        e = (x - xs).cpu().numpy()
        return float(e @ A.matvec(e))

    f = []
    for k in range(10):
        x, st = s.solve(b, x=x0.clone(), rtol=1e-13, max_iter=k, check=False)
        assert st.iters == k and st.status == cps._cps.ERR_NOT_CONVERGED
        r = b.cpu().numpy() - A.matvec(x.cpu().numpy())
        assert abs(np.linalg.norm(r) / float(b.norm()) - st.rel_res) < 1e-6 * st.rel_res
        f.append(energy(x))
        if k == 0:
            assert float((x - x0).norm()) <= 4e-16 * float(x0.norm())
        if k == 1:
            r0 = b - s.matvec(x0)
            d = s.export_matrix()[0]
            z = r0 / d
            x1 = x0 + (r0 @ z) / (z @ s.matvec(z)) * z
            assert float((x - x1).norm()) <= 1e-12 * float((x1 - x0).norm()) + 1e-15 * float(x1.norm())
    assert all(f[k + 1] < f[k] for k in range(2, 9))
    assert f[1] < f[0] and f[2] < f[0]
    s.free()


@pytest.mark.parametrize("sizes", [[600], [30000, 600]])
def test_max_iter_bounds_the_ensembles_iterations(ctx, sizes):
    probs = [synth.ensemble_member_problem(nt, seed=70 + i) for i, nt in enumerate(sizes)]
    systems = [_assemble(ctx, p) for p in probs]
    bs = [torch.as_tensor(synth.rhs(p.mesh, 80), device="cuda") for p in probs]

    def run(k):
        xs = [0.5 * torch.ones_like(b) for b in bs]
        return xs, cps.solve_batch(systems, bs, xs, rtol=1e-13, max_iter=k, check=False)

    for k in (0, 1):
        xs, st = run(k)
        assert all(t.iters == k for t in st)
        if k == 0:
            assert all(bool(torch.all((x - 0.5).abs() <= 1e-15)) for x in xs)
    for k in (2, 6, 7, 9):
        xs, st = run(k)
        assert all(t.iters == k - k % 2 for t in st)
        for u, v in zip(xs, run(k - k % 2)[0]):            # no work beyond what is counted
            assert torch.equal(u, v)
    for s in systems:
        s.free()


def test_max_iter_bounds_the_cp1_steps_solves(ctx):
    p = _walls(synth.channel_block_problem(24, seed=6))
    du_b = synth.cell_vector_field(p.mesh, 9, mean=(0.01, -0.02), scale=0.05)
    sx, sy = _cp1_pair(ctx, p)
    cps.cp1_step(sx, sy, du_b)                             # a coupled pair: on the Schur rows
    for k in (0, 1, 2, 3):
        # the uncoupled sweep only: two solves
        _, st = cps.cp1_step(sx, sy, du_b, max_outer=0, rtol=1e-15, max_iter=k, check=False)
        assert st["solve_iters"] == 2 * (k if k < 2 else 2)
    sx.free()
    sy.free()


@pytest.mark.parametrize("path", [cps.PATH_AUTO, cps.PATH_PERSISTENT_1RED])
def test_ic0_solve_of_no_iteration_leaves_x(ctx, path):
    p = synth.channel_block_problem(40, seed=4)
    s = _assemble(ctx, p)
    s.set_precond(cps.PC_IC0)
    s.set_solver_path(path)
    b = torch.as_tensor(synth.rhs(p.mesh, 1), device="cuda")
    s.solve(b, rtol=1e-6)
    x0 = torch.sin(torch.arange(p.mesh.nt, device="cuda").double())
    x, st = s.solve(b, x=x0.clone(), max_iter=0, check=False)
    assert st.iters == 0 and float((x - x0).norm()) <= 4e-16 * float(x0.norm())
    s.free()


def test_a_refused_pin_changes_nothing(ctx):
    p = synth.channel_block_problem(200, seed=4)           # no cluster holds 79,202 cells
    s = _assemble(ctx, p)
    b = torch.as_tensor(synth.rhs(p.mesh, 1), device="cuda")
    x, st = s.solve(b, rtol=1e-10)
    before = s.tuning()
    assert before["two_cyclic"]
    for path in (-1, 14, 99, cps.PATH_CLUSTER, cps.PATH_CLUSTER_1RED, cps.PATH_CLUSTER_SSTEP2):
        with pytest.raises(cps.CpsError):
            s.set_solver_path(path)
        assert s.tuning() == before
        x2, st2 = s.solve(b, rtol=1e-10)
        assert st2.iters == st.iters and torch.equal(x, x2)
        _, st3 = s.solve(b, rtol=1e-10, precision=cps.MIXED)
        assert st3.refinements == 1                        # the FP64 loop
    s.free()


def test_first_calls_on_fresh_systems_pay_little(ctx):
    """The Schur rows are set up by a system's first solve: for an ensemble of small
    systems in less time than a call takes (2.1 ms before there were rows, 1.1
    with them, the set-up in between)."""
    first, later = [], []
    for rep in range(6):
        probs = [synth.ensemble_member_problem(512, seed=200 + i) for i in range(16)]
        systems = [_assemble(ctx, p) for p in probs]
        bs = [torch.as_tensor(synth.rhs(p.mesh, 80), device="cuda") for p in probs]
        for call in range(3):
            xs = [torch.zeros_like(b) for b in bs]
            torch.cuda.synchronize()
            t = time.perf_counter()
            cps.solve_batch(systems, bs, xs, rtol=1e-10)
            torch.cuda.synchronize()
            if rep:
                (later if call else first).append(time.perf_counter() - t)
        for s in systems:
            s.free()
    print("first", np.median(first), "later", np.median(later))
    assert min(first) < 2.2 * np.median(later)             # (the least: a busy host only adds)


def test_a_graph_of_more_colours_keeps_no_order(ctx):
    """8 bytes a cell that no loop would read: the colouring decides before the order
    is allocated (722,000 cells: 5.8 MB)."""
    p = synth.defect_problem(600, seed=3)
    s = _assemble(ctx, p)
    b = torch.as_tensor(synth.rhs(p.mesh, 1), device="cuda")
    x = torch.zeros_like(b)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s.solve(b, x=x, rtol=1e-3)
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    print("held", held)
    assert not s.tuning()["two_cyclic"] and held < 5 << 20
    s.free()


@pytest.mark.parametrize("n", [40, 150])
def test_first_cp1_step_of_a_pair_pays_little(ctx, n):
    """A pair that settles in one coupled sweep (isotropic) makes its first steps on
    all cells: they take less than twice the later ones on the Schur rows (1.3
    times; with the rows set up by the first step, 2.9 times)."""
    p = _walls(synth.centred_block_problem(n, seed=2))
    du_b = torch.as_tensor(synth.cell_vector_field(p.mesh, 3, mean=(0.02, 0.01), scale=0.05),
                           device="cuda")
    times = []
    for rep in range(6):
        sx, sy = _cp1_pair(ctx, p)
        t = []
        for step in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            _, st = cps.cp1_step(sx, sy, du_b)
            t.append(time.perf_counter() - t0)
            assert st["outer"] == 1
        if rep:
            times.append(t)
        sx.free()
        sy.free()
    t = np.median(np.array(times), axis=0)
    print("steps", 1e3 * t)
    assert min(u[0] for u in times) < 2.0 * min(t[5:])     # (the least: a busy host only adds)


@pytest.mark.parametrize("shuffled", [False, True])
def test_a_pair_whose_systems_number_their_cells_differently(ctx, shuffled):
    """The y system's order is its own where its columns are not the x system's: the
    solve of each of them on the Schur rows matches the oracle's."""
    p = _walls(synth.channel_block_problem(30, seed=6))
    m = p.mesh
    q = p
    if shuffled:
        order = np.random.default_rng(3).permutation(m.nt)
        back = np.argsort(order)
        q = dataclasses.replace(p, mesh=dataclasses.replace(
            m, tri=np.ascontiguousarray(m.tri[order]),
            dirichlet=(back[m.dirichlet // 3] * 3 + m.dirichlet % 3).astype(np.int32)))
    sx = _assemble(ctx, p, cps.KIND_CP1_X)
    sy = _assemble(ctx, q, cps.KIND_CP1_Y)
    cps.cp1_setup(sx, sy, m.xy, m.tri, p.eps, p.kinv)
    du_b = synth.cell_vector_field(m, 9, mean=(0.01, -0.02), scale=0.05)
    cps.cp1_step(sx, sy, du_b, max_outer=3, check=False)   # sets the rows up
    du, _ = cps.cp1_step(sx, sy, du_b, max_outer=0, rtol=1e-12, check=False)
    f = (p.eps, p.kinv, p.field_loc)
    T, _, isd, nbr = oracle.side_coefficients(m.xy, m.tri, m.dirichlet, *f, oracle.CP1_X, p.nu, p.dt)
    for k, (s, r, kind) in enumerate(((sx, p, oracle.CP1_X), (sy, q, oracle.CP1_Y))):
        A = oracle.assemble(m.xy, r.mesh.tri, r.mesh.dirichlet, *f, kind, p.nu, p.dt)
        lap = -oracle.cp1_laplacian(T, nbr, isd, du_b[k])
        assert np.linalg.norm(A.matvec(du[k].cpu().numpy()) - lap) <= 1e-11 * np.linalg.norm(lap)
    sx.free()
    sy.free()


@pytest.mark.parametrize("n,launches", [(400, 3), (900, 4)])
def test_launches_of_the_persistent_loop_are_counted(ctx, n, launches):
    """Start, loop and end; above 1.44M cells the streamed loop has a kernel of its
    own before it."""
    p = synth.centred_block_problem(n, seed=1)
    s = _assemble(ctx, p)
    s.set_solver_path(cps.PATH_PERSISTENT_1RED)
    b = torch.as_tensor(synth.rhs(p.mesh, 2), device="cuda")
    _, st = s.solve(b, rtol=1e-6)                          # one run: far from the FP64 floor
    assert st.launches == launches
    s.free()


@pytest.mark.parametrize("n,vectors,rows", [(200, 5, True), (900, 0, False)])
def test_what_the_persistent_loop_keeps_on_chip_is_reported(cuda_device, n, vectors, rows):
    c = cps.Context(0)                                     # remembers no size yet
    s = _assemble(c, synth.centred_block_problem(n, seed=1))
    assert s.tuning()["resident_vectors"] == 0             # not chosen yet
    s.set_solver_path(cps.PATH_PERSISTENT_1RED)
    tu = s.tuning()
    assert tu["resident_vectors"] == vectors and tu["resident_rows"] == rows
    s.set_solver_path(cps.PATH_STREAM)
    assert s.tuning()["resident_vectors"] == 0
    s.free()
    c.close()
