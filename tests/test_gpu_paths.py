"""The routes a multigrid solve can take (which kernels run which levels of a
V-cycle) reach the same solution with the same iteration."""
import numpy as np
import pytest

from gpu_helpers import oracle_plane
from paper_2606_17636_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ps():
    import paper_2606_17636_gb300 as m
    m.lib()
    return m


def _planes(shape, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


# n_r, n_tz, smoothing counts of the levels that fit in shared memory (0: the level-0 counts)
FP64_GRIDS = [(16, 16, 0, 0), (32, 32, 0, 0), (64, 32, 3, 1), (32, 64, 1, 2), (128, 64, 0, 0)]


@pytest.mark.parametrize("nr,nt,nu1f,nu2f", FP64_GRIDS)
def test_fp64_levels_run_level_wide(ps, nr, nt, nu1f, nu2f):
    """FP64: every level above the coarsest on the line passes, with its own
    smoothing counts; the direct solution to 1e-10 at a relative residual of
    1e-12, and the oracle's cycle counts for equal counts on all levels."""
    import scipy.sparse.linalg as spla

    from oracle import mg, operator
    sp = workloads.spec(workloads.SPHERICAL, nr, nt, 8, workloads.LOG, 1.0, 8.0)
    s = ps.Solver.from_spec(sp, precision=ps.FP64, use_graph=False)
    if nu1f:
        s.set_schedule(2, 2, 2, nu_pre_fused=nu1f, nu_post_fused=nu2f)
    f = _planes((s.n_modes, nt, nr), nr + nt)
    u, cyc, rc = s.stage_mg_solve(torch.from_numpy(f).cuda(), tol=1e-12)
    assert rc == ps.OK
    u = u.cpu().numpy()
    p = oracle_plane(sp)
    H = mg.Hierarchy(p)
    for m in (0, 1, s.n_modes - 1):
        A = operator.matrix(p, m).tocsc()
        b = f[m].T
        x = spla.spsolve(A, operator.to_vec(b.real)) + 1j * spla.spsolve(A, operator.to_vec(b.imag))
        ref = operator.from_vec(x, nr, nt).T
        assert np.abs(u[m] - ref).max() <= 1e-10 * np.abs(ref).max()
        if not nu1f:
            assert abs(cyc[m] - H.solve(m, b, 1e-12)[1]) <= 1
    s.close()


# n_r, n_tz, n_phi, SOR sweeps.  Above 1.5 M cells over all planes lines of 32 to
# 512 cells are relaxed in registers (16 cells a lane at 512; column tiles of at
# most 30 pairs a warp; segments of columns); the others, 4 sweeps and lines of
# 16 cells stay with the staged passes, whose sizes are here too.
SMOOTH_GRIDS = [(32, 32, 4, 2), (64, 16, 4, 2), (512, 32, 4, 2), (32, 512, 4, 3), (32, 256, 512, 2), (256, 32, 512, 1),
                (64, 64, 1024, 3), (128, 128, 256, 2), (512, 32, 256, 2), (32, 512, 256, 2), (512, 64, 128, 3), (64, 512, 128, 1),
                (512, 512, 16, 2), (256, 128, 128, 4)]


@pytest.mark.parametrize("nr,nt,n_phi,n_sor", SMOOTH_GRIDS)
def test_level_wide_smoothing_of_every_line_length(ps, nr, nt, n_phi, n_sor):
    """Two cycles on the finest level against the oracle's Algorithm 1 in some
    modes (FP32 rounding through the sweeps: 2e-5 of the largest value, as for
    the stage tests)."""
    from oracle import mg
    sp = workloads.spec(workloads.CYLINDRICAL, nr, nt, n_phi, workloads.UNIFORM, 1.0, 2.0, 0.0, nt / nr)
    s = ps.Solver.from_spec(sp, precision=ps.MIXED, use_graph=False)
    s.set_schedule(2, 2, n_sor)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(nr + nt)
    e0 = torch.randn((s.n_modes, nt, nr), generator=gen, dtype=torch.complex64, device="cuda")
    f = torch.randn((s.n_modes, nt, nr), generator=gen, dtype=torch.complex64, device="cuda")
    got = s.stage_smooth(0, e0.clone(), f, 2)
    H = mg.Hierarchy(oracle_plane(sp), n_sor=n_sor)
    for m in (0, s.n_modes - 1):
        u = np.zeros((nr + 2, nt + 2), complex)
        u[1:-1, 1:-1] = e0[m].cpu().numpy().T
        H.smooth(0, m, u, f[m].cpu().numpy().T.astype(complex), 2)
        ref = u[1:-1, 1:-1].T
        assert np.abs(got[m].cpu().numpy() - ref).max() <= 2e-5 * np.abs(ref).max()
    s.close()


# finest level 256 x 128 (one level above the shared-memory ones) and 512 x 256
# (two), schedules that need one or several launches a leg or none at all
FEW = [(256, 128, (2, 1, 2, 3, 1)), (256, 128, (3, 2, 2, 0, 0)), (256, 128, (1, 1, 1, 0, 0)), (256, 128, (2, 2, 3, 0, 0)),
       (256, 128, (2, 2, 5, 0, 0)), (512, 256, (2, 2, 2, 0, 0)), (256, 256, (2, 1, 2, 0, 0)), (512, 32, (2, 2, 2, 0, 0))]


@pytest.mark.parametrize("nr,nt,sched", FEW)
def test_last_planes_take_the_window_passes_with_the_same_result(ps, nr, nt, sched):
    """A plane's iteration does not depend on how many others are active: the
    level-wide passes and, for the last few, the passes on windows give the same
    bits (mixed path), and the same cycle counts."""
    sp = workloads.spec(workloads.CYLINDRICAL, nr, nt, 64, workloads.UNIFORM, 1.0, 3.0, 0.0, 2.0 * nt / nr)
    s = ps.Solver.from_spec(sp, precision=ps.MIXED, use_graph=False)
    s.set_schedule(*sched[:3], nu_pre_fused=sched[3], nu_post_fused=sched[4])
    f = torch.from_numpy(_planes((s.n_modes, nt, nr), 5)).cuda()
    u, cyc, rc = s.stage_mg_solve(f, tol=1e-8)
    assert rc == ps.OK
    for modes in ([0], [1, 7, 32]):
        g = torch.zeros_like(f)
        g[modes] = f[modes]
        v, cyc2, rc = s.stage_mg_solve(g, tol=1e-8)
        assert rc == ps.OK
        assert torch.equal(v[modes], u[modes]) and [cyc2[m] for m in modes] == [cyc[m] for m in modes]
        assert torch.count_nonzero(v) == torch.count_nonzero(v[modes])
    s.close()


# n_r, n_tz, large coarsest level, smoothing counts, SOR sweeps, whole polar
# range: the first fused level as patches of 4 rows (8192 cells) and of 2
# (4096 cells), a level below it, both forms of the coarsest solve, factors
# beside the levels and over the right-hand side
PATCH_GRIDS = [(256, 128, True, 2, 2, 2, True), (128, 64, True, 1, 1, 2, True), (64, 128, True, 3, 1, 1, True),
               (128, 64, True, 2, 1, 2, False), (128, 32, True, 2, 2, 3, True), (64, 64, False, 1, 2, 2, True),
               (32, 128, False, 2, 2, 2, True), (128, 64, False, 2, 2, 2, True), (16, 256, False, 2, 2, 2, True)]


@pytest.mark.parametrize("nr,nt,large,nu1,nu2,n_sor,whole", PATCH_GRIDS)
def test_fused_first_level_held_in_registers(ps, nr, nt, large, nu1, nu2, n_sor, whole):
    """The fused V-cycle against the oracle's (1e-4, the bound of the V-cycle's
    stage test), and bitwise against the general kernel, which takes
    right-hand sides that do not start on a 32-byte boundary."""
    from oracle import mg
    sp = workloads.spec(workloads.SPHERICAL, nr, nt, 8, workloads.UNIFORM, 1.0, 2.0,
                        *(() if whole else (0.3 * np.pi, 0.65 * np.pi)))
    s = ps.Solver.from_spec(sp, precision=ps.MIXED, use_graph=False,
                            coarsest_size=ps.COARSEST_LARGE if large else ps.COARSEST_SMALL)
    s.set_schedule(nu1, nu2, n_sor)
    lev = s.fused_level()
    shape = (s.n_modes, nt >> lev, nr >> lev)
    f = torch.from_numpy(_planes(shape, nr + nt)).to(torch.complex64).cuda()
    got = s.stage_vcycle(f)
    room = torch.zeros(f.numel() + 2, dtype=f.dtype, device="cuda")
    shifted = room[2:].view(shape)
    shifted.copy_(f)
    assert f.data_ptr() % 32 == 0 and shifted.data_ptr() % 32 == 16
    assert torch.equal(got, s.stage_vcycle(shifted))
    H = mg.Hierarchy(oracle_plane(sp), nu1=nu1, nu2=nu2, n_sor=n_sor,
                     **(dict(min_cells=32, max_coarse=2048) if large else {}))
    for m in (0, s.n_modes - 1):
        u = np.zeros((shape[2] + 2, shape[1] + 2), complex)
        H.vcycle(lev, m, u, f[m].cpu().numpy().T.astype(complex))
        ref = u[1:-1, 1:-1].T
        assert np.abs(got[m].cpu().numpy() - ref).max() <= 1e-4 * np.abs(ref).max()
    s.close()


# n_r, n_tz, n_phi: work items of 256 cells per launch of the residual, and its
# arrivals: 3 (one per plane), 10, 160 (one counter for all), 288 and 384 (a
# counter per plane until planes retire), and 16 planes and more
RETIRE_GRIDS = [(8, 8, 4), (16, 32, 8), (128, 64, 8), (128, 64, 16), (256, 128, 4), (32, 32, 64)]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nr,nt,n_phi", RETIRE_GRIDS)
def test_planes_retire_by_either_arrival_count(ps, nr, nt, n_phi, precision):
    """A plane of zeros retires at once, every other one at the direct solution
    (1e-9 at a relative residual of 1e-11), and a plane that is not finite
    is reported without touching the others."""
    import scipy.sparse.linalg as spla

    from oracle import operator
    sp = workloads.spec(workloads.SPHERICAL, nr, nt, n_phi, workloads.LOG, 1.0, 8.0)
    s = ps.Solver.from_spec(sp, precision=precision, use_graph=False)
    f = _planes((s.n_modes, nt, nr), nr + nt + n_phi)
    f[1] = 0.0
    u, cyc, rc = s.stage_mg_solve(torch.from_numpy(f).cuda(), tol=1e-11)
    assert rc == ps.OK and cyc[1] == 0 and min(cyc[0], cyc[-1]) > 0
    u = u.cpu().numpy()
    assert not u[1].any()
    p = oracle_plane(sp)
    for m in (0, s.n_modes - 1):
        A = operator.matrix(p, m).tocsc()
        b = f[m].T
        x = spla.spsolve(A, operator.to_vec(b.real)) + 1j * spla.spsolve(A, operator.to_vec(b.imag))
        ref = operator.from_vec(x, nr, nt).T
        assert np.abs(u[m] - ref).max() <= 1e-9 * np.abs(ref).max()
    f[1] = np.nan
    v, cyc2, rc = s.stage_mg_solve(torch.from_numpy(f).cuda(), tol=1e-11)
    assert rc == ps.ERR_NONFINITE
    assert cyc2[0] == cyc[0] and np.array_equal(v[0].cpu().numpy(), u[0])
    s.close()


# n_r, n_tz, n_phi: enough planes for whole tiles at first (a warp relaxes
# several columns in turn), narrower ones as they retire; lines of one, two and
# four cells a lane
FP64_MANY = [(32, 32, 256), (64, 32, 128), (32, 64, 128), (128, 64, 128)]


@pytest.mark.parametrize("nr,nt,n_phi", FP64_MANY)
def test_fp64_solves_with_stored_inverse_diagonals(ps, nr, nt, n_phi):
    """Many planes on the FP64 line passes: the direct solution to 1e-10 at a
    relative residual of 1e-12, and the oracle's cycle counts."""
    import scipy.sparse.linalg as spla

    from oracle import mg, operator
    sp = workloads.spec(workloads.SPHERICAL, nr, nt, n_phi, workloads.LOG, 1.0, 8.0)
    s = ps.Solver.from_spec(sp, precision=ps.FP64, use_graph=False)
    f = _planes((s.n_modes, nt, nr), nr + nt)
    u, cyc, rc = s.stage_mg_solve(torch.from_numpy(f).cuda(), tol=1e-12)
    assert rc == ps.OK
    p = oracle_plane(sp)
    H = mg.Hierarchy(p)
    for m in (0, 1, s.n_modes - 1):
        A = operator.matrix(p, m).tocsc()
        b = f[m].T
        x = spla.spsolve(A, operator.to_vec(b.real)) + 1j * spla.spsolve(A, operator.to_vec(b.imag))
        ref = operator.from_vec(x, nr, nt).T
        assert np.abs(u[m].cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
        assert abs(cyc[m] - H.solve(m, b, 1e-12)[1]) <= 1
    s.close()


# finest level, schedule, whether windows take its planes: the halo of one smoothing
# cycle (4 n_sor + 1 cells, one more for the restriction) leaves a 64-cell window 16
# cells of its own, and no level above the fused ones has lines of less than 32 cells
# (512 x 32: 256 x 16)
WINDOWS = [(256, 128, (2, 1, 2, 3, 1), True), (256, 128, (2, 2, 3, 0, 0), True), (256, 128, (2, 2, 5, 0, 0), True),
           (512, 256, (2, 2, 2, 0, 0), True), (512, 32, (2, 2, 2, 0, 0), False), (256, 128, (2, 2, 6, 0, 0), False)]


@pytest.mark.parametrize("nr,nt,sched,windows", WINDOWS)
def test_window_passes_run_where_they_fit_also_in_a_captured_solve(ps, nr, nt, sched, windows):
    """The handle says whether a solve's last planes take the window passes, and a
    captured solve (two loops with a hand-over, several iterations per pass) gives
    the bits and cycle counts of the eager one."""
    from gpu_helpers import clumps
    sp = workloads.spec(workloads.CYLINDRICAL, nr, nt, 64, workloads.UNIFORM, 1.0, 3.0, 0.0, 2.0 * nt / nr)
    rho = torch.from_numpy(clumps(sp, 3)).cuda()
    out = []
    for graph in (False, True):
        s = ps.Solver.from_spec(sp, precision=ps.MIXED, use_graph=graph)
        s.set_schedule(*sched[:3], nu_pre_fused=sched[3], nu_post_fused=sched[4])
        few = s.loops()["few_planes"]
        assert (0 < few < s.n_modes) if windows else few == 0
        phi, rc = s.solve(rho, tol=1e-8)
        assert rc == ps.OK
        st = s.stats()
        out.append((phi.clone(), st["cycles_psi"], st["cycles_phi"]))
        assert sum(1 for c in st["cycles_phi"] if c == max(st["cycles_phi"])) < s.n_modes
        s.close()
    assert torch.equal(out[0][0], out[1][0]) and out[0][1:] == out[1][1:]
