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
