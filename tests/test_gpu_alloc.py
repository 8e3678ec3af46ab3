"""Creating a handle on an allocator that runs out: the create reports it, or
goes without the buffers that a solve can do without."""
import pytest

from paper_2606_17636_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ps():
    import paper_2606_17636_gb300 as m
    m.lib()
    _create.base = m._TorchAllocator
    return m


def _create(ps, monkeypatch, refuse, spec, **kw):
    """A solver (or None when the create fails for want of memory) whose
    allocator refuses where refuse(index of the request, bytes, bytes held)."""
    class Allocator(_create.base):
        def __init__(self):
            super().__init__()
            self.sizes, self.peak = [], 0

        def _alloc(self, nbytes, user):
            held = sum(t.numel() for t in self.live.values())
            self.sizes.append(nbytes)
            if refuse(len(self.sizes) - 1, nbytes, held):
                return None
            self.peak = max(self.peak, held + nbytes)
            return super()._alloc(nbytes, user)

    monkeypatch.setattr(ps, "_TorchAllocator", Allocator)
    try:
        return ps.Solver.from_spec(spec, **kw)
    except ps.PSolveError as e:
        assert e.code == ps.ERR_NOMEM
        return None


SPECS = {
    # levels above the shared-memory ones, auxiliary windows
    "wide": (dict(precision=1), workloads.spec(workloads.CYLINDRICAL, 256, 32, 4, workloads.UNIFORM, 1.0, 3.0, 0.0, 0.25)),
    "fp64": (dict(precision=0), workloads.spec(workloads.SPHERICAL, 32, 32, 4, workloads.UNIFORM, 1.0, 2.0)),
    # the extended-domain tables, whose set-up solves on planes of its own
    "extended": (dict(precision=1), workloads.spec(workloads.SPHERICAL, 32, 32, 4, workloads.LOG, 0.1, 10.0)),
}


@pytest.mark.parametrize("key", list(SPECS))
def test_a_refused_request_is_reported_or_done_without(ps, monkeypatch, key):
    """Each request in turn is refused and the later ones granted: no kernel may
    run on a missing buffer."""
    kw, sp = SPECS[key]
    rho = torch.rand((sp["n_r"], sp["n_tz"], sp["n_phi"]), dtype=torch.float64, device="cuda")
    s = _create(ps, monkeypatch, lambda k, n, held: False, sp, **kw)
    ref = s.solve(rho, tol=1e-9)[0].clone()
    requests = len(s._alloc.sizes)
    s.close()
    without = 0
    for q in range(requests):
        s = _create(ps, monkeypatch, lambda k, n, held: k == q, sp, **kw)
        torch.cuda.synchronize()
        if s is not None:
            without += 1
            assert torch.equal(s.solve(rho, tol=1e-9)[0], ref)
            s.close()
    assert without < requests // 4


@pytest.mark.parametrize("key,optional", [("wide", 1), ("fp64", 2)])
def test_a_create_that_fits_without_the_optional_buffers(ps, monkeypatch, key, optional):
    """The window passes' buffer (mixed) and the stored inverse diagonals (FP64)
    are asked for last: an allocator with room for everything else, and no more,
    gives a working handle with the same result."""
    kw, sp = SPECS[key]
    rho = torch.rand((sp["n_r"], sp["n_tz"], sp["n_phi"]), dtype=torch.float64, device="cuda")
    s = _create(ps, monkeypatch, lambda k, n, held: False, sp, **kw)
    requests = len(s._alloc.sizes)
    ref = s.solve(rho, tol=1e-9)[0].clone()
    if key == "wide":
        assert s.loops()["few_planes"] > 0
    s.close()
    s = _create(ps, monkeypatch, lambda k, n, held: k >= requests - optional, sp, **kw)
    assert s is not None and len(s._alloc.sizes) in range(requests - optional + 1, requests + 1)
    room = s._alloc.peak
    if key == "wide":
        assert s.loops()["few_planes"] == 0
    assert torch.equal(s.solve(rho, tol=1e-9)[0], ref)
    s.close()
    s = _create(ps, monkeypatch, lambda k, n, held: held + n > room, sp, **kw)
    assert s is not None
    assert torch.equal(s.solve(rho, tol=1e-9)[0], ref)
    s.close()


@pytest.mark.parametrize("nr,nt,arrays", [(64, 32, 2), (512, 32, 1), (32, 512, 1)])
def test_fp64_diagonals_only_where_lines_read_them(ps, monkeypatch, nr, nt, arrays):
    """The FP64 passes read stored inverse diagonals along lines of up to 256
    cells: the finest level asks for one array per such direction (besides the
    residual's diagonal of the same size)."""
    sp = workloads.spec(workloads.CYLINDRICAL, nr, nt, 8, workloads.UNIFORM, 1.0, 3.0, 0.0, 2.0 * nt / nr)
    s = _create(ps, monkeypatch, lambda k, n, held: False, sp, precision=0)
    want = 8 * s.n_modes * nr * nt
    tail = s._alloc.sizes[-12:]
    assert tail.count(want) == arrays
    s.close()
