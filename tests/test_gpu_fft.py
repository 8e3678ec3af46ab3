"""The azimuthal transforms' block fixed point: error against extended precision
for rows of every kind of scale, special rows, every length and ragged rows."""
import numpy as np
import pytest

from paper_2606_17636_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTHS = [4, 8, 16, 32, 64, 128, 256, 512, 1024]


@pytest.fixture(scope="module")
def ps():
    import paper_2606_17636_gb300 as m
    m.lib()
    return m


def _solver(ps, n_phi, nr=32, nt=16):
    sp = workloads.spec(workloads.CYLINDRICAL, nr, nt, n_phi, workloads.UNIFORM, 1.0, 2.0)
    return ps.Solver.from_spec(sp, precision=ps.FP64, use_graph=False)


def _rows(rng, shape):
    """Rows of different kinds side by side: noise, flat, one spike, a smooth
    bump, values over twenty decades, rows 200 decades apart."""
    n = shape[-1]
    x = rng.standard_normal(shape)
    ph = (np.arange(n) + 0.5) * 2 * np.pi / n
    x[1::6] = 1.0 + 0.01 * x[1::6]
    x[2::6] *= 1e-3
    x[2::6, :, n // 2] += 1.0
    x[3::6] = np.exp(-20.0 * (1.0 - np.cos(ph - rng.uniform(0, 6, x[3::6].shape[:2])[..., None])))
    x[4::6] *= 10.0 ** rng.uniform(-20, 0, x[4::6].shape)
    x[5::6] *= 10.0 ** rng.uniform(-100, 100, x[5::6].shape[:2])[..., None]
    return x


def _dft(x, n, sign):
    """Sums in extended precision: the exact angles' cosines and sines."""
    k = np.arange(n)
    idx = np.outer(k, k) % n
    ang = 2 * np.pi * np.arange(n, dtype=np.longdouble) / n if np.finfo(np.longdouble).eps < 1e-18 else None
    if ang is None:
        pytest.skip("no extended precision on this machine")
    pi = np.longdouble("3.14159265358979323846264338327950288")
    ang = 2 * pi * np.arange(n, dtype=np.longdouble) / n
    return x @ np.cos(ang)[idx], sign * (x @ np.sin(ang)[idx])


@pytest.mark.parametrize("n", LENGTHS)
def test_transforms_within_fp64_rounding_of_each_row(ps, n):
    """Relative to a row's 2-norm both transforms stay within the error of an
    FP64 transform of log2 n passes: (1 + log2 n) 2^-53 (one rounding per pass
    and one of the output), each row by itself though rows share a transform."""
    rng = np.random.default_rng(n)
    s = _solver(ps, n)
    x = _rows(rng, (32, 16, n))
    bound = (1 + np.log2(n)) * 2.0 ** -53
    f = s.stage_forward(torch.from_numpy(x).cuda()).cpu().numpy().transpose(2, 1, 0)
    rows = rng.choice(32 * 16, 48, replace=False)
    xr = x.reshape(-1, n)[rows].astype(np.longdouble)
    c, si = _dft(xr, n, -1)
    scale = np.longdouble(4 * np.pi * 1.0 / n)
    ref = (c + 1j * si)[:, : n // 2 + 1] * scale
    got = f.reshape(-1, n // 2 + 1)[rows]
    err = np.sqrt((np.abs(got - ref) ** 2).sum(1) / (np.abs(ref) ** 2).sum(1))
    assert err.max() <= bound, (err.max(), bound)
    # inverse: the real signal of random half spectra of the same kinds
    h = _rows(rng, (32, 16, n))[..., : n // 2 + 1] + 1j * rng.standard_normal((32, 16, n // 2 + 1))
    g = s.stage_inverse(torch.from_numpy(np.ascontiguousarray(h.transpose(2, 1, 0))).cuda()).cpu().numpy()
    hr = h.reshape(-1, n // 2 + 1)[rows].astype(np.clongdouble)
    hr[:, 0] = hr[:, 0].real
    hr[:, -1] = hr[:, -1].real
    full = np.concatenate([hr, np.conj(hr[:, 1:-1][:, ::-1])], axis=1)
    ca, sa = _dft(full.real, n, 1)
    cb, sb = _dft(full.imag, n, 1)
    ref = ca - sb
    got = g.reshape(-1, n)[rows]
    err = np.sqrt(((got - ref) ** 2).sum(1) / (ref ** 2).sum(1))
    assert err.max() <= bound, (err.max(), bound)
    s.close()


@pytest.mark.parametrize("n", [8, 32, 256, 512])
def test_special_rows(ps, n):
    """Zero rows transform to exact zeros beside other rows; a power of two
    scales the result exactly, down to subnormal values' neighbourhood; an
    infinity or NaN makes its row pair NaN and leaves the other rows as they were."""
    rng = np.random.default_rng(7)
    s = _solver(ps, n)
    x = rng.standard_normal((32, 16, n))
    x[3], x[10], x[11] = 0.0, 0.0, 0.0
    f = s.stage_forward(torch.from_numpy(x).cuda())
    assert torch.count_nonzero(f[:, :, 3]) == 0 and torch.count_nonzero(f[:, :, 10:12]) == 0
    for e in (-900, 600):
        fe = s.stage_forward(torch.from_numpy(np.ldexp(x, e)).cuda())
        assert np.array_equal(np.ldexp(f.cpu().numpy().view(np.float64), e), fe.cpu().numpy().view(np.float64))
    back = s.stage_inverse(f)
    assert torch.count_nonzero(back[3]) == 0 and torch.count_nonzero(back[10:12]) == 0
    assert np.abs(back.cpu().numpy() - 4 * np.pi * x).max() <= 1e-13 * np.abs(x).max() * 4 * np.pi
    for bad in (np.inf, np.nan):
        y = x.copy()
        y[6, 5, n // 2] = bad
        fy = s.stage_forward(torch.from_numpy(y).cuda())
        assert torch.isnan(fy[:, 5, 6:8].real).all()
        same = torch.ones_like(f, dtype=torch.bool)
        same[:, 5, 6:8] = False
        assert torch.equal(fy[same], f[same])
        by = s.stage_inverse(fy)
        assert torch.isnan(by[6:8, 5]).all() and torch.equal(by[8:], back[8:])
    tiny = s.stage_forward(torch.full((32, 16, n), 2.0 ** -1070, dtype=torch.float64, device="cuda"))
    assert abs(tiny[0, 0, 0].real.item() - 4 * np.pi * 2.0 ** -1070) <= 2.0 ** -1074
    s.close()


@pytest.mark.parametrize("n,rows", [(4, 1), (16, 5), (32, 31), (128, 17), (256, 1), (256, 33), (512, 37), (1024, 9)])
def test_ragged_slabs_equal_the_whole_grid(ps, n, rows):
    """A slab of any number of rows gives the rows of the whole transform
    (pairs counted from its first row)."""
    s = _solver(ps, n, nr=64)
    x = torch.from_numpy(np.random.default_rng(rows).standard_normal((64, 16, n))).cuda()
    f = s.stage_forward(x)
    part = s.stage_forward_rows(x[:rows].contiguous())
    even = rows - rows % 2
    assert torch.equal(part[:, :, :even], f[:, :, :even])
    assert torch.allclose(part, f[:, :, :rows], rtol=0, atol=1e-14)
    g = s.stage_inverse(f)
    gp = s.stage_inverse_rows(f[:, :, :rows].contiguous())
    assert torch.equal(gp[:even], g[:even]) and torch.allclose(gp, g[:rows], rtol=0, atol=1e-12)
    s.close()


@pytest.mark.parametrize("n", LENGTHS)
def test_exact_zeros_of_periodic_rows(ps, n):
    """Differences of equal values are zero and stay zero through the twiddles:
    rows constant along phi have no modes above m = 0, rows of period n / p only
    every p-th one; the inverse of such spectra has rows of that period."""
    rng = np.random.default_rng(n)
    s = _solver(ps, n)
    for p in (2, 4, n):
        if p > n // 2 and p != n:
            continue
        x = np.tile(rng.standard_normal((32, 16, n // p)) + 3.0, p)
        f = s.stage_forward(torch.from_numpy(x).cuda())
        others = torch.arange(n // 2 + 1, device="cuda") % p != 0
        assert torch.count_nonzero(f[others]) == 0
        ref = np.fft.rfft(x, axis=2).transpose(2, 1, 0) * (4 * np.pi / n)
        assert np.abs(f.cpu().numpy() - ref).max() <= 1e-14 * np.abs(ref).max()
        g = s.stage_inverse(f)
        assert torch.equal(g, g[:, :, : n // p].repeat(1, 1, p))
    s.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("graph", [False, True])
def test_modes_of_an_axisymmetric_density_retire_at_once(ps, precision, graph):
    """A density without phi dependence: every m > 0 is an exact zero and takes no
    cycle in either solve, and the potential does not depend on phi."""
    sp = workloads.spec(workloads.SPHERICAL, 64, 32, 32, workloads.LOG, 0.1, 10.0)
    s = ps.Solver.from_spec(sp, precision=precision, use_graph=graph)
    rho = torch.rand((64, 32, 1), dtype=torch.float64, device="cuda").expand(64, 32, 32).contiguous()
    phi, rc = s.solve(rho, tol=1e-9)
    assert rc == ps.OK
    st = s.stats()
    assert st["cycles_psi"][0] > 0 and st["cycles_phi"][0] > 0
    assert not any(st["cycles_psi"][1:]) and not any(st["cycles_phi"][1:])
    assert torch.equal(phi, phi[:, :, :1].expand_as(phi))
    s.close()


def _rms(got, ref):
    return float(np.sqrt(((np.abs(got - ref) ** 2).sum(1) / (np.abs(ref) ** 2).sum(1)).mean()))


def _rounded(ref):
    out = np.empty_like(ref)
    if np.iscomplexobj(ref):
        out.real, out.imag = ref.real.astype(np.float64), ref.imag.astype(np.float64)
    else:
        out[...] = ref.astype(np.float64)
    return out


@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024])
@pytest.mark.parametrize("kind", ["cosine", "constant", "noise", "spike"])
def test_flat_rows_and_spectra_keep_53_bits(ps, n, kind):
    """Rows nearly constant along phi (forward) and spectra of equal magnitudes
    (inverse, a spike): the rounding of the exact result to FP64, and per output
    two units of 2^-60 of the row's sum of magnitudes.  That sum is the norm of a
    flat row's spectrum, and up to sqrt(2) times that of a spike, so relative to
    the norm two units of sqrt(n) 2^-60, times sqrt(2) for the spike."""
    rng = np.random.default_rng(n)
    s = _solver(ps, n)
    ph = (np.arange(n) + 0.5) * 2 * np.pi / n
    shape = (32, 16, 1)
    rows = rng.choice(32 * 16, 64, replace=False)
    units = 2 * np.sqrt(n) * 2.0 ** -60
    if kind == "spike":
        k = np.exp(-2j * np.pi * np.arange(n // 2 + 1) * rng.integers(0, n, shape) / n) * rng.uniform(1, 2, shape)
        g = s.stage_inverse(torch.from_numpy(np.ascontiguousarray(k.transpose(2, 1, 0))).cuda()).cpu().numpy()
        h = k.reshape(-1, n // 2 + 1)[rows].astype(np.clongdouble)
        h[:, 0], h[:, -1] = h[:, 0].real, h[:, -1].real
        full = np.concatenate([h, np.conj(h[:, 1:-1][:, ::-1])], axis=1)
        ref = _dft(full.real, n, 1)[0] - _dft(full.imag, n, 1)[1]
        got = g.reshape(-1, n)[rows]
        units *= np.sqrt(2.0)
    else:
        c = rng.uniform(1, 2, shape)
        x = {"cosine": 1.0 + 0.01 * np.cos(ph * rng.integers(1, 4, shape) + rng.uniform(0, 6, shape)),
             "constant": c * np.ones(n), "noise": c * (1.0 + 0.01 * rng.standard_normal((32, 16, n)))}[kind]
        f = s.stage_forward(torch.from_numpy(x).cuda()).cpu().numpy().transpose(2, 1, 0)
        co, si = _dft(x.reshape(-1, n)[rows].astype(np.longdouble), n, -1)
        ref = (co + 1j * si)[:, : n // 2 + 1] * np.longdouble(4 * np.pi * 1.0 / n)
        got = f.reshape(-1, n // 2 + 1)[rows]
    bound = np.hypot(_rms(_rounded(ref), ref), units)
    assert _rms(got, ref) <= bound, (_rms(got, ref), bound)
    s.close()
