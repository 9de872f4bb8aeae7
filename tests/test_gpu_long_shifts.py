"""Solves whose sources are carried beyond the splat's reach: these go through
the overflow list and are added after the splat has stored the residual D - P
and its split over the lines.  Against the FP64 oracle.

Tolerance (relative L2, fixed beforehand): 2e-5, that of solves of three
iterations or fewer; the residual norm rho 1e-5 relative (a sum of squares
of values that are off by a few 6e-8)."""
import numpy as np
import pytest

from paper_2601_22793_gb300 import phantoms as ph

pytestmark = pytest.mark.gpu

PIXEL, L = 20e-6, 30.0


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_22793_gb300 import build
    build.build()
    from paper_2601_22793_gb300 import epr
    epr.load()
    return torch


@pytest.fixture(scope="module")
def E():
    from paper_2601_22793_gb300 import epr
    return epr


def rel(a, b):
    a = np.asarray(a, np.float64)
    b = np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def cuda(torch, a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def spec(n_lines, seed=5):
    return ph.spectrum(n_lines, 60.0, 160.0, 95.0, 30.0, ph.BONE[0], ph.BONE[1], 80.0, seed)


def phantom(ny, nx, seed=11):
    hi = min(20.0, min(ny, nx) / 5.0)
    ells = ph.random_ellipsoids(ny, nx, 8, 0.4 * hi, hi, margin=4.0, seed=seed)
    return ph.project_ellipsoids(ells, ny, nx, PIXEL).astype(np.float32)


# a spectrum that varies across the columns: one line has no split (and none of
# the maps that a split needs); row lengths with and without compile-time kernels
@pytest.mark.parametrize("lines,ny,nx", [(1, 96, 144), (1, 48, 1024), (1, 144, 96), (2, 96, 144), (4, 48, 1024)])
@pytest.mark.parametrize("fixed", [False, True])
def test_xspec_solve_with_long_shifts(torch, E, oracle, lines, ny, nx, fixed):
    Es, d, b, w = spec(lines)
    g = np.random.default_rng(17)
    tab = (np.linspace(-3.0, nx + 2.0, 5), w[:, None] * g.uniform(0.7, 1.3, size=(lines, 5)),
           d[:, None] * g.uniform(0.8, 1.2, size=(lines, 5)), b[:, None] * g.uniform(0.8, 1.2, size=(lines, 5)))
    xs = oracle.XSpec(Es, *tab, L, PIXEL, nx)
    T0 = phantom(ny, nx) * 2.0
    D = ph.poisson(oracle.forward_x(xs, phantom(ny, nx, 12).astype(np.float64)), 1e4, 3).astype(np.float32)
    Tref, info = oracle.solve_x(xs, D.astype(np.float64), T0=T0, n_iter=2, omega=0.4)
    with E.Plan(nx, ny, PIXEL, L, Es, d, b, w, deterministic=fixed, max_shift_px=1) as p:
        E.epr_plan_set_xspec(p.handle, *tab)
        T, Dd = cuda(torch, np.stack([T0, T0])), cuda(torch, np.stack([D, D]))
        got = E.epr_solve_nonlocal(p.handle, Dd, T, batch=2, n_iter=2, omega=0.4, init=1)
        assert got["overflow_sources"] > 0
        for k in range(2):
            assert rel(T[k].cpu().numpy(), Tref) <= 2e-5
            assert np.allclose(got["rho_hist"][k], info["rho"], rtol=1e-5)


# the size groups of a batch run on streams of their own that do not wait for
# the default stream: the marks of the first long-shift pass after an
# allocation must not meet the clearing of the workspace
def test_first_solve_after_an_allocation(torch, E, oracle):
    Es, d, b, w = spec(4)
    ln = oracle.Lines(Es, d, b, w, L, PIXEL)
    shapes = [(256, 384), (384, 256), (128, 128), (256, 384)]
    T0s = [phantom(ny, nx, 30 + i) * 2.0 for i, (ny, nx) in enumerate(shapes)]
    Ds = [ph.poisson(oracle.forward(ln, phantom(ny, nx, 40 + i)), 1e4, i).astype(np.float32)
          for i, (ny, nx) in enumerate(shapes)]
    refs = [oracle.solve(ln, D.astype(np.float64), T0=T0, n_iter=1, omega=0.4)[0] for D, T0 in zip(Ds, T0s)]
    Dd = [cuda(torch, D) for D in Ds]
    for _ in range(4):
        bh = E.epr_batch_create(PIXEL, L, Es, d, b, w, max_shift_px=1)
        try:
            Ts = [cuda(torch, T0) for T0 in T0s]
            info = E.epr_solve_nonlocal_batched(bh, Dd, Ts, n_iter=1, omega=0.4, init=1)
            assert info["overflow_sources"] > 0
            for T, ref in zip(Ts, refs):
                assert rel(T.cpu().numpy(), ref) <= 2e-5
        finally:
            E.epr_batch_destroy(bh)


# data far above the prediction (hot pixels, dark caustics): the split of a
# pixel that long shifts reach needs the prediction itself, whose digits D - P
# does not keep.  Absorption strong enough for predictions down to 1e-2, and
# pixels that only long shifts reach.
@pytest.mark.parametrize("lines", [2, 4, 5, 8])
@pytest.mark.parametrize("level", [1.0, 1e3, 1e5, 1e7])
def test_split_keeps_the_prediction(torch, E, oracle, lines, level):
    Es, d, b, w = spec(lines)
    b = b * 8.0
    ln = oracle.Lines(Es, d, b, w, L, PIXEL)
    T0 = phantom(96, 144) * 2.0
    D = (level * ph.rng(4).uniform(0.9, 1.1, size=(96, 144))).astype(np.float32)
    Tref, info = oracle.solve(ln, D.astype(np.float64), T0=T0, n_iter=1, omega=0.4)
    with E.Plan(144, 96, PIXEL, L, Es, d, b, w, max_shift_px=1) as p:
        T = cuda(torch, T0)
        got = E.epr_solve_nonlocal(p.handle, cuda(torch, D), T, n_iter=1, omega=0.4, init=1)
        assert got["overflow_sources"] > 0
        err = rel(T.cpu().numpy(), Tref)
        print("lines %d level %g: %.2e" % (lines, level, err))
        assert err <= 2e-5
        assert abs(got["rho"][0] - info["rho"][0]) <= 1e-5 * info["rho"][0]
