"""The rules that choose a kernel by size, type and option, at the sizes where
they can go wrong: every row and column length with compile-time kernels, both
block shapes of a row pass, the splat's tile, reach and accumulator choices,
the strips of the stencil and gradient kernels, the split's line counts, and
maps that overlap.

Tolerances (relative L2, fixed beforehand): one preconditioner application is
four transforms of at most five stages, each with about eight roundings of
6e-8: 4 x 5 x 8 x 6e-8 = 1e-5.  The forward models are a few products, an
exponential and four weights per contribution: 2e-6.  Solves of three
iterations: 2e-5.  Gradients: 1e-5."""
import numpy as np
import pytest

from paper_2601_22793_gb300 import phantoms as ph

pytestmark = pytest.mark.gpu

LENGTHS = [128, 144, 192, 216, 256, 288, 384, 432, 512, 576, 648, 768, 864, 1024, 1152, 1296, 1536,
           1728, 1944, 2048, 2304, 2592, 3072, 3456, 3888, 4096]


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


def host(t):
    return t.detach().cpu().numpy().astype(np.float64)


def spec(n_lines, seed=5):
    return ph.spectrum(n_lines, 60.0, 160.0, 95.0, 30.0, ph.BONE[0], ph.BONE[1], 80.0, seed)


def phantom(ny, nx, pixel=20e-6, n=8, seed=11):
    hi = min(20.0, min(ny, nx) / 5.0)
    ells = ph.random_ellipsoids(ny, nx, n, 0.4 * hi, hi, margin=4.0, seed=seed)
    return ph.project_ellipsoids(ells, ny, nx, pixel).astype(np.float32)


PIXEL, L = 20e-6, 30.0


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("axis", ["rows", "columns"])
def test_precondition_every_length(torch, E, n, axis):
    nx, ny = (n, 48) if axis == "rows" else (48, n)
    g = ph.rng(n).normal(size=(3, ny, nx)).astype(np.float32)
    mu = 2.0 * (2.0 * np.pi / (1.2398419843320026e-6 / 80e3)) * ph.BONE[1]
    fy, fx = np.fft.fftfreq(ny, PIXEL)[:, None], np.fft.rfftfreq(nx, PIXEL)[None, :]
    H = mu / (mu + L * ph.BONE[0] * 4.0 * np.pi ** 2 * (fx * fx + fy * fy))
    ref = np.fft.irfft2(np.fft.rfft2(g.astype(np.float64)) * H, s=(ny, nx))
    for batch in (1, 3):
        with E.Plan(nx, ny, PIXEL, L, [80.0], [ph.BONE[0]], [ph.BONE[1]]) as p:
            x = cuda(torch, g[:batch])
            E.epr_precondition(p.handle, x, batch=batch)
            assert rel(host(x), ref[:batch]) <= 1e-5
            y = cuda(torch, g[:batch])
            E.epr_precondition_noalloc(y, nx, ny, PIXEL, L, 80.0, ph.BONE[0], ph.BONE[1], batch=batch)
            assert rel(host(y), ref[:batch]) <= 1e-5


# few blocks (one row pair each, narrow column tiles) and many of each length
@pytest.mark.parametrize("nx,ny,lines", [(128, 48, 1), (144, 96, 2), (216, 24, 1), (256, 64, 1), (288, 72, 3),
                                         (512, 32, 2), (512, 512, 1), (648, 48, 1), (1024, 16, 1), (72, 1024, 2), (1296, 24, 1),
                                         (2048, 16, 1), (2304, 16, 2), (3456, 24, 1), (3888, 16, 2)])
def test_solve_few_and_many_blocks(torch, E, oracle, nx, ny, lines):
    Es, d, b, w = spec(lines)
    ln = oracle.Lines(Es, d, b, w, L, PIXEL)
    tau = phantom(ny, nx)
    D = ph.poisson(oracle.forward(ln, tau), 1e4, 3).astype(np.float32)
    Tref, info = oracle.solve(ln, D.astype(np.float64), n_iter=3, omega=0.4)
    rp = 1   # row pairs of a large block, and the batch that fills the GPU with them
    while 2 * rp * nx <= 1152 and nx <= 512 and (ny // 2) % (2 * rp) == 0:
        rp *= 2
    many = 608 // (ny // (2 * rp)) + 1 if rp > 1 else 3
    for batch in (1, many):
        with E.Plan(nx, ny, PIXEL, L, Es, d, b, w) as p:
            Dd = cuda(torch, np.repeat(D[None], batch, 0))
            T = torch.empty_like(Dd)
            got = E.epr_solve_nonlocal(p.handle, Dd, T, batch=batch, n_iter=3, omega=0.4)
            for k in {0, batch // 2, batch - 1}:
                assert rel(host(T[k]), Tref) <= 2e-5
                assert np.allclose(got["rho_hist"][k], info["rho"], rtol=1e-4)
                assert np.allclose(got["kappa_hist"][k], info["kappa"], rtol=1e-3)


# the float accumulators resolve 2^-24 up to reach 4 and 2^-18 at reach 32 (the
# sums must fit in 32 bits), which 2e-6 does not cover: long reaches in fixed
# point only, where 21 is the longest with two 32-bit planes
@pytest.mark.parametrize("reach,fixed", [(1, False), (3, False), (4, False), (5, False), (1, True), (4, True),
                                         (5, True), (21, True), (22, True), (32, True)])
@pytest.mark.parametrize("nx,ny,lines", [(16, 16, 1), (72, 96, 1), (72, 96, 3), (128, 72, 4), (96, 72, 8)])
def test_forward_reach_and_accumulators(torch, E, oracle, nx, ny, lines, reach, fixed):
    Es, d, b, w = spec(lines)
    ln = oracle.Lines(Es, d, b, w, L, PIXEL)
    tau = phantom(ny, nx) * 2.0   # shifts beyond the short reaches
    tau[ny // 2, nx // 3] = -0.012    # a pixel far brighter than the accumulators' bound
    P, Ps, _ = oracle.forward(ln, tau, per_line=True)
    with E.Plan(nx, ny, PIXEL, L, Es, d, b, w, max_shift_px=reach, deterministic=fixed) as p:
        T = cuda(torch, tau)
        Pd = torch.empty_like(T)
        Psd = torch.empty(lines, ny, nx, device="cuda")
        E.epr_forward(p.handle, T, Pd, Psd)
        assert rel(host(Pd), P) <= 2e-6
        assert rel(host(Psd), Ps) <= 2e-6
        E.epr_forward(p.handle, T, Pd.zero_())   # without the lines' predictions
        assert rel(host(Pd), P) <= 2e-6


def test_forward_not_a_number_stays_local(torch, E, oracle):
    """A NaN thickness reaches the pixels its own source and the sources whose
    gradient it enters are carried to, no more."""
    tau = phantom(96, 96)
    ln = oracle.Lines([80.0], [ph.BONE[0]], [ph.BONE[1]], [1.0], L, PIXEL)
    P = oracle.forward(ln, tau)
    bad = tau.copy()
    bad[40, 50] = np.nan
    with E.Plan(96, 96, PIXEL, L, [80.0], [ph.BONE[0]], [ph.BONE[1]]) as p:
        Pd = torch.empty(96, 96, device="cuda")
        E.epr_forward(p.handle, cuda(torch, bad), Pd)
        got = host(Pd)
    far = np.ones_like(tau, bool)
    far[28:54, 38:64] = False
    assert rel(got[far], P[far]) <= 2e-6


def test_forward_of_overlapping_maps(torch, E):
    Es, d, b, w = spec(2)
    tau = phantom(96, 144)
    with E.Plan(144, 96, PIXEL, L, Es, d, b, w) as p:
        T = cuda(torch, tau)
        P, Ps = torch.empty_like(T), torch.empty(2, 96, 144, device="cuda")
        E.epr_forward(p.handle, T, P, Ps)
        Q, X = Ps.clone(), T.clone()
        E.epr_forward(p.handle, X, X, Q)            # in place
        assert torch.equal(X, P) and torch.equal(Q, Ps)
        buf = torch.empty(3, 96, 144, device="cuda")
        buf[1] = T
        E.epr_forward(p.handle, buf[1], P, buf[:2])   # the thickness inside P_s
        assert torch.equal(buf[:2], Ps)


# one line: 304 and 608 blocks are the fewest of 32 x 64 and 64 x 64 tiles;
# several: 243.  Sizes on both sides of each line, and a ragged last tile.
@pytest.mark.parametrize("nx,ny,batch,lines,fixed", [(1024, 576, 2, 1, False), (1152, 1152, 1, 1, False),
                                                     (1152, 1152, 2, 1, True), (1536, 1296, 1, 3, False),
                                                     (512, 512, 1, 2, False), (768, 648, 1, 2, True),
                                                     (512, 512, 1, 8, False), (1024, 576, 1, 8, False)])
def test_forward_tile_shapes(torch, E, oracle, nx, ny, batch, lines, fixed):
    Es, d, b, w = spec(lines)
    tau = phantom(ny, nx)
    P, _, _ = oracle.forward(oracle.Lines(Es, d, b, w, L, PIXEL), tau, per_line=True)
    with E.Plan(nx, ny, PIXEL, L, Es, d, b, w, deterministic=fixed) as p:
        T = cuda(torch, np.stack([tau] * batch))
        Pd = torch.empty_like(T)
        E.epr_forward(p.handle, T, Pd, batch=batch)
        assert rel(host(Pd), np.stack([P] * batch)) <= 2e-6


# strips of 26 (28) columns, of 4 rows, then of 15 and of 43 (the last cut short)
@pytest.mark.parametrize("nx,ny", [(16, 16), (24, 48), (32, 24), (64, 32), (96, 72), (144, 16), (288, 96),
                                   (1024, 768), (2048, 1152)])
@pytest.mark.parametrize("lines", [1, 3])
@pytest.mark.parametrize("model", [1, 2, 3])
def test_stencils_at_strip_edges(torch, E, oracle, nx, ny, lines, model):
    Es, d, b, w = spec(lines)
    pixel, dist = (6.5e-6, 0.3) if model < 3 else (PIXEL, L)
    ln = oracle.Lines(Es, d, b, w, dist, pixel)
    tau = phantom(ny, nx, pixel)
    tau[ny // 2:, nx // 2:] += 4e-3   # a step whose |mu dT / 2| exceeds 1/4 at 60 keV
    P, Ps, _ = oracle.forward(ln, tau, model=model, per_line=True)
    with E.Plan(nx, ny, pixel, dist, Es, d, b, w) as p:
        T = cuda(torch, np.stack([tau, tau]))
        Pd, Psd = torch.empty_like(T), torch.empty(2, lines, ny, nx, device="cuda")
        E.epr_forward(p.handle, T, Pd, Psd, batch=2, model=model)
        assert rel(host(Pd), np.stack([P, P])) <= 2e-6
        assert rel(host(Psd), np.stack([Ps, Ps])) <= 2e-6


@pytest.mark.parametrize("lines", [1, 3])
@pytest.mark.parametrize("model", [1, 2, 3])
def test_stencil_solves_split_in_the_kernel(torch, E, oracle, lines, model):
    Es, d, b, w = spec(lines)
    pixel, dist = (6.5e-6, 0.3) if model < 3 else (PIXEL, L)
    ln = oracle.Lines(Es, d, b, w, dist, pixel)
    D = ph.poisson(oracle.forward(ln, phantom(48, 72, pixel)), 1e4, 3).astype(np.float32)
    Tref, _ = oracle.solve(ln, D.astype(np.float64), n_iter=3, omega=0.4, model=model)
    with E.Plan(72, 48, pixel, dist, Es, d, b, w) as p:
        Dd = cuda(torch, D)
        T = torch.empty_like(Dd)
        if model == 3:
            E.epr_solve_nonlocal_wkb1(p.handle, Dd, T, n_iter=3, omega=0.4)
        else:
            E.epr_solve_local(p.handle, Dd, T, order=model, n_iter=3, omega=0.4)
        assert rel(host(T), Tref) <= 2e-5


@pytest.mark.parametrize("lines", [2, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("fixed", [False, True])
def test_split_line_counts(torch, E, oracle, lines, fixed):
    Es, d, b, w = spec(lines)
    ln = oracle.Lines(Es, d, b, w, L, PIXEL)
    D = ph.poisson(oracle.forward(ln, phantom(48, 72)), 1e4, 3).astype(np.float32)
    Tref, _ = oracle.solve(ln, D.astype(np.float64), n_iter=3, omega=0.4)
    with E.Plan(72, 48, PIXEL, L, Es, d, b, w, deterministic=fixed) as p:
        Dd = cuda(torch, D)
        T = torch.empty_like(Dd)
        E.epr_solve_nonlocal(p.handle, Dd, T, n_iter=3, omega=0.4)
        assert rel(host(T), Tref) <= 2e-5


# several lines, or fixed point: pixels that long shifts reach are redone after
# the splat has split their residual (reach 1 sends most sources that way and
# leaves pixels that only they reach)
@pytest.mark.parametrize("lines,fixed", [(1, True), (2, False), (2, True), (4, False), (8, False), (8, True),
                                         (11, False)])
@pytest.mark.parametrize("reach", [1, 4])
def test_split_with_long_shifts(torch, E, oracle, lines, fixed, reach):
    Es, d, b, w = spec(lines)
    ln = oracle.Lines(Es, d, b, w, L, PIXEL)
    T0 = phantom(96, 144) * 2.0
    D = ph.poisson(oracle.forward(ln, phantom(96, 144, seed=12)), 1e4, 3).astype(np.float32)
    D[40:44, 60:70] = oracle.forward(ln, T0)[40:44, 60:70]   # and pixels whose residual vanishes
    Tref, info = oracle.solve(ln, D.astype(np.float64), T0=T0, n_iter=1, omega=0.4)
    with E.Plan(144, 96, PIXEL, L, Es, d, b, w, deterministic=fixed, max_shift_px=reach) as p:
        Dd = cuda(torch, np.stack([D, D]))
        first = None
        for _ in range(2):   # the second solve finds the workspace as the first left it
            T = cuda(torch, np.stack([T0, T0]))
            got = E.epr_solve_nonlocal(p.handle, Dd, T, batch=2, n_iter=1, omega=0.4, init=1)
            assert (got["overflow_sources"] > 0) == (lines > 1 or reach == 1)   # one line: up to 2.4 px
            for k in range(2):
                assert rel(host(T[k]), Tref) <= 2e-5
                assert abs(got["rho"][k] - info["rho"][0]) <= 1e-5 * info["rho"][0]
            if fixed:
                assert first is None or torch.equal(T, first)
                first = T.clone()


@pytest.mark.parametrize("os_", [2, 3, 4, 5])
@pytest.mark.parametrize("lines", [1, 2])
def test_oversampled_split_factors(torch, E, oracle, os_, lines):
    ny, nx = (48, 72) if os_ != 5 else (16, 16)
    if os_ == 5:
        with pytest.raises(E.EprError):   # 5 n is not a supported length
            E.Plan(nx, ny, PIXEL, L, [80.0], [ph.BONE[0]], [ph.BONE[1]], oversample=os_)
        return
    Es, d, b, w = spec(lines)
    fine = phantom(ny * os_, nx * os_, PIXEL / os_)
    P = oracle.forward(oracle.Lines(Es, d, b, w, L, PIXEL / os_), fine)
    D = ph.poisson(oracle.bin_mean(P, os_), 1e4, 3).astype(np.float32)
    Tref, _ = oracle.solve_os(oracle.Lines(Es, d, b, w, L, PIXEL), D.astype(np.float64), os_, n_iter=3, omega=0.4)
    with E.Plan(nx, ny, PIXEL, L, Es, d, b, w, oversample=os_) as p:
        T = torch.empty(ny * os_, nx * os_, device="cuda")
        E.epr_solve_nonlocal(p.handle, cuda(torch, D), T, n_iter=3, omega=0.4)
        assert rel(host(T), Tref) <= 2e-5


# strips of 8 rows, then of 19 (the last cut short) and of 32
@pytest.mark.parametrize("nx,ny,batch,lines", [(nx, ny, 2, n) for nx, ny in
                                               [(16, 16), (24, 32), (32, 72), (64, 96), (96, 48)]
                                               for n in (1, 2, 3, 4, 5)] +
                         [(1024, 512, 5, 2), (1024, 512, 10, 1), (1024, 512, 10, 4)])
def test_gradient_at_strip_edges(torch, E, oracle, nx, ny, batch, lines):
    Es, d, b, w = spec(lines)
    ln = oracle.Lines(Es, d, b, w, L, PIXEL)
    tau = phantom(ny, nx)
    g = ph.rng(7).normal(size=(ny, nx)).astype(np.float32)
    Tb, db, bb, lb = oracle.vjp(ln, tau, g)
    with E.Plan(nx, ny, PIXEL, L, Es, d, b, w) as p:
        T, gd = cuda(torch, np.stack([tau] * batch)), cuda(torch, np.stack([g] * batch))
        out = torch.empty_like(T)
        gdb, gbb, glb = E.epr_vjp(p.handle, T, gd, out, lines, batch=batch)
    assert rel(host(out), np.stack([Tb] * batch)) <= 1e-5
    for k in range(batch):
        for a, ref in ((gdb[k], db), (gbb[k], bb), (glb[k:k + 1], [lb])):
            assert np.allclose(a, ref, rtol=1e-3, atol=1e-5 * np.abs(np.asarray(ref)).max())
