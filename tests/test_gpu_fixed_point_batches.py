"""Fixed-point results do not depend on the batch a projection is solved in:
its maps, its convergence record and its gradients are the same bits alone and
in a call of several, on both sides of the sizes at which a float launch takes
another block shape, column tile or strip height."""
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


def plan(E, nx, ny, lines, near=False):
    Es, d, b, w = ph.spectrum(lines, 60.0, 160.0, 95.0, 30.0, ph.BONE[0], ph.BONE[1], 80.0, 5)
    pixel, dist = (6.5e-6, 0.3) if near else (PIXEL, L)
    return E.Plan(nx, ny, pixel, dist, Es, d, b, w, deterministic=True)


def thickness(torch, nx, ny, batch, pixel=PIXEL):
    """`batch` different maps: one phantom, rolled and scaled."""
    hi = min(20.0, min(ny, nx) / 5.0)
    ells = ph.random_ellipsoids(ny, nx, 8, 0.4 * hi, hi, margin=4.0, seed=nx + ny)
    t = ph.project_ellipsoids(ells, ny, nx, pixel).astype(np.float32)
    return torch.from_numpy(np.stack([np.roll(t, 3 * k, 1) * np.float32(1.0 + 0.03 * k)
                                      for k in range(batch)])).cuda()


@pytest.mark.parametrize("nx,ny,lines,batch", [(512, 512, 1, 16), (512, 512, 2, 20), (256, 256, 1, 40),
                                               (128, 512, 1, 24), (144, 288, 1, 20), (512, 1024, 1, 4),
                                               (1024, 768, 2, 6), (648, 1296, 1, 3), (384, 192, 3, 32)])
def test_solve_bits_alone_and_in_a_batch(torch, E, nx, ny, lines, batch):
    Tr = thickness(torch, nx, ny, batch)
    with plan(E, nx, ny, lines) as p:
        D = torch.empty_like(Tr)
        E.epr_forward(p.handle, Tr, D, batch=batch)
        T = torch.empty_like(D)
        all_ = E.epr_solve_nonlocal(p.handle, D, T, batch=batch, n_iter=4, omega=0.4)
        for k in (0, batch // 2, batch - 1):
            one, Dk = torch.empty_like(D[k]), D[k].clone()
            got = E.epr_solve_nonlocal(p.handle, Dk, one, n_iter=4, omega=0.4)
            assert torch.equal(one, T[k])
            assert np.array_equal(got["rho_hist"][0], all_["rho_hist"][k])
            assert np.array_equal(got["kappa_hist"][0], all_["kappa_hist"][k])


@pytest.mark.parametrize("model", [1, 2, 3])
def test_stencil_solve_bits_alone_and_in_a_batch(torch, E, model):
    nx, ny, batch = 512, 288, 12
    Tr = thickness(torch, nx, ny, batch, PIXEL if model == 3 else 6.5e-6)
    with plan(E, nx, ny, 2, near=model < 3) as p:
        D = torch.empty_like(Tr)
        E.epr_forward(p.handle, Tr, D, batch=batch, model=model)

        def solve(Dk, Tk, n):
            if model == 3:
                return E.epr_solve_nonlocal_wkb1(p.handle, Dk, Tk, batch=n, n_iter=4, omega=0.4)
            return E.epr_solve_local(p.handle, Dk, Tk, order=model, batch=n, n_iter=4, omega=0.4)

        T = torch.empty_like(D)
        all_ = solve(D, T, batch)
        for k in (0, batch - 1):
            one, Dk = torch.empty_like(D[k]), D[k].clone()
            got = solve(Dk, one, 1)
            assert torch.equal(one, T[k])
            assert np.array_equal(got["rho_hist"][0], all_["rho_hist"][k])
            assert np.array_equal(got["kappa_hist"][0], all_["kappa_hist"][k])


def test_gradient_bits_alone_and_in_a_batch(torch, E):
    nx, ny, lines, batch = 512, 384, 3, 12
    T = thickness(torch, nx, ny, batch)
    g = torch.randn(T.shape, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    with plan(E, nx, ny, lines) as p:
        out = torch.empty_like(T)
        all_ = E.epr_vjp(p.handle, T, g, out, lines, batch=batch)
        for k in (0, batch - 1):
            one = torch.empty_like(T[k])
            got = E.epr_vjp(p.handle, T[k].clone(), g[k].clone(), one, lines)
            assert torch.equal(one, out[k])
            for a, b in zip(got, all_):
                assert np.array_equal(np.ravel(a), np.ravel(np.asarray(b)[k]))
