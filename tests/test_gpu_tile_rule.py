"""The rules that choose the splat's tile at each launch: their place in the
tuning vector, and the kernels they count."""
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


def host(t):
    return t.detach().cpu().numpy().astype(np.float64)


def test_default_tile_survives_a_tuning_round_trip(torch, E):
    """An untuned plan has no one splat tile: it is chosen at each launch.  The
    tuning says so, and a plan that is given it chooses at each launch too."""
    args = (512, 512, PIXEL, L, [80.0], [ph.BONE[0]], [ph.BONE[1]])
    D = cuda(torch, ph.rng(2).uniform(0.5, 1.0, size=(512, 512)))

    def solve(p):
        T = torch.empty_like(D)
        E.epr_solve_nonlocal(p.handle, D, T, n_iter=2, omega=0.4, want_info=False)
        return T

    with E.Plan(*args) as a, E.Plan(*args) as b:
        tun = E.epr_plan_get_tuning(a.handle)
        assert tun["splat_tile"] == [0, 0] and not tun["tuned"]
        E.epr_plan_set_tuning(b.handle, tun)
        assert E.epr_plan_get_tuning(b.handle) == dict(tun, tuned=True)
        ref = solve(a)
        assert rel(host(solve(b)), host(ref)) <= 1e-6
        E.epr_plan_set_tuning(b.handle, dict(tun, splat_tile=[64, 32]))   # one tile, and back
        assert E.epr_plan_get_tuning(b.handle)["splat_tile"] == [64, 32]
        assert rel(host(solve(b)), host(ref)) <= 1e-6
        E.epr_plan_set_tuning(b.handle, tun)
        assert E.epr_plan_get_tuning(b.handle)["splat_tile"] == [0, 0]
        for bad in ([0, 64], [64, 0], [16, 16]):
            with pytest.raises(E.EprError):
                E.epr_plan_set_tuning(b.handle, dict(tun, splat_tile=bad))
        with pytest.raises(E.EprError):   # six blocks per SM belong to a tile
            E.epr_plan_set_tuning(b.handle, dict(tun, splat_blocks_per_sm=6))


# an x-dependent spectrum runs two 512-thread blocks per SM with one line too:
# 243 blocks of a tile fill the chip.  Sizes on both sides of the 32 x 64 and
# the 64 x 64 line; the tile does not change a bit of the integer sums.
@pytest.mark.parametrize("nx,ny,batch", [(512, 768, 1), (768, 768, 1), (1024, 768, 1), (1024, 1024, 1),
                                         (512, 512, 4)])
def test_xspec_tiles_of_one_line(torch, E, nx, ny, batch):
    ells = ph.random_ellipsoids(ny, nx, 8, 8.0, 20.0, margin=4.0, seed=nx)
    tau = ph.project_ellipsoids(ells, ny, nx, PIXEL).astype(np.float32)
    X = np.array([0.0, nx - 1.0])
    W, Dl, Bt = np.ones((1, 2)), ph.BONE[0] * np.array([[0.9, 1.1]]), ph.BONE[1] * np.array([[1.1, 0.9]])
    with E.Plan(nx, ny, PIXEL, L, [80.0], [ph.BONE[0]], [ph.BONE[1]]) as p:
        E.epr_plan_set_xspec(p.handle, X, W, Dl, Bt)
        T = cuda(torch, np.stack([tau] * batch))
        tun = E.epr_plan_get_tuning(p.handle)
        got = []
        for tile in ([0, 0], [64, 64], [32, 64], [64, 32], [32, 32]):
            E.epr_plan_set_tuning(p.handle, dict(tun, splat_tile=tile))
            P = torch.empty_like(T)
            E.epr_forward(p.handle, T, P, batch=batch)
            got.append(P)
    for P in got[1:]:
        assert torch.equal(P, got[0])
