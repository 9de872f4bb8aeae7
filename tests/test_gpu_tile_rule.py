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
