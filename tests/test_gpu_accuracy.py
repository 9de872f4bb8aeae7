"""Errors against 64 bits, with bounds taken from the arithmetic."""
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


# The filter is four transforms along an axis.  Of one transform of up to 2592
# points: at most 11.4 levels of additions, each off by 2.4e-8 rms (a rounding of
# 2^-25 to 2^-24, uniform), and at most four layers of twiddle products, each off
# by 5.5e-8 (the table's rounding and a complex product's):
# sqrt(4 (11.4 2.4^2 + 4 5.5^2)) 1e-8 = 2.7e-7; the bound leaves 35 %.
@pytest.mark.parametrize("n", [144, 384, 648, 768, 864, 1152, 1296, 1728, 2304, 2592])
def test_filter_error_of_ragged_lengths(torch, E, n):
    g = torch.randn(n, n, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    mu = 2.0 * (2.0 * np.pi / (1.2398419843320026e-6 / 80e3)) * ph.BONE[1]
    fy = torch.fft.fftfreq(n, PIXEL, dtype=torch.float64, device="cuda")[:, None]
    fx = torch.fft.rfftfreq(n, PIXEL, dtype=torch.float64, device="cuda")[None]
    H = mu / (mu + L * ph.BONE[0] * 4.0 * np.pi ** 2 * (fx * fx + fy * fy))
    ref = torch.fft.irfft2(torch.fft.rfft2(g.double()) * H, s=(n, n))
    with E.Plan(n, n, PIXEL, L, [80.0], [ph.BONE[0]], [ph.BONE[1]]) as p:
        E.epr_precondition(p.handle, g)
    err = ((g.double() - ref).norm() / ref.norm()).item()
    print("filter %d: %.2e" % (n, err))
    assert err <= 3.7e-7


# A thickness ramp whose shift is exactly half a pixel, and a misfit gradient of
# 2^24 and 1 - 2^24 in turn: the bilinear value is exactly 1/2 everywhere (the
# weights, their products and their sum are exact), and dF/dbeta = -2 k sum of
# T I / 2.  The difference of two corners needs 25 bits: a value formed from it
# is 0 and 1 in turn.  5e-6: exponentials, products and float sums of 48 terms.
def test_gradient_of_large_alternating_misfits(torch, E):
    nx, ny = 96, 48
    delta, dist, pixel, beta = 2.0 ** -21, 1.0, 2.0 ** -16, 1e-11   # the shift constant is -2^11
    k = 2.0 * np.pi / (1.2398419843320026e-6 / 80e3)
    x = np.arange(nx)
    T = np.broadcast_to((x * 2.0 ** -12).astype(np.float32), (ny, nx))
    g = np.broadcast_to(np.where(x % 2 == 0, 2.0 ** 24, 1.0 - 2.0 ** 24).astype(np.float32), (ny, nx))
    with E.Plan(nx, ny, pixel, dist, [80.0], [delta], [beta]) as p:
        Td, gd = (torch.from_numpy(a.copy()).cuda() for a in (T, g))
        _, got, _ = E.epr_vjp(p.handle, Td, gd, torch.empty_like(Td), 1)
    T = T.astype(np.float64)
    ref = -2.0 * k * 0.5 * (T * np.exp(-2.0 * k * beta * T)).sum()   # T = 0 in the column with a corner outside
    assert abs(np.ravel(got)[0] / ref - 1.0) <= 5e-6


# No shift (L = 0), unit intensity, a thickness ramp of 2^-12 per column and a
# misfit gradient in every eighth row: dF/dL = -delta / p^2 times the sum of 2^-12
# (g(x + 1) - g(x)), with nothing beyond the last column, which telescopes to
# -2^-12 g(0) per row.  Every term is a multiple of 2^-12 that a float holds (up to
# 2^23 of them); the sums of a warp's lanes are not.
def test_gradient_scalars_that_cancel(torch, E):
    nx, ny = 96, 48
    delta, pixel, beta = 2.0 ** -21, 2.0 ** -16, 1e-19   # exp(-mu T) is 1
    g = np.zeros((ny, nx), np.float32)
    g[::8] = ph.rng(3).integers(-2 ** 22, 2 ** 22, size=(ny // 8, nx))
    g[::8, 0] = 1.0
    T = np.tile((np.arange(nx) * 2.0 ** -12).astype(np.float32), (ny, 1))
    with E.Plan(nx, ny, pixel, 0.0, [80.0], [delta], [beta]) as p:
        Td, gd = torch.from_numpy(T).cuda(), torch.from_numpy(g).cuda()
        _, _, got = E.epr_vjp(p.handle, Td, gd, torch.empty_like(Td), 1)
    ref = -delta / pixel ** 2 * (ny // 8) * (-2.0 ** -12)
    assert abs(np.ravel(got)[0] / ref - 1.0) <= 1e-12
