"""The gradient's mass entries ray by ray: images of one ray (1 x 1, k = 1),
whose gradient is that ray's derivatives alone, so that rounding does not
average out over rays. Bounds in units of 2^-24 of the norm of the eight mass
entries, against the FP64 oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402

pytestmark = pytest.mark.gpu

B = 2048


@pytest.fixture(scope="module")
def abi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_07663_gb300 import abi as _abi, build
    build.build()
    oracle.build()
    return _abi


def _rays(eps, seed, gamma=(1.6, 2.4)):
    """B vectors, each with its lens centre elsewhere around the one ray and a
    broad source (n = 1, R = 4) whose centre lies five arcsec off: its slope is
    the same over the rounding of a position."""
    rng = np.random.default_rng(seed)
    p = np.zeros((B, 22))
    r, phi, psi = rng.uniform(0.3, 2.0, B), rng.uniform(0, 2 * np.pi, B), rng.uniform(0, 2 * np.pi, B)
    p[:, 0], p[:, 1] = rng.uniform(0.8, 1.4, B), rng.uniform(*gamma, B)
    p[:, 2], p[:, 3] = eps * np.cos(phi), eps * np.sin(phi)
    p[:, 4], p[:, 5] = r * np.cos(psi), r * np.sin(psi)
    p[:, 8:15] = [1.0, 1.0, 0.0, 0.0, 3.0, 3.0, 1e-3]
    p[:, 15:22] = [4.0, 1.0, 0.0, 0.0, 5.0, 0.0, 1.0]
    return p.astype(np.float32)


def _errors(abi, p):
    """|error| of the eight mass entries over their norm, per vector, and the entries' own."""
    image, one = np.full((1, 1), 100.0, np.float32), np.ones((1, 1), np.float32)
    s = abi.GLSystem(image, one, 0.065, 1, 0.0, sigma_bkg=1.0)
    g = s.loglik_grad(torch.from_numpy(p).cuda())[1].cpu().numpy()[:, :8]
    s.close()
    ref = oracle.loglik(p.astype(np.float64), image, np.float32(1.0), one, 0.065, 1, 0.0, grad=True)[2][:, :8]
    return np.linalg.norm(g - ref, axis=1) / np.linalg.norm(ref, axis=1), g, ref


@pytest.mark.parametrize("eps", [0.3, 0.7, 0.8, 0.85])
def test_ellipticity_enters_the_error_once(abi, eps):
    """dF/du carries 1 / (1 - u), |u| = |eps|: a rounding of u is 1 / (1 - |eps|)
    of it. Six such roundings and eight of the rest hold for 99 in 100 rays; a
    squared modulus formed as 1 + |u|^2 - 2 Re u has it to the second power."""
    err = _errors(abi, _rays(eps, int(100 * eps)))[0]
    assert np.percentile(err, 99) <= (8 + 6 / (1 - eps)) * 2.0 ** -24


@pytest.mark.parametrize("eps", [0.2, 0.5, 0.8, 0.85])
def test_slope_derivative_of_long_series(abi, eps):
    """d/dgamma takes dF/dt, a sum of up to 90 terms here. Half of the rays
    within three roundings and three that 1 / (1 - |eps|) enlarges, of the
    entry: the sum of a long series adds none of its own."""
    _, g, ref = _errors(abi, _rays(eps, 7 + int(100 * eps), gamma=(2.6, 2.9)))
    assert np.median(np.abs(g[:, 1] - ref[:, 1]) / np.abs(ref[:, 1])) <= (3 + 3 / (1 - eps)) * 2.0 ** -24


@pytest.mark.parametrize("gamma", [1.0, 1.001, 1.1, 1.26, 0.9])
@pytest.mark.parametrize("eps", [0.05, 0.3, 0.6])
def test_slope_derivative_near_the_isothermal_limit(abi, eps, gamma):
    """At gamma = 1 every coefficient of F vanishes and its derivative does
    not: the series is as long as dF/dt needs. The bound of the long series."""
    _, g, ref = _errors(abi, _rays(eps, 11, gamma=(gamma, gamma)))
    assert np.median(np.abs(g[:, 1] - ref[:, 1]) / np.abs(ref[:, 1])) <= (3 + 3 / (1 - eps)) * 2.0 ** -24
