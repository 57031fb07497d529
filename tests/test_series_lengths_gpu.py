"""Every compiled series length of the ray kernels (one to six pairs of terms)
and the loop beyond them, alone and in a batch large enough to be ordered;
and the profiled likelihood's weighted sums at the ends of their range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2202_07663_gb300 import inputs  # noqa: E402
from gpu_common import assert_plain_parity, oracle_eval  # noqa: E402

pytestmark = pytest.mark.gpu

# |eps| from 0 (one term) over each pair count up to past the compiled ones
ELLIPTICITIES = [0.0, 1e-5, 1e-3, 0.01, 0.03, 0.06, 0.1, 0.14, 0.17, 0.2, 0.23, 0.26, 0.3, 0.4, 0.55]


@pytest.fixture(scope="module")
def abi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_07663_gb300 import abi as _abi, build
    build.build()
    oracle.build()
    return _abi


def _problem(k=2, H=30, W=27):
    """A system with flat-cored profiles (n about 1), one vector per ellipticity."""
    spec = inputs.SystemSpec(H, W, k, 5, "moffat", inputs.PIXEL_SCALE, 0.2, 100.0)
    rng = np.random.default_rng(11)
    truth = inputs.draw_truth(rng)
    truth[9], truth[16] = 1.2, 0.8
    psf = inputs.make_psf(spec).astype(np.float32)
    model = oracle.simulate(truth, H, W, psf, spec.pixel_scale, k)[0]
    image = inputs.add_noise(rng, model, spec.sigma_bkg, spec.gain_exposure).astype(np.float32)
    p = inputs.draw_perturbed(rng, truth, len(ELLIPTICITIES)).astype(np.float32)
    phi = rng.uniform(0.0, 2.0 * np.pi, len(p))
    p[:, 2], p[:, 3] = ELLIPTICITIES * np.cos(phi), ELLIPTICITIES * np.sin(phi)
    # the oracle's angle is undefined at eps = 0 and its gradient with it
    return spec, image, psf, p.astype(np.float32)


@pytest.mark.parametrize("copies", [1, 11])
def test_every_series_length(abi, copies):
    spec, image, psf, p = _problem()
    s = abi.GLSystem(image, psf, spec.pixel_scale, spec.k, spec.gain_exposure, sigma_bkg=spec.sigma_bkg)
    d = torch.from_numpy(np.tile(p, (copies, 1))).cuda()
    ll, g = [t.cpu().numpy() for t in s.loglik_grad(d)]
    images = s.simulate(d).cpu().numpy()
    for c in range(1, copies):
        np.testing.assert_array_equal(g[c * len(p):(c + 1) * len(p)], g[:len(p)])
    ref = oracle.simulate(p.astype(np.float64), spec.H, spec.W, psf, spec.pixel_scale, spec.k)
    err = np.abs(images[:len(p)] - ref) / (1e-4 * np.abs(ref) + 1e-5 * np.abs(ref).max(axis=(1, 2), keepdims=True))
    assert err.max() <= 1.0
    rl, _, rg = oracle_eval(spec, image, psf, p[1:])
    assert_plain_parity(ll[1:len(p)], g[1:len(p)], rl, rg, "series lengths, %d copies" % copies)
    s.close()


@pytest.mark.parametrize("lo,hi", [(0.2, 0.2), (1e-3, 1e3), (1e-12, 1e-12), (1e-15, 1e10), (1e12, 1e12)])
def test_solved_amplitudes_over_noise_ranges(abi, lo, hi):
    """Noise maps from equal to 25 decades apart, the last ones beyond what a
    float's range carries (the FP64 sums): the amplitudes solve the normal
    equations of the unit images in FP64, to FP32 images' rounding."""
    spec, image, psf, p = _problem(k=1)
    noise = np.where(np.arange(spec.H * spec.W).reshape(spec.H, spec.W) % 3 == 0, lo, hi).astype(np.float32)
    s = abi.GLSystem(image, psf, spec.pixel_scale, spec.k, 0.0, noise_map=noise, observed_variance=True)
    p = p[4:8]
    _, _, amps = s.loglik_grad_profiled(torch.from_numpy(p).cuda())
    unit = []
    for keep, drop in ((14, 21), (21, 14)):
        q = p.copy()
        q[:, keep], q[:, drop] = 1.0, 0.0
        unit.append(s.simulate(torch.from_numpy(q).cuda()).cpu().numpy().astype(np.float64))
    w = 1.0 / (noise * noise).astype(np.float64)
    for b in range(len(p)):
        A = np.stack([u[b].ravel() for u in unit], 1) * np.sqrt(w.ravel())[:, None]
        ref = np.linalg.lstsq(A, image.astype(np.float64).ravel() * np.sqrt(w.ravel()), rcond=None)[0]
        np.testing.assert_allclose(amps[b].cpu().numpy(), ref, rtol=1e-6)
    s.close()
