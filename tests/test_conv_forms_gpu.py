"""The convolution's forms over PSF sides, symmetries and batch sizes: row
strips (compiled sides and groups of 16 taps with every remainder), mirrored
rows, separable passes of any side, row bands, and column strips for images
that fit only so."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2202_07663_gb300 import inputs  # noqa: E402
from gpu_common import assert_plain_parity, oracle_eval  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def abi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_07663_gb300 import abi as _abi, build
    build.build()
    oracle.build()
    return _abi


def _psf(K, kind, seed):
    """full: no symmetry and full rank; mirror: the same rows from the top and
    the bottom, full rank; gaussian: rank 1."""
    if kind == "gaussian":
        return inputs.gaussian_psf(K).astype(np.float32)
    p = np.random.default_rng(seed).uniform(0.1, 1.0, (K, K))
    if kind == "mirror":
        p = p + p[::-1]
    return (p / p.sum()).astype(np.float32)


def _problem(H, W, k, psf, B, seed):
    """A system with flat-cored profiles (n about 1), whose gradient has no
    cusp for a ray to land on, and B vectors around its truth."""
    spec = inputs.SystemSpec(H, W, k, psf.shape[0], "gaussian", inputs.PIXEL_SCALE, 0.2, 100.0)
    rng = np.random.default_rng(seed)
    truth = inputs.draw_truth(rng)
    truth[9], truth[16] = 1.2, 0.8
    model = oracle.simulate(truth, H, W, psf, spec.pixel_scale, k)[0]
    image = inputs.add_noise(rng, model, spec.sigma_bkg, spec.gain_exposure).astype(np.float32)
    return spec, image, inputs.draw_perturbed(rng, truth, B).astype(np.float32)


def _system(abi, spec, image, psf):
    return abi.GLSystem(image, psf, spec.pixel_scale, spec.k, spec.gain_exposure, sigma_bkg=spec.sigma_bkg)


@pytest.mark.parametrize("kind", ["full", "mirror", "gaussian"])
@pytest.mark.parametrize("K", [1, 3, 5, 7, 9, 11, 13, 15, 17, 19, 21, 31, 33, 47])
def test_images_are_the_convolution_of_the_unblurred_image(abi, K, kind):
    """Row bands (2 vectors) and one block per vector (160), W at and past a
    strip: |M - psf * I| <= (K^2 + 8) 2^-24 (|psf| * |I|), the rounding of a
    K^2-term FP32 sum and of its factors, I from the 1 x 1 PSF."""
    for H, W, B in ((40, 37, 2), (33, 48, 160)):
        psf = _psf(K, kind, K)
        spec, image, p = _problem(H, W, 1, psf, B, 10 * K + B)
        p = torch.from_numpy(p).cuda()
        one = _system(abi, spec, image, np.ones((1, 1), np.float32))
        I = one.simulate(p).cpu().numpy().astype(np.float64)
        s = _system(abi, spec, image, psf)
        M = s.simulate(p).cpu().numpy().astype(np.float64)
        if kind == "gaussian" and K >= 5:
            assert s.psf_rank() == 1
        q = psf.astype(np.float64)
        c = K // 2
        ref = np.zeros_like(M)
        pad = np.pad(I, ((0, 0), (c, c), (c, c)))
        for a in range(K):
            for b in range(K):
                ref += q[a, b] * pad[:, 2 * c - a:2 * c - a + H, 2 * c - b:2 * c - b + W]
        assert np.all(np.abs(M - ref) <= (K * K + 8) * 2.0 ** -24 * ref), (K, kind, B)
        one.close()
        s.close()


@pytest.mark.parametrize("K,kind", [(3, "mirror"), (5, "gaussian"), (9, "full"), (13, "mirror"), (13, "gaussian"),
                                    (17, "full"), (17, "gaussian"), (21, "full"), (33, "mirror")])
def test_gradient_of_every_form(abi, K, kind):
    """log L and gradient in bands, in blocks and in a grouped launch: the
    oracle's, and the same gradient bits in the grouped launch."""
    psf = _psf(K, kind, K)
    for B in (3, 153):
        spec, image, p = _problem(41, 46, 2, psf, B, 77 * K + B)
        s, t = _system(abi, spec, image, psf), _system(abi, spec, image, psf)
        d = torch.from_numpy(p).cuda()
        ll, g = [x.cpu().numpy() for x in s.loglik_grad(d)]
        rows = np.unique([0, 1, 2, B - 1])
        rl, _, rg = oracle_eval(spec, image, psf, p[rows])
        assert_plain_parity(ll[rows], g[rows], rl, rg, "conv form K=%d %s B=%d" % (K, kind, B))
        _, grads, _ = abi.loglik_grad_grouped([s, t], [d, d[:1].contiguous()])
        np.testing.assert_array_equal(grads[0].cpu().numpy(), g)
        s.close()
        t.close()


def test_column_strips_where_row_strips_do_not_fit(abi):
    """240 x 225, K = 5: the padded rows of 244 floats need 238 KB, more than a
    block has; the strips' rows of 229 fit. Images of any size that was
    accepted stay accepted, alone and in a grouped launch."""
    psf = _psf(5, "full", 3)
    spec, image, p = _problem(240, 225, 1, psf, 160, 5)
    s, t = _system(abi, spec, image, psf), _system(abi, spec, image, psf)
    for B in (160, 2):
        d = torch.from_numpy(p[:B]).cuda()
        ll, g = [x.cpu().numpy() for x in s.loglik_grad(d)]
        rows = np.unique([0, B // 2, B - 1])
        rl, _, rg = oracle_eval(spec, image, psf, p[rows])
        assert_plain_parity(ll[rows], g[rows], rl, rg, "column strips 240x225 K=5 B=%d" % B)
        _, grads, _ = abi.loglik_grad_grouped([s, t], [d, d[:1].contiguous()])
        np.testing.assert_array_equal(grads[0].cpu().numpy(), g)
    s.close()
    t.close()


def test_profiled_likelihood_in_row_bands(abi):
    """The correlation-only pass in bands (3 vectors, side 13) against the
    same vectors in one block each (160): the tiling of the rays is all that
    differs, a sum's order."""
    psf = _psf(13, "full", 4)
    spec, image, p = _problem(50, 45, 2, psf, 160, 6)
    s = abi.GLSystem(image, psf, spec.pixel_scale, spec.k, spec.gain_exposure, sigma_bkg=spec.sigma_bkg,
                     observed_variance=True)
    d = torch.from_numpy(p).cuda()
    ll, g, amps = [x.cpu().numpy() for x in s.loglik_grad_profiled(d)]
    l3, g3, a3 = [x.cpu().numpy() for x in s.loglik_grad_profiled(d[:3].contiguous())]
    np.testing.assert_array_equal(a3, amps[:3])
    np.testing.assert_array_equal(l3, ll[:3])
    scale = np.abs(g[:3]).max(axis=1, keepdims=True)
    assert np.all(np.abs(g3 - g[:3]) <= 1e-5 * scale)
    s.close()
