"""The profiled likelihood's solved amplitudes where the two unit images are
nearly the same, so that the solve magnifies the rounding of its five weighted
inner products, and where they are not: against the normal equations of the
same FP32 images in extended precision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2202_07663_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def abi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_07663_gb300 import abi as _abi, build
    build.build()
    return _abi


@pytest.mark.parametrize("side,delta", [(40, 1e-5), (80, 1e-5), (80, 1e-3), (80, 0.3)])
def test_inner_products_carry_double_precision(abi, side, delta):
    """A lens too light to deflect in front of a source delta larger than its
    own light. Their correlation leaves 1 / kappa = det / (<A,A> <S,S>), and a
    relative rounding r of the sums moves I_l by r ((<S,S><A,D> + <A,S><S,D>) /
    det + 2 kappa |I_l|). Sums in FP64 keep r below 2 x 2^-53 (three products
    and a tree, averaged over the pixels), root mean square over 24 vectors."""
    rng = np.random.default_rng(side)
    B = 24
    p = np.zeros((B, 22), np.float32)
    p[:, 0], p[:, 1] = 1e-7, 2.0
    R = 0.5 * (1 + 0.1 * rng.random(B))
    p[:, 8], p[:, 9], p[:, 12], p[:, 13], p[:, 14] = R, 1.0, 0.011, -0.023, 1.0
    p[:, 15], p[:, 16], p[:, 19], p[:, 20], p[:, 21] = R * (1 + delta), 1.0, 0.011, -0.023, 1.0
    noise = rng.uniform(0.2, 0.4, (side, side)).astype(np.float32)
    psf = inputs.gaussian_psf(5).astype(np.float32)
    blank = np.ones((side, side), np.float32)
    scene = abi.GLSystem(blank, psf, inputs.PIXEL_SCALE, 1, 0.0, noise_map=noise)
    unit = []
    for keep, drop in ((14, 21), (21, 14)):
        q = p.copy()
        q[:, keep], q[:, drop] = 1.0, 0.0
        unit.append(scene.simulate(torch.from_numpy(q).cuda()).cpu().numpy().reshape(B, -1).astype(np.longdouble))
    scene.close()
    scale = float(unit[0].max())
    image = (20 * unit[0][0] + 5 * unit[1][0]).reshape(side, side) / scale + 0.3 * rng.standard_normal((side, side))
    image = image.astype(np.float32)
    s = abi.GLSystem(image, psf, inputs.PIXEL_SCALE, 1, 0.0, noise_map=noise, observed_variance=True)
    amps = s.loglik_grad_profiled(torch.from_numpy(p).cuda())[2].cpu().numpy()
    s.close()
    w = 1 / (noise * noise).ravel().astype(np.longdouble)
    D = image.ravel().astype(np.longdouble)
    over = []
    for b in range(B):
        A, S = unit[0][b], unit[1][b]
        aa, as_, ss, ad, sd = [(w * u * v).sum() for u, v in ((A, A), (A, S), (S, S), (A, D), (S, D))]
        det = aa * ss - as_ * as_
        Il = (ss * ad - as_ * sd) / det
        bound = 2 * 2.0 ** -53 * ((abs(ss * ad) + abs(as_ * sd)) / det + 2 * aa * ss / det * abs(Il))
        over.append(float(abs(amps[b, 0] - Il) / bound))
    assert np.sqrt(np.mean(np.square(over))) <= 1.0
