"""The gradient with respect to a light's Sersic index against the FP64 oracle
on a residual of one sign, where the sums over rays do not cancel by chance."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2202_07663_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def abi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_07663_gb300 import abi as _abi, build
    build.build()
    oracle.build()
    return _abi


@pytest.mark.parametrize("n", [0.7, 1.0, 2.0, 8.0])
def test_index_entry_on_a_bright_image(abi, n):
    """A ray's term is b_n s ln s / n - 1.9992 (s - 1), whose parts cancel to
    about 1 / (6 n) of them. With a third of a rounding left of each after the
    sum, nine vectors in ten are within 2 n roundings (two at least) of the
    entry. From sums of g e s and g e over all rays, so from parts that cancel
    to s - 1 once more, they are not."""
    rng = np.random.default_rng(17)
    truth = inputs.draw_truth(np.random.default_rng(3))
    truth[8:15] = [0.5, n, 0.05, -0.1, 0.01, 0.02, 30.0]
    truth[21] = 0.01
    p = (truth * (1 + 0.01 * rng.standard_normal((256, 22)))).astype(np.float32)
    one = np.ones((1, 1), np.float32)
    model = oracle.simulate(p[:1].astype(np.float64), 40, 40, one, 0.065, 2)[0]
    image = (2 * model + 3).astype(np.float32)
    s = abi.GLSystem(image, one, 0.065, 2, 0.0, sigma_bkg=0.3)
    g = s.loglik_grad(torch.from_numpy(p).cuda())[1].cpu().numpy()
    s.close()
    ref = oracle.loglik(p.astype(np.float64), image, np.float32(0.3), one, 0.065, 2, 0.0, grad=True)[2]
    err = np.abs(g[:, 9] - ref[:, 9]) / np.abs(ref[:, 9])
    assert np.percentile(err, 90) <= max(2.0, 2 * n) * 2.0 ** -24
