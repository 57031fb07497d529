"""gl_system_reserve(B): no call of 1 .. B vectors grows the scratch."""
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


@pytest.mark.parametrize("H,W,k,B", [(40, 40, 2, 100), (30, 27, 1, 300), (100, 90, 3, 60), (200, 200, 4, 150)])
def test_no_smaller_call_grows_the_scratch(abi, H, W, k, B):
    """The tiles of a call are not monotone in its size: 40 x 40, k = 2 has 400
    at 100 vectors and 455 at 91."""
    rng = np.random.default_rng(H + B)
    image = rng.normal(1.0, 0.3, (H, W)).astype(np.float32)
    psf = inputs.gaussian_psf(5).astype(np.float32)
    s = abi.GLSystem(image, psf, inputs.PIXEL_SCALE, k, 100.0, sigma_bkg=0.2)
    p = torch.from_numpy(inputs.draw_perturbed(rng, inputs.draw_truth(rng), B).astype(np.float32)).cuda()
    s.reserve(B)
    held = s.scratch_held()
    for b in range(B, 0, -1):
        assert s.scratch_bytes(b) <= held
        s.loglik_grad(p[:b].contiguous())
        assert s.scratch_held() == held, b
    s.close()
