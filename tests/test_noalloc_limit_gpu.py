"""gl_loglik_grad_noalloc up to the edge of its static scratch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2202_07663_gb300 import inputs  # noqa: E402
from gpu_common import assert_plain_parity, make_system  # noqa: E402

pytestmark = pytest.mark.gpu

SCRATCH_BYTES = 32 << 20


def _call(side, k, past):
    from paper_2202_07663_gb300 import abi, build
    build.build()
    oracle.build()
    up = lambda n: (n + 255) & ~255  # noqa: E731
    B = SCRATCH_BYTES // (4 * side * side + 1232 + 192)
    while up(1232 * B) + up(4 * side * side * B) + up(192 * B) > SCRATCH_BYTES:
        B -= 1
    B += past
    spec = inputs.SystemSpec(side, side, k, 5, "gaussian")
    truth, image, psf = make_system(spec, side)
    s = abi.GLSystem(image, psf, spec.pixel_scale, k, spec.gain_exposure, sigma_bkg=spec.sigma_bkg)
    p = torch.from_numpy(inputs.draw_perturbed(np.random.default_rng(side), truth, B).astype(np.float32)).cuda()
    ll = torch.empty(B, dtype=torch.float64, device="cuda")
    g = torch.empty(B, 22, dtype=torch.float64, device="cuda")
    rc = abi.lib_handle().gl_loglik_grad_noalloc(s.handle, p.data_ptr(), B, ll.data_ptr(), None, g.data_ptr(),
                                                 torch.cuda.current_stream().cuda_stream)
    return rc, s, p, ll, g


@pytest.mark.parametrize("side,k", [(100, 4), (200, 4)])
def test_largest_batches_take_the_tiles_that_fit(side, k):
    """100 x 100, k = 4: 810 vectors fit with one tile each, and the plan for
    speed wants more from 799 on. The results of gl_loglik_grad."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rc, s, p, ll, g = _call(side, k, 0)
    assert rc == 0
    rl, rg = s.loglik_grad(p)
    assert_plain_parity(*[t.cpu().numpy() for t in (ll, g, rl, rg)], "no-alloc limit %d" % side)
    s.close()


def test_one_vector_more_is_refused():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rc, s, *_ = _call(100, 4, 1)
    assert rc == -1
    s.close()
