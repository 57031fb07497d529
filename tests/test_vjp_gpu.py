"""The fused backward of the autograd log-likelihood (gl_scale_rows_f32)
against the torch expression it stands for, and the cases that must keep that
expression: gradients of gradients, batched gradients, float64 parameters."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2202_07663_gb300 import inputs  # noqa: E402
from gpu_common import make_system  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_07663_gb300 import abi, build, hmc
    build.build()
    oracle.build()
    spec = inputs.SystemSpec(20, 23, 1, 5)
    truth, image, psf = make_system(spec, 31)
    s = abi.GLSystem(image, psf, spec.pixel_scale, spec.k, spec.gain_exposure, sigma_bkg=spec.sigma_bkg)
    p = inputs.draw_perturbed(np.random.default_rng(3), truth, 37).astype(np.float32)
    return hmc, s, torch.from_numpy(p).cuda()


@pytest.mark.parametrize("B", [1, 2, 37])
def test_fused_backward_equals_the_torch_expression(setup, B):
    hmc, s, p0 = setup
    p = p0[:B].clone().requires_grad_()
    g = s.loglik_grad(p0[:B].contiguous())[1]
    w = torch.randn(2 * B, device="cuda")
    for make in (lambda ll: ll.sum(), lambda ll: (ll * w[:B]).sum(), lambda ll: (ll * w[::2]).sum(),
                 lambda ll: ll.mean()):
        ll = hmc.loglik(p, s)
        (go,) = torch.autograd.grad(make(ll), ll, retain_graph=True)
        (out,) = torch.autograd.grad(make(ll), p)
        assert out.dtype == torch.float32
        assert torch.equal(out, (go.to(torch.float64)[:, None] * g).to(torch.float32))
    # a strided incoming gradient
    ll = hmc.loglik(p, s)
    (out,) = torch.autograd.grad(ll, p, grad_outputs=w[::2])
    assert torch.equal(out, (w[::2].to(torch.float64)[:, None] * g).to(torch.float32))


def test_other_uses_keep_the_torch_expression(setup):
    hmc, s, p0 = setup
    g = s.loglik_grad(p0)[1]
    # the product's own derivative with respect to the incoming gradient
    p = p0.clone().requires_grad_()
    w = torch.randn(len(p0), device="cuda", requires_grad=True)
    (out,) = torch.autograd.grad(hmc.loglik(p, s), p, grad_outputs=w, create_graph=True)
    (dw,) = torch.autograd.grad(out.sum(), w)
    np.testing.assert_allclose(dw.cpu().numpy(), g.sum(1).cpu().numpy(), rtol=1e-5, atol=1e-5 * float(g.abs().max()))
    # a batch of incoming gradients
    W = torch.randn(3, len(p0), device="cuda")
    (out,) = torch.autograd.grad(hmc.loglik(p, s), p, grad_outputs=W, is_grads_batched=True)
    assert torch.equal(out, (W.to(torch.float64)[:, :, None] * g).to(torch.float32))
    # float64 parameters
    q = p0.double().requires_grad_()
    (out,) = torch.autograd.grad(hmc.loglik(q, s).sum(), q)
    assert out.dtype == torch.float64 and torch.equal(out, g)
    # a hook that holds the saved gradient on the host and brings it back
    with torch.autograd.graph.save_on_cpu():
        ll = hmc.loglik(p, s)
    (out,) = torch.autograd.grad(ll.sum(), p)
    assert torch.equal(out, g.to(torch.float32))


def _expression(go, g):
    return (go.to(torch.float64)[:, None] * g).to(torch.float32)


def test_incoming_gradient_whose_memory_holds_its_negative(setup):
    """The imaginary part of a conjugate is a view of the unconjugated memory
    with torch's negative bit; given as grad_outputs and as the engine forms it
    for a complex function of log L. A zero tensor has no memory at all."""
    hmc, s, p0 = setup
    p = p0.clone().requires_grad_()
    g = s.loglik_grad(p0)[1]
    z = torch.complex(torch.randn(len(p0), device="cuda"), torch.randn(len(p0), device="cuda"))
    go = z.conj().imag
    assert go.is_neg()
    (out,) = torch.autograd.grad(hmc.loglik(p, s), p, grad_outputs=go)
    assert torch.equal(out, _expression(-z.imag, g))
    ll = hmc.loglik(p, s)
    value = (torch.complex(torch.zeros_like(ll), ll).conj() * z.conj()).imag.sum()
    (go,) = torch.autograd.grad(value, ll, retain_graph=True)
    (out,) = torch.autograd.grad(value, p)
    assert torch.equal(out, _expression(-z.real, g)) and torch.equal(out, _expression(go, g))
    zero = torch._efficientzerotensor((len(p0),), device="cuda")
    (out,) = torch.autograd.grad(hmc.loglik(p, s), p, grad_outputs=zero)
    assert torch.equal(out, torch.zeros_like(out))


def test_sparse_incoming_gradient(setup):
    """gather(sparse_grad=True) on log L sends back a sparse gradient: the rows
    of the gathered vectors, whole."""
    hmc, s, p0 = setup
    p = p0.clone().requires_grad_()
    g = s.loglik_grad(p0)[1]
    rows = torch.tensor([1, 5, 20], device="cuda")
    (out,) = torch.autograd.grad(torch.gather(hmc.loglik(p, s), 0, rows, sparse_grad=True).sum(), p)
    ref = torch.zeros(g.shape, device="cuda")
    ref[rows] = g[rows].to(torch.float32)
    assert torch.equal(out, ref)


def test_dispatch_mode_sees_the_product(setup):
    """A dispatch mode (a tracer, an operation counter) that is active during
    the backward pass gets the product as torch operations."""
    from torch.utils._python_dispatch import TorchDispatchMode
    hmc, s, p0 = setup
    seen = []

    class Record(TorchDispatchMode):
        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            seen.append(str(func))
            return func(*args, **(kwargs or {}))

    p = p0.clone().requires_grad_()
    ll = hmc.loglik(p, s)
    w = torch.randn(len(p0), device="cuda")
    with Record():
        (out,) = torch.autograd.grad(ll, p, grad_outputs=w)
    assert any(name.startswith("aten.mul") for name in seen)
    assert torch.equal(out, _expression(w, s.loglik_grad(p0)[1]))


def test_scaled_rows_up_to_the_largest_product(setup):
    """B d = 2^31 - 4096, where a 32-bit signed index would step past its range:
    the first and last rows scaled, nothing else touched (26 GB)."""
    from paper_2202_07663_gb300 import abi
    B, d = (1 << 19) - 1, 4096
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB free")
    rows = torch.zeros(B, d, dtype=torch.float64, device="cuda")
    out = torch.full((B, d), 7.0, dtype=torch.float32, device="cuda")
    rows[0], rows[-1] = 1.0, torch.arange(d, dtype=torch.float64, device="cuda")
    scale = torch.full((B,), 2.0, device="cuda")
    scale[-1] = 3.0
    abi.gl_scale_rows_f32(B, d, scale.data_ptr(), 1, rows.data_ptr(), out.data_ptr(), abi._stream_ptr(out.device))
    assert torch.equal(out[0], torch.full((d,), 2.0, device="cuda"))
    assert torch.equal(out[-1], 3.0 * torch.arange(d, dtype=torch.float32, device="cuda"))
    assert int(torch.count_nonzero(out)) == d + d - 1
    del rows, out
    torch.cuda.empty_cache()
