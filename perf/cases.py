"""What a user of this framework has it do, as timed calls through its public entry points.

A case is one lens system (image H x W, supersampling k, PSF side K and shape, noise model), a batch of B
parameter vectors with the distribution they come from, and the call that is made on them:

- ``grad``: log L and its gradient, ``GLSystem.loglik_grad``, both taken to the parameters' own float32 as
  an optimiser or sampler over float32 parameters does;
- ``autograd``: the same through ``hmc.loglik`` and ``torch.autograd.grad`` (float32 in, float32 out);
- ``graph``: ``grad`` captured once into a CUDA graph and replayed, as the HMC driver replays its steps;
- ``loglik``: log L alone; ``simulate``: the model images; ``profiled``: the likelihood with the observed-image
  variance and solved amplitudes; ``grouped``: several systems in one set of launches.

Observed images come from the float64 model below (the seed's truth plus noise), so that inputs do not depend
on the code that is timed.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2202_07663_gb300 import abi, hmc, inputs

NPARAM = inputs.NPARAM
I_L, I_S = 14, 21


def _case(name, call, H, W, k, K, psf, B, draw, sigma, gain):
    c = {"call": call, "H": H, "W": W, "k": k, "K": K, "psf": psf, "B": B, "draw": draw, "sigma": sigma, "gain": gain}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a single evaluation of the smallest image of the serving stream: launches and latency only
        _case("one-40-b1", "grad", 40, 40, 2, 11, "gaussian", 1, "mode", 0.01, 1000.0),
        # one leapfrog step of the paper's 50 HMC chains on its 80 x 80 system
        _case("chains-80-b50", "graph", 80, 80, 2, 11, "gaussian", 50, "mode", 0.2, 100.0),
        # one iteration of the paper's variational inference: 500 draws around the mode
        _case("draws-80-b500", "autograd", 80, 80, 2, 11, "gaussian", 500, "mode", 0.2, 100.0),
        # one iteration of the paper's multi-start MAP: 300 starts from its prior (long and short series mixed)
        _case("starts-80-b300", "autograd", 80, 80, 2, 11, "gaussian", 300, "prior", 0.2, 100.0),
        # the benchmark's multi-start batch
        _case("multistart-60-b4096", "autograd", 60, 60, 2, 11, "gaussian", 4096, "box", 0.01, 1000.0),
        # 512 HMC chains on the benchmark's 100 x 100 system: a PSF with no separable form
        _case("hmc-100-k4-b512", "grad", 100, 100, 4, 21, "moffat", 512, "mode", 0.01, 1000.0),
        # the benchmark's largest image, a sixteenth of its batch
        _case("stress-200-k4-b1024", "grad", 200, 200, 4, 21, "gaussian", 1024, "box", 0.01, 1000.0),
        # odd sizes: an oblong cut-out, odd supersampling, a PSF side with no kernel of its own
        _case("ragged-61x59-k3-b200", "autograd", 61, 59, 3, 13, "moffat", 200, "box", 0.01, 1000.0),
        # log L alone: ranking many candidate starts before an optimisation
        _case("loglik-80-b2000", "loglik", 80, 80, 2, 11, "gaussian", 2000, "prior", 0.2, 100.0),
        # posterior-predictive images
        _case("simulate-80-b256", "simulate", 80, 80, 2, 11, "moffat", 256, "mode", 0.2, 100.0),
        # starts with the two amplitudes solved in closed form
        _case("profiled-80-b300", "profiled", 80, 80, 2, 11, "gaussian", 300, "box", 0.2, 100.0),
        # requests of four lenses of different shapes evaluated together, as a serving batch is
        _case("grouped-4-b320", "grouped", 60, 60, 2, 11, "gaussian", 320, "box", 0.01, 1000.0),
    ]


# the largest listed case's rays; drawn cases stay below half of it
MAX_RAYS = 1024 * (200 * 4) ** 2


def draw(rng):
    call = rng.choice(["grad", "autograd", "graph", "grad", "autograd", "loglik", "simulate", "profiled"])
    H = round(math.exp(rng.uniform(math.log(24), math.log(200))))
    W = H if rng.random() < 0.6 else max(16, min(200, round(H * rng.uniform(0.7, 1.4))))
    k = rng.choice([1, 2, 2, 2, 3, 4, 4])
    K = rng.choice([11, 11, 11, 21, 21, 5, 9, 13, 17])
    psf = rng.choice(["gaussian", "gaussian", "moffat"])
    most = min(4096, MAX_RAYS // (2 * H * W * k * k))
    if call == "simulate":
        most = min(most, 4_000_000 // (H * W))
    if call in ("graph", "profiled"):
        most = min(most, 512)
    B = max(1, round(math.exp(rng.uniform(0.0, math.log(max(2, most))))))
    how = rng.choice(["mode", "box", "prior"])
    sigma, gain = (0.2, 100.0) if how == "prior" or call == "profiled" or rng.random() < 0.4 else (0.01, 1000.0)
    return _case(None, call, H, W, k, K, psf, B, how, sigma, gain)


# ------------------------------------------------------- inputs of a case ----

def _spec(case, **over):
    c = dict(case, **over)
    return inputs.SystemSpec(c["H"], c["W"], c["k"], c["K"], c["psf"], inputs.PIXEL_SCALE, c["sigma"], c["gain"])


def _specs(case):
    """The systems of a case with their vector counts: four for a grouped call, else one."""
    if case["call"] != "grouped":
        return [(_spec(case), case["B"])]
    B = case["B"]
    return [(_spec(case), B), (_spec(case, H=40, W=40, k=4), B), (_spec(case, H=80, W=80, K=21), B // 2),
            (_spec(case, H=50, W=70, k=1, K=9, psf="moffat"), B)]


def _problem(spec, case, B, seed):
    """(image float32 [H, W], PSF float32 [K, K], parameters float32 [B, 22]) from the seed alone."""
    rng = np.random.default_rng(seed)
    paper = case["draw"] == "prior" or case["sigma"] > 0.1
    truth = inputs.draw_table(rng, inputs.PAPER_SIM, 1)[0] if paper else inputs.draw_truth(rng)
    psf = inputs.make_psf(spec).astype(np.float32)
    model = _images(torch.from_numpy(truth).cuda()[None], spec, torch.from_numpy(psf).cuda().double())[0]
    image = inputs.add_noise(rng, model.cpu().numpy(), spec.sigma_bkg, spec.gain_exposure).astype(np.float32)
    if case["draw"] == "prior":
        params = inputs.draw_table(rng, inputs.PAPER_PRIOR_DRAW, B)
    elif case["draw"] == "box":
        params = inputs.draw_box(rng, B)
    else:   # around the mode
        params = inputs.draw_perturbed(rng, truth, B)
    return image, psf, params.astype(np.float32)


def _problems(case, seed):
    return [(spec, *_problem(spec, case, B, 1_000_003 * i + seed)) for i, (spec, B) in enumerate(_specs(case))]


def prepare(case, seed):
    state = {"call": case["call"], "systems": [], "params": []}
    for spec, image, psf, params in _problems(case, seed):
        s = abi.GLSystem(image, psf, spec.pixel_scale, spec.k, spec.gain_exposure, sigma_bkg=spec.sigma_bkg,
                         observed_variance=case["call"] == "profiled")
        s.reserve(len(params))
        state["systems"].append(s)
        p = torch.from_numpy(params).cuda()
        state["params"].append(p.requires_grad_() if case["call"] == "autograd" else p)
    if case["call"] == "graph":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _grad(state["systems"][0], state["params"][0])
        torch.cuda.current_stream().wait_stream(side)
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            state["out"] = _grad(state["systems"][0], state["params"][0])
    return state


def _grad(system, params):
    ll, g = system.loglik_grad(params)
    return ll.to(params.dtype), g.to(params.dtype)


def run(state):
    call, system, params = state["call"], state["systems"][0], state["params"][0]
    if call == "grad":
        return _grad(system, params)
    if call == "graph":
        state["graph"].replay()
        return state["out"]
    if call == "autograd":
        ll = hmc.loglik(params, system)
        return ll.detach(), torch.autograd.grad(ll.sum(), params)[0]
    if call == "loglik":
        return hmc.loglik(params, system)
    if call == "simulate":
        return system.simulate(params)
    if call == "profiled":
        ll, g, amps = system.loglik_grad_profiled(params)
        return ll.to(params.dtype), g.to(params.dtype), amps.to(params.dtype)
    lls, grads, _ = abi.loglik_grad_grouped(state["systems"], state["params"])
    return [ll.to(torch.float32) for ll in lls], [g.to(torch.float32) for g in grads]


# --------------------------------------------------------------- the work ----

def work(case):
    """Per ray: the deflection (its power and the lens equation, about 50 operations, and two multiply-adds per
    term for about 8 series terms) and two Sersic profiles (18 operations each); a gradient in reverse takes about
    twice that again. Per pixel: the PSF's K^2 (2 K where separable) multiply-adds, twice with the gradient."""
    bytes_, flops = 0.0, 0.0
    for spec, B in _specs(case):
        px = float(B) * spec.H * spec.W
        ray = 50 + 2 * 2 * 8 + 2 * 18
        taps = 2 * (2 * spec.K if spec.psf == "gaussian" else spec.K ** 2)
        both = 2 if case["call"] not in ("loglik", "simulate") else 1
        flops += px * (spec.k ** 2 * ray * (3 if both == 2 else 1) + taps * both + 20)
        out = px * 4 if case["call"] == "simulate" else B * 4.0 * (1 + (NPARAM if both == 2 else 0))
        bytes_ += B * NPARAM * 4.0 + 2 * spec.H * spec.W * 4.0 + out
    return {"bytes": bytes_, "flops": flops}


# --------------------------------------------- the model in 64 bits (torch) ----

def _sersic(x, y, l):
    """Elliptical Sersic at (x, y); l: seven parameters (R, n, e1, e2, xc, yc, I), each [b, 1, 1]."""
    R, n, e1, e2, xc, yc, I0 = l
    dx, dy = x - xc, y - yc
    e = e1 * e1 + e2 * e2
    rho2 = ((1 + e) * (dx * dx + dy * dy) - 2 * e1 * (dx * dx - dy * dy) - 4 * e2 * dx * dy) / (1 - e)
    rho2 = torch.clamp(rho2, min=1e-12)
    return I0 * torch.exp(-(1.9992 * n - 0.3271) * (torch.exp(torch.log(rho2 / (R * R)) / (2 * n)) - 1))


def _deflection(x, y, m, terms):
    """EPL deflection: Tessore & Metcalf's angular series in the image frame, as complex numbers."""
    thE, gamma, e1, e2, xc, yc = m
    t = gamma - 1
    z = torch.complex(x - xc, y - yc)
    eps = torch.complex(e1, e2)
    w = z - eps * z.conj()
    rho2 = (w.real ** 2 + w.imag ** 2) / (1 - e1 * e1 - e2 * e2)
    inside = rho2 < 1e-12
    rho2 = torch.where(inside, torch.ones_like(rho2), rho2)
    w = torch.where(inside, torch.ones_like(w), w)
    u = -eps.conj() * w / w.conj()
    s = torch.ones_like(u)
    for n in range(terms, 0, -1):
        s = 1 + u * s * ((2 * n - 2 + t) / (2 * n + 2 - t))
    a = torch.exp(t * (torch.log(thE) - torch.log(rho2) / 2)) * w * s
    a = torch.where(inside, torch.zeros_like(a), a)
    return a.real, a.imag


def _images(p, spec, psf, parts=False):
    """PSF-convolved images [b, H, W] of the rows of p (float64); with parts, both lights apart."""
    H, W, k = spec.H, spec.W, spec.k
    h = spec.pixel_scale / k
    y = ((torch.arange(H * k, device=p.device, dtype=torch.float64) - (H * k - 1) / 2) * h)[:, None]
    x = ((torch.arange(W * k, device=p.device, dtype=torch.float64) - (W * k - 1) / 2) * h)[None, :]
    q = [c[:, None, None] for c in p.unbind(1)]
    f = min(0.9, float(p.detach()[:, 2:4].norm(dim=1).max()))
    terms = 2 if f < 1e-17 else min(400, int(math.ceil(-40 / math.log(f))) + 2)
    ax, ay = _deflection(x, y, q[:6], terms)
    bx = x - ax - q[6] * x - q[7] * y
    by = y - ay - q[7] * x + q[6] * y
    light, source = _sersic(x, y, q[8:15]), _sersic(bx, by, q[15:22])
    out = []
    for I in ([light, source] if parts else [light + source]):
        I = I.reshape(-1, H, k, W, k).mean((2, 4)) * spec.pixel_scale ** 2
        out.append(F.conv2d(I[:, None], psf.flip(0, 1)[None, None], padding=psf.shape[0] // 2)[:, 0])
    return out if parts else out[0]


def _loglik(p, spec, image, psf, profiled):
    """log L [b], and the solved amplitudes [b, 2] (None without profiling)."""
    inv = 1.0 / spec.gain_exposure
    s2 = float(np.float32(spec.sigma_bkg)) ** 2
    amps = None
    if profiled:
        v = s2 + image.clamp(min=0) * inv
        ones = torch.ones_like(p[:, :1])
        unit = torch.cat([p[:, :I_L], ones, p[:, I_L + 1:I_S], ones], 1)
        light, source = _images(unit, spec, psf, parts=True)
        with torch.no_grad():
            dot = lambda a, b: (a * b / v).sum((1, 2))  # noqa: E731
            ll_, ls, ss, dl, ds = (dot(light, light), dot(light, source), dot(source, source), dot(light, image),
                                   dot(source, image))
            det = ll_ * ss - ls * ls
            amps = torch.stack([(ss * dl - ls * ds) / det, (ll_ * ds - ls * dl) / det], 1)
        model = amps[:, 0, None, None] * light + amps[:, 1, None, None] * source
    else:
        model = _images(p, spec, psf)
        v = s2 + model * inv
    res = image - model
    return -0.5 * (res * res / v + torch.log(2 * math.pi * v)).sum((1, 2)), amps


def exact(case, seed):
    lls, grads, amps, images = [], [], [], []
    for spec, image, psf, params in _problems(case, seed):
        image, psf = torch.from_numpy(image).cuda().double(), torch.from_numpy(psf).cuda().double()
        p = torch.from_numpy(params).cuda().double()
        rays = spec.H * spec.W * spec.k ** 2
        step = max(1, int((1 << 20 if case["draw"] != "prior" else 1 << 18) / rays))
        ll, g, am, im = [], [], [], []
        # by the length of the series, so that few vectors set the number of terms of the others
        order = p[:, 2:4].norm(dim=1).argsort()
        for rows in order.split(step):
            if case["call"] == "simulate":
                im.append(_images(p[rows], spec, psf))
            elif case["call"] == "loglik":
                ll.append(_loglik(p[rows], spec, image, psf, False)[0])
            else:
                q = p[rows].requires_grad_()
                l, a = _loglik(q, spec, image, psf, case["call"] == "profiled")
                g.append(torch.autograd.grad(l.sum(), q)[0])
                ll.append(l.detach())
                am.append(a)
        back = order.argsort()
        if im:
            images.append(torch.cat(im)[back])
        if ll:
            lls.append(torch.cat(ll)[back])
        if g:
            grads.append(torch.cat(g)[back])
        if am and am[0] is not None:
            amps.append(torch.cat(am)[back])
    if case["call"] == "grouped":
        return lls, grads
    if case["call"] == "simulate":
        return images[0]
    if case["call"] == "loglik":
        return lls[0]
    return (lls[0], grads[0], amps[0]) if amps else (lls[0], grads[0])
