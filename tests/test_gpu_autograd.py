"""Differentiable F(c), theta(c) through torch.autograd (needs a GB300).

g(x) = exp(i sum_a c_a(x) lambda_a).  The reference values come from the oracle's F and
theta (Eqs. (1)-(3)) of the field transformed on the CPU; gradients are checked against
central finite differences of that oracle forward (float64, h = 1e-6) and, at c = 0,
against the analytic gradient Tr[lambda_a Delta] / (2i nd Nc V).
"""
import numpy as np
import pytest

import oracle
from paper_1412_1498_gb300 import fields

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gf():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1412_1498_gb300 import build
    build.build()
    from paper_1412_1498_gb300 import gf as m
    return m


def oracle_F_theta(U, c, gauge):
    # g = exp(i c.lambda) by scipy's matrix exponential (batched over the sites)
    from scipy.linalg import expm
    Lt, Lz, Ly, Lx = U.shape[:4]
    X = np.einsum("...a,aij->...ij", c.reshape(Lt, Lz, Ly, Lx, 8), fields.gell_mann())
    W = fields.gauge_transform(U, expm(1j * X))
    F, th, _, _ = oracle.measure(W, gauge)
    return F, th


def make(gf, dims, gauge, U):
    fx = gf.GaugeFixer(dims, gauge, gf.GF_FP64_18, autograd=True)
    fx.upload(U)
    return fx


@pytest.mark.parametrize("gauge", [0, 1])
def test_forward_matches_oracle(gf, gauge):
    from paper_1412_1498_gb300.autograd import functional_theta
    dims = (4, 4, 4, 6)
    V = int(np.prod(dims))
    U = fields.random_gauge_config(dims, 0.5, 100)
    c = np.random.default_rng(1).normal(scale=0.3, size=(V, 8))
    fx = make(gf, dims, gauge, U)
    F, th = functional_theta(torch.from_numpy(c).cuda(), fx)
    rF, rth = oracle_F_theta(U, c, gauge)
    assert abs(F.item() - rF) < 1e-12 * abs(rF) and abs(th.item() - rth) < 1e-12 * rth
    fx.close()


@pytest.mark.parametrize("gauge", [0, 1])
def test_gradient_at_zero_is_delta(gf, gauge):
    from paper_1412_1498_gb300.autograd import functional_theta
    dims = (4, 4, 6, 4)
    V = int(np.prod(dims))
    nd = 4 if gauge == 0 else 3
    U = fields.random_gauge_config(dims, 0.5, 101)
    fx = make(gf, dims, gauge, U)
    c = torch.zeros((V, 8), dtype=torch.float64, device="cuda", requires_grad=True)
    F, th = functional_theta(c, fx)
    F.backward()
    D = oracle.delta(U, gauge).reshape(V, 3, 3)
    want = (np.einsum("aij,sji->sa", fields.gell_mann(), D) / (2j * nd * 3 * V)).real
    got = c.grad.cpu().numpy()
    assert np.abs(got - want).max() < 1e-12 * np.abs(want).max()
    fx.close()


@pytest.mark.parametrize("gauge", [0, 1])
def test_gradients_match_central_differences(gf, gauge):
    from paper_1412_1498_gb300.autograd import functional_theta
    dims = (4, 4, 4, 4)
    V = int(np.prod(dims))
    U = fields.random_gauge_config(dims, 0.5, 102)
    rng = np.random.default_rng(2)
    c0 = rng.normal(scale=0.2, size=(V, 8))
    fx = make(gf, dims, gauge, U)
    grads = []
    for which in (0, 1):
        c = torch.from_numpy(c0.copy()).cuda().requires_grad_(True)
        out = functional_theta(c, fx)
        out[which].backward()
        grads.append(c.grad.cpu().numpy())
    h = 1e-6
    for _ in range(12):
        s, a = int(rng.integers(V)), int(rng.integers(8))
        cp, cm = c0.copy(), c0.copy()
        cp[s, a] += h
        cm[s, a] -= h
        fp, tp = oracle_F_theta(U, cp, gauge)
        fm, tm = oracle_F_theta(U, cm, gauge)
        for which, (vp, vm) in enumerate(((fp, fm), (tp, tm))):
            fd = (vp - vm) / (2 * h)
            scale = np.abs(grads[which]).max()
            assert abs(grads[which][s, a] - fd) < 1e-6 * scale, (which, s, a, grads[which][s, a], fd)
    fx.close()


def test_sgd_first_step_is_naive_descent_and_50_steps_ascend(gf):
    # loss = -F, lr = alpha nd Nc V / 2: the first SGD step from c = 0 is g = exp((alpha/2)
    # Delta), the naive steepest-descent step of Eq. (7) with the exact exponential
    from paper_1412_1498_gb300.autograd import functional_theta
    dims = (8, 8, 8, 8)
    V = int(np.prod(dims))
    alpha = 0.08
    U = fields.random_gauge_config(dims, 0.4, 1, 2)
    fx = make(gf, dims, 0, U)
    c = torch.zeros((V, 8), dtype=torch.float64, device="cuda", requires_grad=True)
    opt = torch.optim.SGD([c], lr=alpha * 4 * 3 * V / 2)
    hist = []
    for step in range(50):
        opt.zero_grad()
        F, th = functional_theta(c, fx)
        hist.append((F.item(), th.item()))
        (-F).backward()
        opt.step()
        if step == 0:
            D = oracle.delta(U).reshape(dims[::-1] + (3, 3))
            from scipy.linalg import expm
            W = fields.gauge_transform(U, expm(0.5 * alpha * D))     # Eq. (7): g = exp(alpha/2 Delta)
            F1, th1 = oracle_F_theta(U, c.detach().cpu().numpy(), 0)
            assert abs(F1 - oracle.measure(W)[0]) < 1e-12
    F, th = functional_theta(c, fx)
    hist.append((F.item(), th.item()))
    Fs = np.array([h[0] for h in hist])
    assert np.all(np.diff(Fs) > -1e-13) and Fs[-1] > Fs[0]
    assert hist[-1][1] < hist[0][1]
    fx.close()


@pytest.mark.parametrize("gauge", [0, 1])
def test_slabs_equal_the_whole(gf, gauge):
    # 32 x 32 x 64 x 256 sites are above the link buffer (8 GiB), so the passes run in slabs of
    # time slices (226 and 30).  The field repeats an 8 x 8 x 8 x 16 one: F, theta are its, and the
    # gradient is its over the number of copies.  Sums of equal terms in FP64: 1e-12.
    from paper_1412_1498_gb300.autograd import functional_theta
    small, reps = (8, 8, 8, 16), (4, 4, 8, 16)
    big = tuple(n * r for n, r in zip(small, reps))
    U = torch.from_numpy(fields.random_gauge_config(small, 0.5, 103)).cuda()
    c = torch.from_numpy(np.random.default_rng(4).normal(scale=0.3, size=small[::-1] + (8,))).cuda()
    res = []
    for dims, r in ((small, (1, 1, 1, 1)), (big, reps)):
        fx = gf.GaugeFixer(dims, gauge, gf.GF_FP64_18, autograd=True)
        fx.upload(U.repeat(*r[::-1], 1, 1, 1))
        p = c.repeat(*r[::-1], 1).reshape(-1, 8).contiguous().requires_grad_(True)
        F, th = functional_theta(p, fx)
        (g,) = torch.autograd.grad(0.3 * th - F, p)
        res.append((F.item(), th.item(), g.reshape(dims[::-1] + (8,)) * float(np.prod(r))))
        fx.close()
        del fx, p
    (F0, t0, g0), (F1, t1, g1) = res
    assert abs(F1 - F0) < 1e-12 * abs(F0) + 1e-15 and abs(t1 - t0) < 1e-12 * t0
    assert float((g1 - g0.repeat(*reps[::-1], 1)).abs().max()) < 1e-12 * float(g0.abs().max())


def _exp_frechet(X, E=None):
    # exp(iX) of Hermitian X and the derivative of exp(i .) in the direction E, from the
    # eigenvalues (Daleckii-Krein; the divided differences i exp(i (a + b) / 2) sinc((a - b) / 2) have
    # no cancellation): errors of a rounding times the spectral radius
    lam, V = np.linalg.eigh(X)
    Vh = V.conj().swapaxes(-1, -2)
    if E is None:
        return (V * np.exp(1j * lam)[..., None, :]) @ Vh
    a, b = lam[..., :, None], lam[..., None, :]
    phi = 1j * np.exp(0.5j * (a + b)) * np.sinc((a - b) / (2 * np.pi))
    return V @ ((Vh @ E @ V) * phi) @ Vh


@pytest.mark.parametrize("along", ["lambda_8", "nearly", "random"])
@pytest.mark.parametrize("radius", [0.3, 3.0, 7.5, 20.0, 200.0, 2000.0])
def test_gradient_at_large_parameters(gf, radius, along):
    # zero to eleven squarings of the exponential, with equal, nearly equal and other eigenvalues.
    # Squaring a unitary matrix doubles its relative error, which after log2(radius) squarings is
    # radius * 2^-52 times a few operations' errors on either side: 50 radius 2^-52 (radius >= 4)
    from paper_1412_1498_gb300.autograd import functional_theta
    dims = (2, 2, 4, 2)
    lat = dims[::-1]
    rng = np.random.default_rng(8)
    c = rng.normal(size=lat + (8,))
    if along != "random":
        c[..., :7] *= 0.0 if along == "lambda_8" else 1e-7
        c[..., 7] = np.where(c[..., 7] < 0, -1.0, 1.0) * (0.5 + 0.5 * rng.random(lat))
    X = np.einsum("...a,aij->...ij", c, fields.gell_mann())
    scale = radius / np.abs(np.linalg.eigvalsh(X)).max()
    c, X = c * scale, X * scale
    U = fields.random_gauge_config(dims, 0.5, 7)
    g = torch.from_numpy(_exp_frechet(X)).requires_grad_(True)
    Ut = torch.from_numpy(U)
    step = lambda f, mu, n: torch.roll(f, -n, dims=3 - mu)
    W = [g @ Ut[..., mu, :, :] @ step(g, mu, 1).mH for mu in range(4)]
    D = sum(step(w, mu, -1) - w for mu, w in enumerate(W))
    D = D - D.mH
    D = D - D.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3 * torch.eye(3)
    n = float(np.prod(dims))
    F = sum(w.diagonal(dim1=-2, dim2=-1).real.sum() for w in W) / (12 * n)
    th = (D.abs() ** 2).sum() / (3 * n)
    (G,) = torch.autograd.grad(0.3 * th - F, g)      # dL = Re sum conj(G) dg = Re Tr[E dg]
    L = _exp_frechet(X, G.numpy().conj().swapaxes(-1, -2))
    want = np.einsum("aij,...ji->...a", fields.gell_mann(), L).real.reshape(-1, 8)
    fx = make(gf, dims, 0, U)
    p = torch.from_numpy(c.reshape(-1, 8)).cuda().requires_grad_(True)
    Fg, tg = functional_theta(p, fx)
    (got,) = torch.autograd.grad(0.3 * tg - Fg, p)
    fx.close()
    tol = 50 * max(radius, 4.0) * 2.0 ** -52
    assert abs(Fg.item() - F.item()) < tol and abs(tg.item() - th.item()) < tol * th.item()
    assert np.abs(got.cpu().numpy() - want).max() < tol * np.abs(want).max()


@pytest.mark.parametrize("gauge", [0, 1])
def test_without_a_link_buffer_equals_the_small_field(gf, gauge):
    # two time slices of 208^3 sites: no link buffer (see test_slabs_equal_the_whole for the rest)
    from paper_1412_1498_gb300.autograd import functional_theta
    small, n = (8, 8, 8, 2), 26
    big = tuple(n * v for v in small[:3]) + (2,)
    U = torch.from_numpy(fields.random_gauge_config(small, 0.5, 104)).cuda()
    c = torch.from_numpy(np.random.default_rng(5).normal(scale=0.3, size=small[::-1] + (8,))).cuda()
    res = []
    for dims, r in ((small, 1), (big, n)):
        fx = gf.GaugeFixer(dims, gauge, gf.GF_FP64_18, autograd=True)
        fx.upload(U.repeat(1, r, r, r, 1, 1, 1))
        p = c.repeat(1, r, r, r, 1).reshape(-1, 8).contiguous().requires_grad_(True)
        F, th = functional_theta(p, fx)
        (g,) = torch.autograd.grad(0.3 * th - F, p)
        res.append((F.item(), th.item(), g.reshape(dims[::-1] + (8,)) * float(r) ** 3))
        fx.close()
        del fx, p
    (F0, t0, g0), (F1, t1, g1) = res
    assert abs(F1 - F0) < 1e-12 * abs(F0) + 1e-15 and abs(t1 - t0) < 1e-12 * t0
    assert float((g1 - g0.repeat(1, n, n, n, 1)).abs().max()) < 1e-12 * float(g0.abs().max())
