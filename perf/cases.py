"""Performance cases of the gauge-fixing library, through its public entry points.

Every case is a call sequence that a user's program makes: hand a configuration to a
handle that the program keeps, fix it (overrelaxation, Fourier-accelerated steepest
descent, or the double-float polish of a mixed run), take the links back with F and theta;
or differentiate F and theta by the gauge transformation's parameters.  Runs take a budget
of sweeps and a stop threshold that is never met, as a production run does between two
looks at its field: the work of a pass does not depend on rounding.

Configurations are U_mu(x) = exp(i eps A_mu(x)) (A with N(0, 1) coefficients on the
Gell-Mann matrices), rotated by a random gauge transformation: the recipe of
``paper_1412_1498_gb300.fields``, drawn on the GPU.  The transformation is Haar-random for
FP64 storage (a raw configuration) and moderate for FP32 storage (a run some sweeps in,
where it spends nearly all its time; the first sweeps of a raw one pass sites where K is
nearly singular, whose update no single precision determines).  The polish takes a field
that is close to its maximum, as the FP32 phase leaves it (A projected to its transverse
part).

Links of FP32 storages come back rounded to complex64 and their F, theta as float32: that
is the precision those storages hold.  So does the polish's theta: its updates g - 1 are
formed to FP32 relative precision, and theta is what they leave.
"""
from __future__ import annotations

import math

import torch

from paper_1412_1498_gb300 import gf
from paper_1412_1498_gb300.autograd import functional_theta

DEVICE = "cuda"
OMEGA = 1.7          # the library's default overrelaxation parameter
REUNIT = 20          # and its default reunitarisation interval
ALPHA = 0.08         # and its default step of Fourier acceleration
NEVER = 1e-300       # a stop threshold below every theta

STORAGE = {"fp64_18": gf.GF_FP64_18, "fp32_18": gf.GF_FP32_18, "fp32_12": gf.GF_FP32_12, "fp64_12": gf.GF_FP64_12}
LINK_BYTES = {"fp64_18": 144, "fp32_18": 72, "fp32_12": 48, "fp64_12": 96}


# ------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------
def _fix(dims, storage, sweeps, gauge="landau", **more):
    return dict(kind="fix", Lx=dims[0], Ly=dims[1], Lz=dims[2], Lt=dims[3], gauge=gauge, storage=storage, sweeps=sweeps, **more)


def listed():
    return [
        # the smallest lattice of the tests and golden runs: every launch and the host's part count
        dict(_fix((8, 8, 8, 8), "fp32_12", 24), name="fix_8x4_fp32_12"),
        # an anisotropic lattice whose slices do not fill whole blocks; fits in L2
        dict(_fix((20, 12, 18, 10), "fp32_12", 20), name="fix_20x12x18x10_fp32_12"),
        # the benchmark's lattice in its default storage: larger than L2
        dict(_fix((32, 32, 32, 32), "fp32_12", 20), name="fix_32x4_fp32_12"),
        # Coulomb gauge: 64 time slices, each a convergence unit of its own
        dict(_fix((32, 32, 32, 64), "fp32_12", 20, "coulomb"), name="fix_coulomb_32x3x64_fp32_12"),
        # an ensemble of configurations of three extents fixed together in one handle
        dict(kind="batch", count=16, sweeps=20, name="fix_ensemble_48_fp32_12"),
        # the paper's double-precision run, held in full matrices
        dict(_fix((16, 16, 16, 16), "fp64_18", 40), name="fix_16x4_fp64_18"),
        # FP32 with full matrices
        dict(_fix((24, 24, 24, 24), "fp32_18", 20), name="fix_24x4_fp32_18"),
        # the second phase of a mixed run to theta < 1e-15: double-float sweeps near the maximum
        dict(kind="polish", Lx=24, Ly=24, Lz=24, Lt=24, sweeps=32, name="polish_24x4"),
        # Fourier-accelerated steepest descent on the benchmark's lattice
        dict(kind="fasd", Lx=32, Ly=32, Lz=32, Lt=32, gauge="landau", storage="fp32_12", sweeps=16, name="fasd_32x4_fp32_12"),
        # the same per time slice and in double precision
        dict(kind="fasd", Lx=16, Ly=16, Lz=16, Lt=32, gauge="coulomb", storage="fp64_18", sweeps=8, name="fasd_coulomb_16x3x32_fp64_18"),
        # one training step's F, theta and gradient in the transformation's parameters
        dict(kind="autograd", Lx=32, Ly=32, Lz=32, Lt=32, gauge="landau", name="autograd_32x4"),
        # a configuration read from and written back to pinned host memory, with a few sweeps
        dict(kind="host", Lx=24, Ly=24, Lz=24, Lt=24, sweeps=4, name="host_24x4_fp64_18"),
    ]


def _even_dims(rng, lo, hi):
    """Even extents with a volume between lo and hi sites, spread over its logarithm."""
    side = math.exp(rng.uniform(math.log(lo), math.log(hi))) ** 0.25
    while True:
        d = [max(2, 2 * round(side * math.exp(rng.uniform(-0.5, 0.5)) / 2)) for _ in range(4)]
        if lo <= math.prod(d) <= hi:
            return d


def draw(rng):
    kind = rng.choice(["fix", "fix", "fix", "fix64", "batch", "polish", "fasd", "fasd", "autograd", "host"])
    gauge = rng.choice(["landau", "coulomb"])
    if kind == "fix":
        return _fix(_even_dims(rng, 1 << 10, 1 << 21), rng.choice(["fp32_12", "fp32_12", "fp32_18"]), rng.randint(10, 20), gauge)
    if kind == "fix64":
        return _fix(_even_dims(rng, 1 << 10, 1 << 18), rng.choice(["fp64_18", "fp64_18", "fp64_12"]), rng.randint(8, 20), gauge)
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 12), sweeps=rng.randint(10, 20))
    if kind == "fasd":
        storage = rng.choice(["fp32_12", "fp64_18"])
        top = 1 << (20 if storage == "fp32_12" else 18)
        while True:
            d = [2 ** rng.randint(2, 5) for _ in range(3)] + [2 * rng.randint(2, 16) if gauge == "coulomb" else 2 ** rng.randint(2, 5)]
            if math.prod(d) <= top:
                break
        return dict(kind="fasd", Lx=d[0], Ly=d[1], Lz=d[2], Lt=d[3], gauge=gauge, storage=storage, sweeps=rng.randint(4, 16))
    if kind == "polish":
        d = _even_dims(rng, 1 << 12, 1 << 19)
        return dict(kind="polish", Lx=d[0], Ly=d[1], Lz=d[2], Lt=d[3], sweeps=rng.randint(10, 32))
    d = _even_dims(rng, 1 << 10, 1 << 19)
    if kind == "autograd":
        return dict(kind="autograd", Lx=d[0], Ly=d[1], Lz=d[2], Lt=d[3], gauge=gauge)
    return dict(kind="host", Lx=d[0], Ly=d[1], Lz=d[2], Lt=d[3], sweeps=rng.randint(1, 4))


def _dims(case):
    return (case["Lx"], case["Ly"], case["Lz"], case["Lt"])


def _dims_list(case):
    """Extents of a case's lattices (the benchmark's ensemble for a batch)."""
    if case["kind"] == "batch":
        return [(16, 16, 16, 16)] * case["count"] + [(24, 24, 24, 24)] * case["count"] + [(16, 16, 16, 32)] * case["count"]
    return [_dims(case)]


def _storage(case):
    return {"fix": case.get("storage"), "fasd": case.get("storage"), "batch": "fp32_12", "polish": "fp32_12",
            "autograd": "fp64_18", "host": "fp64_18"}[case["kind"]]


def _nd(case):
    return 3 if case.get("gauge") == "coulomb" else 4


# ------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------
def _mm(a, b):
    """a b for stacks of 3 x 3 matrices."""
    return a[..., :, 0:1] * b[..., 0:1, :] + a[..., :, 1:2] * b[..., 1:2, :] + a[..., :, 2:3] * b[..., 2:3, :]


def _dag(a):
    return a.mH


def _reunit(U):
    """Gram-Schmidt on rows 0, 1; row 2 = conj(row 0 x row 1)."""
    r0 = U[..., 0, :]
    r0 = r0 / (r0.abs() ** 2).sum(-1, keepdim=True).sqrt()
    r1 = U[..., 1, :]
    r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / (r1.abs() ** 2).sum(-1, keepdim=True).sqrt()
    return torch.stack([r0, r1, _cross(r0, r1)], dim=-2)


def _cross(r0, r1):
    return torch.stack([r0[..., 1] * r1[..., 2] - r0[..., 2] * r1[..., 1],
                        r0[..., 2] * r1[..., 0] - r0[..., 0] * r1[..., 2],
                        r0[..., 0] * r1[..., 1] - r0[..., 1] * r1[..., 0]], dim=-1).conj()


def _hermitian(c):
    """sum_a c_a lambda_a over the last axis (Gell-Mann matrices), traceless Hermitian."""
    s3 = 1.0 / math.sqrt(3.0)
    z = torch.zeros_like(c[..., 0])
    X = [torch.complex(c[..., 2] + s3 * c[..., 7], z), torch.complex(c[..., 0], -c[..., 1]), torch.complex(c[..., 3], -c[..., 4]),
         torch.complex(c[..., 0], c[..., 1]), torch.complex(-c[..., 2] + s3 * c[..., 7], z), torch.complex(c[..., 5], -c[..., 6]),
         torch.complex(c[..., 3], c[..., 4]), torch.complex(c[..., 5], c[..., 6]), torch.complex(-2 * s3 * c[..., 7], z)]
    return torch.stack(X, dim=-1).unflatten(-1, (3, 3))


def _exp_i(c, eps):
    """exp(i eps sum_a c_a lambda_a): Taylor series of the eighth part, squared three times."""
    Y = _hermitian(c) * (1j * eps / 8)
    one = torch.eye(3, dtype=Y.dtype, device=Y.device)
    E = one + Y / 12
    for k in range(11, 0, -1):
        E = one + _mm(Y, E) / k
    for _ in range(3):
        E = _mm(E, E)
    return _reunit(E)


def _step(f, mu, n):
    """f(x + n mu) of a field with axes (t, z, y, x, ...)."""
    return torch.roll(f, -n, dims=3 - mu)


def _transform(U, g):
    """g(x) U_mu(x) g(x + mu)^dagger."""
    return torch.stack([_mm(_mm(g, U[..., mu, :, :]), _dag(_step(g, mu, 1))) for mu in range(4)], dim=-3)


def _field(dims, seed, haar, eps=0.5):
    """A configuration in canonical layout (Lt, Lz, Ly, Lx, 4, 3, 3), complex128."""
    r = torch.Generator(device=DEVICE).manual_seed(seed)
    V = dims[::-1]
    U = _exp_i(torch.randn(*V, 4, 8, dtype=torch.float64, device=DEVICE, generator=r), eps)
    if haar:
        g = _reunit(torch.randn(*V, 3, 3, dtype=torch.complex128, device=DEVICE, generator=r))
    else:
        g = _exp_i(torch.randn(*V, 8, dtype=torch.float64, device=DEVICE, generator=r), 0.2)
    return _transform(U, g).contiguous()


def _near_field(dims, seed, eps=0.02):
    """A field close to the maximum of F: A with its longitudinal part removed, so that the
    divergence of Eq. (3) starts at third order in eps (theta of a few 1e-9, below the
    1e-8 at which a mixed run leaves its FP32 phase)."""
    r = torch.Generator(device=DEVICE).manual_seed(seed)
    V = dims[::-1]
    A = torch.randn(*V, 4, 8, dtype=torch.float64, device=DEVICE, generator=r)
    k = torch.fft.fftn(A, dim=(0, 1, 2, 3))
    d = []
    for mu in range(4):
        w = 1 - torch.exp(-2j * math.pi * torch.arange(dims[mu], device=DEVICE, dtype=torch.float64) / dims[mu])
        shape = [1] * 4
        shape[3 - mu] = dims[mu]
        d.append(w.reshape(shape).expand(V))
    d = torch.stack(d, dim=-1)[..., None]
    norm = (d.abs() ** 2).sum(-2, keepdim=True)
    k = k - d.conj() * (d * k).sum(-2, keepdim=True) / torch.where(norm > 1e-12, norm, 1.0)
    return _exp_i(torch.fft.ifftn(k, dim=(0, 1, 2, 3)).real, eps).contiguous()


def _inputs(case, seed):
    if case["kind"] == "polish":
        return [_near_field(_dims(case), seed)]
    haar = _storage(case).startswith("fp64")
    return [_field(d, seed * 64 + i, haar) for i, d in enumerate(_dims_list(case))]


def _parameters(case, seed):
    """Lie-algebra parameters of a transformation in the middle of a descent."""
    r = torch.Generator(device=DEVICE).manual_seed(seed * 64 + 63)
    return 0.3 * torch.randn(math.prod(_dims(case)), 8, dtype=torch.float64, device=DEVICE, generator=r)


def prepare(case, seed):
    kind, dims = case["kind"], _dims_list(case)
    fields = _inputs(case, seed)
    gauge = gf.GF_COULOMB if case.get("gauge") == "coulomb" else gf.GF_LANDAU
    fixer = gf.GaugeFixer(dims if kind == "batch" else dims[0], gauge, STORAGE[_storage(case)],
                          mixed=kind == "polish", fasd=kind == "fasd", autograd=kind == "autograd", device=DEVICE)
    state = dict(kind=kind, fixer=fixer, fields=fields, sweeps=case.get("sweeps", 0), single=_storage(case).startswith("fp32") and kind != "polish")
    if kind == "fasd":
        gf.gf_set_method(fixer.h, gf.GF_METHOD_FASD)
    if kind == "autograd":
        fixer.upload(fields[0])
        state["c"] = _parameters(case, seed).requires_grad_(True)
    elif kind == "host":
        state["fields"] = [f.cpu().pin_memory() for f in fields]
        state["out"] = [torch.empty_like(f, device="cpu").pin_memory() for f in fields]
    else:
        state["out"] = [torch.empty_like(f) for f in fields]
    return state


# ------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------
def run(state):
    fixer = state["fixer"]
    if state["kind"] == "autograd":
        F, theta = functional_theta(state["c"], fixer)
        (grad,) = torch.autograd.grad(0.1 * theta - F, state["c"])
        return {"F": F.detach(), "theta": theta.detach(), "grad": grad}
    for lat, U in enumerate(state["fields"]):
        fixer.upload(U, lat)
    r = fixer.fix(NEVER, state["sweeps"])
    links = [fixer.download(lat, out) for lat, out in enumerate(state["out"])]
    single = state["single"]
    return {"F": r["F"].astype("float32") if single else r["F"],
            "theta": r["theta"].astype("float32") if single or state["kind"] == "polish" else r["theta"],
            "iters": r["iters"],
            "links": [u.to(torch.complex64) for u in links] if single else links}


# ------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------
def work(case):
    """Bytes: the configuration in and the links out, and the stored links read and written
    once by each half-sweep (two of them a sweep; in Fourier acceleration read by Delta and
    read and written by the update).  Flops: a multiply-add counts two."""
    V = sum(math.prod(d) for d in _dims_list(case))
    kind, n = case["kind"], case.get("sweeps", 0)
    b = 144 if kind == "polish" else LINK_BYTES[_storage(case)]
    if kind == "autograd":
        # forward: links and parameters in; backward: the same and the gradient out.  g, the
        # four transformed links and Delta once per site, and the adjoint of each
        return {"bytes": V * (2 * 4 * 144 + 3 * 64), "flops": V * (600 + 4 * 2 * 216 + 8 * 216 + 900)}
    canonical = V * 4 * (2 * 144)
    if kind == "fasd":
        fft = 8 if _nd(case) == 4 else 6
        logs = sum(math.log2(L) for L in _dims(case)[: _nd(case)]) / _nd(case)
        return {"bytes": canonical + n * 12 * V * b, "flops": n * V * (8 * 216 + 8 * 18 + fft * 4 * 5 * logs)}
    # eight links times g, K and the three subgroup steps
    return {"bytes": canonical + n * 16 * V * b, "flops": n * V * (8 * 216 + 8 * 18 + 270)}


# ------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------
def _as_stored(U, storage):
    """The configuration as the storage holds it after an upload."""
    if storage.startswith("fp32"):
        U = U.to(torch.complex64).to(torch.complex128)
    if storage.endswith("12"):
        U = torch.stack([U[..., 0, :], U[..., 1, :], _cross(U[..., 0, :], U[..., 1, :])], dim=-2)
    return U


def _delta(U, nd):
    """Eq. (3): A - A^dagger without its trace, A = sum_nu U_nu(x - nu) - U_nu(x)."""
    A = sum(_step(U[..., nu, :, :], nu, -1) - U[..., nu, :, :] for nu in range(nd))
    D = A - _dag(A)
    tr = D.diagonal(dim1=-2, dim2=-1).sum(-1) / 3
    return D - tr[..., None, None] * torch.eye(3, dtype=D.dtype, device=D.device)


def _F_theta(U, nd):
    V = U.shape[0] * U.shape[1] * U.shape[2] * U.shape[3]
    F = U[..., :nd, :, :].diagonal(dim1=-2, dim2=-1).real.sum() / (nd * 3 * V)
    theta = (_delta(U, nd).abs() ** 2).sum() / (3 * V)
    return F, theta


def _parity(U):
    t, z, y, x = torch.meshgrid(*[torch.arange(n, device=U.device) for n in U.shape[:4]], indexing="ij")
    return (t + z + y + x) % 2


def _half_sweep(U, nd, sites):
    """Algorithm 1 on the sites of one parity: g from the three SU(2) subgroups, applied."""
    K = sum(U[..., mu, :, :] + _dag(_step(U[..., mu, :, :], mu, -1)) for mu in range(nd))
    K = list(K.flatten(-2).unbind(-1))
    G = [torch.full_like(K[0], float(e % 4 == 0)) for e in range(9)]
    for i, j in ((0, 1), (0, 2), (1, 2)):
        a = (K[4 * i] + K[4 * j].conj()).conj()
        b = (K[3 * j + i] - K[3 * i + j].conj()).conj()
        n = (a.abs() ** 2 + b.abs() ** 2).sqrt()
        a, b = 1 - OMEGA + OMEGA * a / n, OMEGA * b / n
        m = (a.abs() ** 2 + b.abs() ** 2).sqrt()
        a, b = a / m, b / m
        for M in (K, G):
            for c in range(3):
                mi, mj = M[3 * i + c], M[3 * j + c]
                M[3 * i + c], M[3 * j + c] = a * mi + b * mj, a.conj() * mj - b.conj() * mi
    g = torch.stack(G, dim=-1).unflatten(-1, (3, 3))
    return _transform(U, torch.where(sites[..., None, None], g, torch.eye(3, dtype=g.dtype, device=g.device)))


def _exact_fix(U, nd, sweeps):
    parity = _parity(U)
    for k in range(sweeps):
        U = _half_sweep(U, nd, parity == 0)
        U = _half_sweep(U, nd, parity == 1)
        if (k + 1) % REUNIT == 0:
            U = _reunit(U)
    return U


def _exact_fasd(U, nd, steps):
    axes = (0, 1, 2, 3) if nd == 4 else (1, 2, 3)
    p2 = 0
    for mu in range(nd):
        L = U.shape[3 - mu]
        shape = [1] * 4
        shape[3 - mu] = L
        p2 = p2 + (4 * torch.sin(math.pi * torch.arange(L, device=U.device, dtype=torch.float64) / L) ** 2).reshape(shape)
    factor = torch.where(p2 > 0, 0.5 * ALPHA * 4 * nd / torch.where(p2 > 0, p2, 1.0), 0.0)[..., None, None]
    one = torch.eye(3, dtype=U.dtype, device=U.device)
    for k in range(steps):
        d = torch.fft.ifftn(torch.fft.fftn(_delta(U, nd), dim=axes) * factor, dim=axes)
        U = _transform(U, _reunit(one + d))
        if (k + 1) % REUNIT == 0:
            U = _reunit(U)
    return U


def _exact_autograd(U, c, nd):
    c = c.requires_grad_(True)
    with torch.enable_grad():
        g = torch.linalg.matrix_exp(1j * _hermitian(c)).reshape(*U.shape[:4], 3, 3)
        F, theta = _F_theta(_transform(U, g), nd)
        (grad,) = torch.autograd.grad(0.1 * theta - F, c)
    return {"F": F.detach(), "theta": theta.detach(), "grad": grad}


def exact(case, seed):
    kind, nd = case["kind"], _nd(case)
    fields = _inputs(case, seed)
    if kind == "autograd":
        return _exact_autograd(fields[0], _parameters(case, seed), nd)
    F, theta, links = [], [], []
    for U in fields:
        U = _as_stored(U, _storage(case))
        if kind == "polish":  # its links are projected to SU(3) on the way in and out
            U = _reunit(_exact_fix(_reunit(U), nd, case["sweeps"]))
        elif kind == "fasd":
            U = _exact_fasd(U, nd, case["sweeps"])
        else:
            U = _exact_fix(U, nd, case["sweeps"])
        f, th = _F_theta(U, nd)
        F.append(f)
        theta.append(th)
        links.append(U)
    return {"F": torch.stack(F), "theta": torch.stack(theta), "iters": None, "links": links}
