"""The measured workloads of the library: applications of the linearized
operator L[g], of the quadratic operator Q(f,f), and the time integration and
Newton steps built from them, each through the calls of
paper_2503_09580_gb300.lbo that a user's program makes.

A case names the operation and its sizes:
  op         linearized  Plan.apply_linearized
             cached      the same with the Maxwellian factors cached (the
                         Krylov products of one Newton step)
             quadratic   Plan.apply_quadratic
             evolve      Plan.evolve, `steps` RK4 steps of df/dt = L_M[f]
             newton      Solver.newton_step on a slab of `batch` cells
  n, j       points per direction, radial nodes
  batch      instances (cells)
  precision  LBO_OPT_PRECISION;  omega: the VHS exponent;  box: L
  p          hemisphere rule order, M = 2 p^2 (quadratic, newton)
  noise      grid noise of the linearized inputs
"""
import math

import numpy as np
import torch

from paper_2503_09580_gb300 import lbo

SIZES = (16, 24, 32, 48, 64)
PAPER_BOX = 6.0 * (3.0 + math.sqrt(2.0)) / 4.0  # R = 6 (Sec. 4.2 of the paper)


def _case(name, op, n, batch, precision="fp64", omega=0.5, j=None, box=8.0, p=4, noise=1e-3, steps=1):
    c = {"op": op, "n": n, "j": n if j is None else j, "batch": batch, "precision": precision, "omega": omega,
         "box": box, "p": p, "noise": noise, "steps": steps}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one spatially homogeneous instance, cubic polynomial times the
        # Maxwellian: launches and latency
        _case("single_16", "linearized", 16, 1, noise=0.0),
        # the cells of a mixed-N slab that carry the coarse grid, a ragged count
        _case("cells_24", "linearized", 24, 37),
        # the benchmark's batch: per-instance Maxwellians, quartic plus noise
        _case("batch_32", "linearized", 32, 256),
        _case("batch_32_fp32", "linearized", 32, 256, precision="fp32"),
        # the few cells of a mixed-N slab on the fine grid
        _case("cells_48", "linearized", 48, 11),
        # the large grid, variable hard spheres
        _case("batch_64", "linearized", 64, 64, omega=0.74),
        # one Krylov product of a 128-cell Newton step
        _case("krylov_32", "cached", 32, 128),
        # homogeneous relaxation of one distribution by RK4, the paper's grid and radial rule
        _case("relax_32", "evolve", 32, 1, omega=1.0, j=17, box=PAPER_BOX, steps=5),
        # Q(f,f) of a group of cells
        _case("q_32", "quadratic", 32, 32),
        _case("q_32_fp32", "quadratic", 32, 128, precision="fp32"),
        # the residual of one backward-Euler step of the BKW relaxation
        _case("bkw_64", "quadratic", 64, 1, precision="fp32x2", omega=1.0),
        # a whole Newton step of the Fourier-flow slab
        _case("newton_8", "newton", 32, 8, p=2),
    ]


def draw(rng):
    op = rng.choice(("linearized", "linearized", "linearized", "cached", "quadratic", "quadratic", "evolve", "newton"))
    n = rng.choice(SIZES)
    precision = rng.choice(("fp64", "fp64", "fp64", "fp64", "fp32", "fp32x2"))
    omega = rng.choice((0.5, 0.74, 1.0))
    j = rng.choice((n, n, n // 2 + 1))
    box = rng.choice((8.0, 8.0, PAPER_BOX))
    noise = rng.choice((1e-3, 1e-3, 0.0))
    p, steps = 4, 1
    if op == "quadratic":
        p = rng.choice((2, 3, 4))
    elif op == "evolve":
        precision, steps = "fp64", rng.randint(1, 6)
    elif op == "newton":
        n, precision, p, omega, box = rng.choice((16, 24, 32)), "fp64", 2, 0.5, 8.0
        j = n
    c = _case(None, op, n, 1, precision, omega, j, box, p, noise, steps)
    # as many instances as the largest listed case's arithmetic allows (the
    # FP32 forms are faster per operation, but their launches are not)
    most = work(_case(None, "linearized", 64, 64))["flops"]
    top = min(512, int(0.9 * most / work(c)["flops"]))
    if op == "newton":
        top = min(top, 24)
        c["batch"] = rng.randint(2, max(2, top))
    else:
        c["batch"] = int(round(math.exp(rng.uniform(0.0, math.log(max(1, top))))))
    return c


# ------------------------------------------------------------------ inputs
def _axis(n, box):
    return (torch.arange(n, dtype=torch.float64, device="cuda") - n // 2) * (2.0 * box / n)


def _gaussian(n, box, theta, u):
    """prod_d exp(-(v_d - u_d)^2 / (2 theta)), theta (B), u (B, 3)."""
    a = _axis(n, box)
    e = [torch.exp(-(a[None, :] - u[:, d:d + 1]) ** 2 / (2.0 * theta[:, None])) for d in range(3)]
    return e[0][:, :, None, None] * e[1][:, None, :, None] * e[2][:, None, None, :]


def _maxwellian(n, box, params):
    rho, theta = params[:, 0], params[:, 4]
    return (rho * (2.0 * math.pi * theta) ** -1.5)[:, None, None, None] * _gaussian(n, box, theta, params[:, 1:4])


def _linearized_inputs(case, seed):
    """Background Maxwellians and g = M * polynomial (+ grid noise): one
    instance about the standard normal with a cubic, batches with drawn
    Maxwellians and a quartic, as the library's workloads are."""
    n, box, B = case["n"], case["box"], case["batch"]
    rng = np.random.Generator(np.random.PCG64(seed))
    params = np.empty((B, 5))
    if B == 1:
        params[0] = (1.0, 0.0, 0.0, 0.0, 1.0)
    else:
        params[:, 0] = rng.uniform(0.5, 2.0, B)
        params[:, 1:4] = rng.uniform(-0.5, 0.5, (B, 3))
        params[:, 4] = rng.uniform(0.5, 2.0, B)
    degree = 3 if B == 1 else 4
    coeff = torch.from_numpy(rng.standard_normal((B, degree + 1, degree + 1, degree + 1))).cuda()
    k = torch.arange(degree + 1, device="cuda")
    coeff *= ((k[:, None, None] + k[None, :, None] + k[None, None, :]) <= degree)
    params = torch.from_numpy(params).cuda()
    a, sq = _axis(n, box), params[:, 4].sqrt()
    pw = [((a[None, :] - params[:, 1 + d:2 + d]) / sq[:, None])[:, None, :] ** k[None, :, None] for d in range(3)]
    g = torch.einsum("bijk,bix->bxjk", coeff, pw[0])
    g = torch.einsum("bxjk,bjy->bxyk", g, pw[1])
    g = torch.einsum("bxyk,bkz->bxyz", g, pw[2])
    g *= _maxwellian(n, box, params)
    if case["noise"]:
        gen = torch.Generator(device="cuda").manual_seed(seed)
        g += case["noise"] * torch.randn(g.shape, dtype=torch.float64, device="cuda", generator=gen)
    return params, g.contiguous()


def _distributions(case, seed):
    """Positive distributions: for one instance the BKW profile at a drawn
    time, for batches the sum of two drawn Maxwellians."""
    n, box, B = case["n"], case["box"], case["batch"]
    rng = np.random.Generator(np.random.PCG64(seed))
    if B == 1:
        K = rng.uniform(0.6, 0.95)
        a = _axis(n, box)
        v2 = a[:, None, None] ** 2 + a[None, :, None] ** 2 + a[None, None, :] ** 2
        f = (2 * math.pi * K) ** -1.5 * torch.exp(-v2 / (2 * K)) * ((5 * K - 3) / (2 * K) + (1 - K) / (2 * K * K) * v2)
        return f[None].contiguous()
    f = 0.0
    for _ in range(2):
        p = np.concatenate([rng.uniform(0.3, 1.0, (B, 1)), rng.uniform(-1.0, 1.0, (B, 3)), rng.uniform(0.5, 1.5, (B, 1))], 1)
        f = f + _maxwellian(n, box, torch.from_numpy(p).cuda())
    return f.contiguous()


def _slab_state(case, seed):
    """Maxwellians between the walls' temperatures, slightly perturbed."""
    nx = case["batch"]
    rng = np.random.Generator(np.random.PCG64(seed))
    p = np.zeros((nx, 5))
    p[:, 0] = 1.0 + 0.1 * rng.uniform(-1.0, 1.0, nx)
    p[:, 1:4] = 0.05 * rng.uniform(-1.0, 1.0, (nx, 3))
    p[:, 4] = 1.5 + 0.1 * rng.uniform(-1.0, 1.0, nx)
    return _maxwellian(case["n"], case["box"], torch.from_numpy(p).cuda()).contiguous()


def _plan(case):
    opts = {"precision": case["precision"]}
    if case["op"] in ("quadratic", "newton"):
        opts["hemisphere_p"] = case["p"]
    return lbo.Plan(case["n"], case["box"], case["omega"], case["j"], **opts)


def prepare(case, seed):
    s = {"op": case["op"], "plan": _plan(case), "steps": case["steps"]}
    if case["op"] in ("linearized", "cached"):
        s["params"], s["g"] = _linearized_inputs(case, seed)
        s["out"] = torch.empty_like(s["g"])
        if case["op"] == "cached":
            s["plan"].cache_maxwellians(s["params"])
    elif case["op"] == "evolve":
        s["f"] = _distributions(case, seed)
        s["params"] = torch.tensor([[1.0, 0.0, 0.0, 0.0, 1.0]], dtype=torch.float64, device="cuda").repeat(case["batch"], 1)
    elif case["op"] == "quadratic":
        s["f"] = _distributions(case, seed)
        s["out"] = torch.empty_like(s["f"])
    else:
        s["f"] = _slab_state(case, seed)
        nx, h = case["batch"], 2.0 * case["box"] / case["n"]
        s["solver"] = s["plan"].solver(kind="slab", nx=nx, x_left=0.0, x_right=1.0, kn=1.0,
                                       wall_left=(1.0, 0.0, 0.0, 0.0), wall_right=(2.0, 0.0, 0.0, 0.0),
                                       total_mass=float(h ** 3 / nx * s["f"].sum()), wall_flux="discrete",
                                       krylov_rtol=1e-3, krylov_atol=1e-12, krylov_restart=40, krylov_maxit=400,
                                       precond="sweep")
    return s


def run(s):
    if s["op"] in ("linearized", "cached"):
        return s["plan"].apply_linearized(s["params"], s["g"], s["out"])
    if s["op"] == "quadratic":
        return s["plan"].apply_quadratic(s["f"], s["out"])
    f = s["f"].clone()
    if s["op"] == "evolve":
        return s["plan"].evolve("linearized", f, 0.1, s["steps"], params=s["params"])
    stats = s["solver"].newton_step(f)
    return {"f": f, "residual_norm": stats["residual_norm"]}


# ------------------------------------------------------------------ work
def work(case):
    """Each field in and out once; real 3-D transforms of n^3 points at
    2.5 n^3 log2 n^3 operations, the even u^_j as DCTs of one octant."""
    n, J, B = case["n"], case["j"], case["batch"]
    n3 = float(n) ** 3
    real3d = 2.5 * n3 * 3.0 * math.log2(n)
    hn = n // 2 + 1
    octant = 3.0 * hn ** 3 * (n / 2.0 + 1.0)
    gain = J * (2.0 * real3d + 8.0 * n3)
    uhat = J * octant + 2.0 * real3d
    nodes = 2 * case["p"] ** 2
    quad = J * (nodes * (2.0 * real3d + 8.0 * n3) + real3d) + 4.0 * real3d
    if case["op"] == "linearized":
        flops = gain + uhat + 4.0 * real3d
    elif case["op"] == "cached":
        flops = gain + 4.0 * real3d
    elif case["op"] == "evolve":
        flops = uhat + 4.0 * case["steps"] * (gain + 4.0 * real3d)
    elif case["op"] == "quadratic":
        flops = quad
    else:  # one residual, and a handful of Krylov products about cached Maxwellians
        flops = quad + uhat + 8.0 * (gain + 4.0 * real3d)
    return {"bytes": B * (16.0 * n3 + (0.0 if case["op"] == "quadratic" else 40.0)), "flops": B * flops}


# ------------------------------------------------------------------ exact
def _fft(x):
    return torch.fft.fftn(x, dim=(-3, -2, -1))


def _ifft(x):
    return torch.fft.ifftn(x, dim=(-3, -2, -1))


def _cyclic(x):
    return torch.fft.ifftshift(x, dim=(-3, -2, -1))


def _centred(x):
    return torch.fft.fftshift(x, dim=(-3, -2, -1))


def _sinc(x):
    return torch.where(x == 0, torch.ones_like(x), torch.sin(x) / torch.where(x == 0, torch.ones_like(x), x))


class _Exact:
    """The operators of Algorithm 1 and Eq. (2.14) in 64 bits, cyclic order."""

    def __init__(self, case):
        self.n, self.L, self.J = case["n"], case["box"], case["j"]
        n, L = self.n, self.L
        R = 4.0 * L / (3.0 + math.sqrt(2.0))
        x, w = np.polynomial.legendre.leggauss(self.J)
        self.g = 0.5 * R * (x + 1.0)
        self.wB = 0.5 * R * w * self.g ** 2 * self.g ** (2.0 * (1.0 - case["omega"])) / (4.0 * math.pi)
        k = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")
        self.k = k
        self.knorm = (k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2).sqrt()
        self.loss = 16.0 * math.pi ** 2 * sum(self.wB[i] * _sinc(math.pi * self.g[i] / L * self.knorm)
                                              for i in range(self.J))
        a = torch.fft.ifftshift(_axis(n, L))
        self.a, self.v2 = a, a[:, None, None] ** 2 + a[None, :, None] ** 2 + a[None, None, :] ** 2

    def shape(self, i):
        return _sinc(0.5 * math.pi * self.g[i] / self.L * self.knorm)

    def linearized(self, params, f, eps=1e-9):
        c = lambda x: x[:, None, None, None]  # noqa: E731
        rho, th = params[:, 0], params[:, 4]
        d = [self.a[None, :] - params[:, 1 + i:2 + i] for i in range(3)]
        d2 = d[0][:, :, None, None] ** 2 + d[1][:, None, :, None] ** 2 + d[2][:, None, None, :] ** 2
        M = c(rho * (2.0 * math.pi * th) ** -1.5) * torch.exp(-d2 / c(2.0 * th))
        pre = c(rho * (math.pi * th) ** -1.5)
        Mg, Mh = pre * torch.exp(-self.v2[None] / c(th)), pre * torch.exp(-d2 / c(th))
        cut = d2 / c(2.0 * th) > c(math.log(1.0 / eps) - 1.5 * torch.log(2.0 * math.pi * th))
        r = _fft(torch.where(cut, torch.zeros_like(f), f / torch.where(cut, torch.ones_like(M), M)))
        acc = torch.zeros_like(r)
        for i in range(self.J):
            s = self.shape(i)
            u = _fft(Mg * _ifft(s).real)
            acc += (4.0 * math.pi ** 2 * self.wB[i]) * s * _fft(Mh * _ifft(u * r).real)
        return _ifft(acc).real - _ifft(_fft(f) * self.loss).real * M - _ifft(_fft(M) * self.loss).real * f

    def quadratic(self, f, p):
        n, k = self.n, self.k
        x, w = np.polynomial.legendre.leggauss(p)
        mu, wmu = 0.5 * (x + 1.0), 0.5 * w
        phi = (np.arange(2 * p) + 0.5) * math.pi / p
        nyq = torch.arange(n, device="cuda") == n // 2
        F = _fft(f)
        acc = torch.zeros_like(F)
        for i in range(self.J):
            prod = torch.zeros_like(f)
            for a in range(p):
                st = math.sqrt(1.0 - mu[a] * mu[a])
                for ph in phi:
                    E = None
                    for dim, sg in enumerate((st * math.cos(ph), st * math.sin(ph), mu[a])):
                        al = 0.5 * math.pi * self.g[i] * sg / self.L
                        e = torch.where(nyq, torch.complex(torch.cos(al * k.abs()), torch.zeros_like(k)),
                                        torch.complex(torch.cos(al * k), torch.sin(al * k)))
                        e = e.reshape([n if q == dim else 1 for q in range(3)])
                        E = e if E is None else E * e
                    t = _ifft(F * E + 1j * (F * E.conj()))  # T+ + i T-
                    prod += (wmu[a] / (2 * p)) * t.real * t.imag
            acc += self.wB[i] * self.shape(i) * _fft(prod)
        return 16.0 * math.pi ** 2 * _ifft(acc).real - f * _ifft(F * self.loss).real


def exact(case, seed):
    if case["op"] == "newton":
        return None  # the step is an iterative solve to a tolerance
    ex = _Exact(case)
    chunk = max(1, (1 << 26) // case["n"] ** 3)
    if case["op"] in ("linearized", "cached"):
        params, g = _linearized_inputs(case, seed)
        return torch.cat([_centred(ex.linearized(params[i:i + chunk], _cyclic(g[i:i + chunk])))
                          for i in range(0, case["batch"], chunk)])
    f = _cyclic(_distributions(case, seed))
    if case["op"] == "quadratic":
        return torch.cat([_centred(ex.quadratic(f[i:i + chunk], case["p"])) for i in range(0, case["batch"], chunk)])
    params = torch.tensor([[1.0, 0.0, 0.0, 0.0, 1.0]], dtype=torch.float64, device="cuda").repeat(case["batch"], 1)
    h = 0.1
    for _ in range(case["steps"]):
        k1 = ex.linearized(params, f)
        k2 = ex.linearized(params, f + 0.5 * h * k1)
        k3 = ex.linearized(params, f + 0.5 * h * k2)
        k4 = ex.linearized(params, f + h * k3)
        f = f + (h / 6.0) * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
    return _centred(f)
