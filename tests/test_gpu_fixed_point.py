"""The fixed-point form of the FP64 precision (fx64.cuh, lin_fx.cuh,
quad_fx.cuh) against the FP64 kernels that LBO_OPT_KERNEL = 1 selects, at the
sizes where it can go wrong: every N, a batch that spans several groups of
the gain loop, few radial nodes, and inputs far from unit scale.

Tolerance: both forms are within the stated bound of FP64, 4 u rms(r) max|L|
(the ratio r = g/M over the grid), of the exact result, so they differ by at
most twice that (64 stands for the rms of r = O(1) inputs, where other FP64
roundings lead); Q transforms f itself, whose two forms are each within
2^-53 times the 3 log2 N^3 additions a value passes, times the 8 sqrt(J M)
of random sums over nodes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2503_09580_gb300 import lbo, workloads

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
U64 = 2.0 ** -53


def apply(plan, params, g, quad=False):
    tp, tg = torch.from_numpy(params).to(DEV), torch.from_numpy(g).to(DEV)
    out = torch.full_like(tg, 7.0)
    if quad:
        plan.apply_quadratic(tg, out)
    else:
        plan.apply_linearized(tp, tg, out)
    plan.sync()
    return out.cpu().numpy()


def ratio_rms(params, g, n, L, eps=1e-9):
    a = workloads.velocity_axis(n, L)
    r = np.zeros(params.shape[0])
    for b, (rho, u1, u2, u3, th) in enumerate(params):
        d2 = (a[:, None, None] - u1) ** 2 + (a[None, :, None] - u2) ** 2 + (a[None, None, :] - u3) ** 2
        M = rho * (2 * np.pi * th) ** -1.5 * np.exp(-d2 / (2 * th))
        keep = d2 / (2 * th) <= np.log(1 / eps) - 1.5 * np.log(2 * np.pi * th)
        r[b] = np.sqrt(((g[b][keep] / M[keep]) ** 2).sum() / n ** 3)
    return r


@pytest.mark.parametrize("n,batch,J,noise", [(16, 1, 16, 0.0), (16, 130, 3, 1e-3), (24, 3, 24, 1e-3), (24, 1, 1, 0.0),
                                             (32, 17, 32, 1e-3), (32, 1, 17, 0.0), (48, 2, 9, 1e-3), (64, 2, 5, 1e-3)])
def test_linearized_matches_the_fp64_kernels(n, batch, J, noise):
    L = 8.0
    params, g = workloads.batched_instances(n, L, batch=batch, seed=70 + n, noise=noise)
    a = apply(lbo.Plan(n, L, 0.74, J), params, g)
    b = apply(lbo.Plan(n, L, 0.74, J, kernel=1), params, g)
    tol = 2 * 4 * U64 * np.maximum(ratio_rms(params, g, n, L), 64.0)
    for i in range(batch):
        assert np.abs(a[i] - b[i]).max() <= tol[i] * np.abs(b[i]).max(), i


def test_scale_and_degenerate_inputs():
    """A power of two on g is exact; a zero field gives zero; a field or a
    Maxwellian that is not finite gives NaN in its own instance alone; a
    negative density and one far from 1 agree with the FP64 kernels."""
    n, L = 16, 8.0
    params, g = workloads.batched_instances(n, L, batch=6, seed=80, noise=1e-3)
    plan, ref = lbo.Plan(n, L, 0.5, n), lbo.Plan(n, L, 0.5, n, kernel=1)
    base = apply(plan, params, g)
    for e in (200, -300):
        assert np.array_equal(apply(plan, params, np.ldexp(g, e)), np.ldexp(base, e))
    p2, g2 = params.copy(), g.copy()
    g2[0] = 0.0
    g2[1, 3, 4, 5] = np.nan
    g2[2, 0, 0, 7] = np.inf
    p2[3, 4] = -1.0
    p2[4, 0] = -0.7
    p2[5, 0] = 1e-100
    a, b = apply(plan, p2, g2), apply(ref, p2, g2)
    assert np.all(a[0] == 0)
    for i in (1, 2, 3):
        assert np.all(np.isnan(a[i])) and np.all(np.isnan(b[i]))
    tol = 2 * 4 * U64 * np.maximum(ratio_rms(np.abs(p2), g2, n, L), 64.0)
    for i in (4, 5):
        assert np.abs(a[i] - b[i]).max() <= tol[i] * np.abs(b[i]).max()


@pytest.mark.parametrize("n,batch,J,p,kw", [(16, 5, 16, 1, {}), (16, 1, 3, 5, {"q_sinc_quadrature": 1}), (24, 3, 24, 2, {}),
                                            (32, 3, 32, 4, {}), (32, 2, 5, 2, {"q_sinc_quadrature": 1}), (48, 2, 4, 3, {}),
                                            (64, 1, 12, 4, {}), (64, 1, 64, 16, {})])  # the last in two cuts of its nodes
def test_quadratic_matches_the_fp64_kernels(n, batch, J, p, kw):
    L = 8.0
    _, g = workloads.batched_instances(n, L, batch=batch, seed=90 + n, noise=0.0)
    params = np.zeros((batch, 5))
    a = apply(lbo.Plan(n, L, 0.5, J, hemisphere_p=p, **kw), params, g, quad=True)
    b = apply(lbo.Plan(n, L, 0.5, J, hemisphere_p=p, kernel=1, **kw), params, g, quad=True)
    tol = 2 * U64 * 3 * 3 * np.log2(n) * 8
    for i in range(batch):
        assert np.abs(a[i] - b[i]).max() <= tol * np.abs(b[i]).max(), i
    g[0] = 0.0
    g[-1, 1, 2, 3] = np.nan
    c = apply(lbo.Plan(n, L, 0.5, J, hemisphere_p=p, **kw), params, g, quad=True)
    assert np.all(np.isnan(c[-1]))
    if batch > 1:
        assert np.all(c[0] == 0)
        assert all(np.array_equal(c[i], a[i]) for i in range(1, batch - 1))


@pytest.mark.parametrize("n", [16, 24, 32, 48, 64])
def test_pairs_of_fp32_stay_reachable(n):
    """FP32X2 runs in fixed point by default, bit for bit as FP64 does;
    kernel = 1 still selects the pairs of FP32, within their 2^-48 bound."""
    L = 8.0
    params, g = workloads.batched_instances(n, L, batch=2, seed=110 + n, noise=1e-3)
    a = apply(lbo.Plan(n, L, 0.5, n), params, g)
    assert np.array_equal(a, apply(lbo.Plan(n, L, 0.5, n, precision="fp32x2"), params, g))
    b = apply(lbo.Plan(n, L, 0.5, n, precision="fp32x2", kernel=1), params, g)
    assert not np.array_equal(a, b)
    tol = 4 * (2.0 ** -48 + U64) * np.maximum(ratio_rms(params, g, n, L), 64.0)
    for i in range(2):
        assert np.abs(a[i] - b[i]).max() <= tol[i] * np.abs(b[i]).max()


@pytest.mark.parametrize("n,precision", [(16, "fp64"), (32, "fp32x2")])
def test_cut_off_changed_after_the_maxwellian_cache(n, precision):
    """The cached tables that depend on the cut-off level are made again when
    it changes: cached and plain applications stay equal bit for bit."""
    L = 8.0
    params, g = workloads.batched_instances(n, L, batch=3, seed=120, noise=1e-3)
    tp, tg = torch.from_numpy(params).to(DEV), torch.from_numpy(g).to(DEV)
    plan, plain = (lbo.Plan(n, L, 0.5, n, precision=precision) for _ in range(2))
    plan.cache_maxwellians(tp)
    for eps in (1e-9, 1e-5, 1e-9):
        plan.set("eps", eps)
        plain.set("eps", eps)
        a, b = torch.empty_like(tg), torch.empty_like(tg)
        plan.apply_linearized(tp, tg, a)
        plain.apply_linearized(tp, tg, b)
        plan.sync(), plain.sync()
        assert torch.equal(a, b)


def test_captured_graph_outlives_other_batches():
    """A smaller batch, and an uncached call after a cached one, need no more
    workspace than the larger, cached one: a graph captured with the plan still
    replays.  1821 instances take two groups of 911, 1820 one group of 1820."""
    n, L = 16, 8.0
    params, g = workloads.batched_instances(n, L, batch=4, seed=130, noise=1e-3)
    tp, tg = (torch.from_numpy(np.resize(x, (1821,) + x.shape[1:])).to(DEV) for x in (params, g))
    plan = lbo.Plan(n, L, 0.5, n)
    plan.cache_maxwellians(tp)
    group = lbo.Group([plan], graph=True)
    out, other = torch.empty_like(tg), torch.empty_like(tg[:1820])
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        for _ in range(2):  # eager, capture
            group.apply_linearized([tp], [tg], [out])
    torch.cuda.synchronize()
    ref = out.clone()
    plan.apply_linearized(tp[:1820].clone(), tg[:1820], other)
    plan.sync()
    out.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        group.apply_linearized([tp], [tg], [out])
    torch.cuda.synchronize()
    assert torch.equal(out, ref) and torch.equal(other, ref[:1820])
    group.close()


@pytest.mark.parametrize("n,precision,kernel", [(16, "fp64", 0), (64, "fp64", 0), (32, "fp64", 1), (32, "fp32", 0),
                                                (16, "fp64x2", 0)])
def test_first_application_on_a_non_blocking_stream(n, precision, kernel):
    """The tables a plan makes at its first application are in place before
    the kernels of a stream that is not ordered behind the legacy one."""
    L = 8.0
    params, g = workloads.batched_instances(n, L, batch=2, seed=140, noise=0.0)
    tp, tg = torch.from_numpy(params).to(DEV), torch.from_numpy(g).to(DEV)
    torch.cuda.synchronize()
    outs = []
    for _ in range(4):
        plan = lbo.Plan(n, L, 0.5, n, hemisphere_p=2, precision=precision, kernel=kernel, q_sinc_quadrature=1)
        with torch.cuda.stream(torch.cuda.Stream()):
            outs.append([plan.apply_linearized(tp, tg, torch.empty_like(tg)),
                         plan.apply_quadratic(tg, torch.empty_like(tg))])
            plan.sync()
    for lin, quad in outs[1:]:
        assert torch.equal(lin, outs[0][0]) and torch.equal(quad, outs[0][1])


@pytest.mark.parametrize("opts", [{}, {"q_sinc_quadrature": 1}, {"precision": "fp32"}, {"kernel": 1}])
def test_radial_cut_and_scale_changed_after_an_application(opts):
    """R and C set after Q and L have run on a plan: everything derived from
    the radial rule is made again, equal to a new plan's."""
    n, L = 32, 8.0
    params, g = workloads.batched_instances(n, L, batch=2, seed=153, noise=0.0)
    opts = dict(opts, hemisphere_p=2)
    plan = lbo.Plan(n, L, 0.5, n, **opts)
    now = {"R": 4 * L / (3 + np.sqrt(2.0)), "C": 1 / (4 * np.pi)}
    for key, factor in (("R", 1.0), ("R", 0.6), ("C", 1 / 64), ("C", 64.0), ("R", 1 / 0.6)):
        now[key] *= factor
        plan.set(key, now[key])
        new = lbo.Plan(n, L, 0.5, n, **opts)
        for k, v in now.items():
            new.set(k, v)
        for quad in (True, False):
            assert np.array_equal(apply(plan, params, g, quad=quad), apply(new, params, g, quad=quad)), (key, factor)


@pytest.mark.parametrize("n", [16, 32, 64])
def test_up_to_the_limits_of_fp64(n):
    """Powers of two on the input are exact up to FP64's own limits: as long
    as r = g/M is finite for L[g], and the two terms of Q(f,f) for Q (the
    result 2^8 below the largest number).  The bounds of intermediate fields,
    which carry the N^3 of unnormalised transforms, reach beyond.  An r that
    is not finite gives NaN in its own instance."""
    L, theta = 8.0, 2.0
    params = np.array([[1.0, 0.1, -0.2, 0.05, theta]] * 2)
    d = [workloads.velocity_axis(n, L) - u for u in params[0, 1:4]]
    d2 = d[0][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[2][None, None, :] ** 2
    g = np.stack([(2 * np.pi * theta) ** -1.5 * np.exp(-d2 / (2 * theta)) * (1 + c * d[0][:, None, None])
                  for c in (0.3, 0.2)])
    plan = lbo.Plan(n, L, 0.5, n, hemisphere_p=2)
    base = apply(plan, params, g)
    for e in (960, 1013, 1020):
        assert np.array_equal(apply(plan, params, np.ldexp(g, e)), np.ldexp(base, e)), e
    out = apply(plan, params, np.stack([np.ldexp(g[0], 1000), np.ldexp(g[1], 1024)]))
    assert np.array_equal(out[0], np.ldexp(base[0], 1000)) and np.all(np.isnan(out[1]))
    base = apply(plan, params, g, quad=True)
    top = int(np.log2(np.abs(base).max())) + 1
    for margin in (60, 20, 12, 8):
        e = (1023 - top - margin) // 2
        assert np.array_equal(apply(plan, params, np.ldexp(g, e), quad=True), np.ldexp(base, 2 * e)), margin


@pytest.mark.parametrize("n,theta,rho", [(32, 0.05, 1.0), (32, 0.05, 1e-40), (16, 0.05, 1e-100), (32, 0.07, 1e-100)])
def test_cold_thin_gases_whose_outer_planes_vanish(n, theta, rho):
    """exp(-|v - u|^2 / theta) underflows on the outer planes of a cold gas;
    they have no part in the exponents of the others, however small rho is."""
    L = 8.0
    params = np.array([[rho, 0.1, -0.2, 0.05, theta]])
    d = [workloads.velocity_axis(n, L) - u for u in params[0, 1:4]]
    assert (np.exp(-d[0] ** 2 / theta) == 0).any()
    d2 = d[0][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[2][None, None, :] ** 2
    g = (rho * (2 * np.pi * theta) ** -1.5 * np.exp(-d2 / (2 * theta)) * (1 + 0.3 * d[0][:, None, None] + d2))[None]
    a = apply(lbo.Plan(n, L, 0.5, n), params, g)
    b = apply(lbo.Plan(n, L, 0.5, n, kernel=1), params, g)
    tol = 2 * 4 * U64 * max(ratio_rms(params, g, n, L)[0], 64.0)
    assert np.abs(a - b).max() <= tol * np.abs(b).max()


def quadratic_errors(n, J, p, batch=8):
    """2-norm errors of Q over a batch of sums of two Maxwellians, as the FP64
    kernels' and the default's, against pairs of FP64 on the same tables."""
    L = 8.0
    rng = np.random.Generator(np.random.PCG64(160 + n))
    a = workloads.velocity_axis(n, L)
    f = np.zeros((batch, n, n, n))
    for b in range(batch):
        for _ in range(2):
            rho, th, u = rng.uniform(0.3, 1.0), rng.uniform(0.5, 1.5), rng.uniform(-1.0, 1.0, 3)
            e = [np.exp(-(a - x) ** 2 / (2 * th)) for x in u]
            f[b] += rho * (2 * np.pi * th) ** -1.5 * e[0][:, None, None] * e[1][None, :, None] * e[2][None, None, :]
    out = [apply(lbo.Plan(n, L, 0.5, J, hemisphere_p=p, **kw), np.zeros((batch, 5)), f, quad=True)
           for kw in ({"precision": "fp64x2"}, {"kernel": 1}, {})]
    return [np.sqrt(((x - out[0]) ** 2).sum(axis=(1, 2, 3)) / (out[0] ** 2).sum(axis=(1, 2, 3))) for x in out[1:]]


@pytest.mark.parametrize("n,J,p", [(16, 16, 4), (16, 9, 2), (16, 9, 4), (32, 17, 4), (16, 16, 16), (32, 17, 12)])
def test_quadratic_errs_no_more_than_the_fp64_kernels(n, J, p):
    """Hard spheres weigh the largest radial nodes most, where T+ and T- hardly
    meet: a mean error of either shows in the mass of Q+.  The errors of a
    batch, together, stay below those of FP64 transforms."""
    fp64, fixed = quadratic_errors(n, J, p)
    assert np.sqrt((fixed ** 2).mean()) <= np.sqrt((fp64 ** 2).mean())


@pytest.mark.parametrize("n,J,p,batch,kw", [(16, 1, 4, 40, {}), (16, 3, 8, 17, {}), (24, 2, 1, 29, {}), (24, 5, 6, 11, {}),
                                            (32, 1, 3, 9, {}), (32, 2, 6, 5, {}), (48, 1, 2, 5, {}),
                                            (64, 1, 2, 4, {"q_sinc_quadrature": 1}), (64, 2, 6, 2, {})])
def test_quadratic_of_few_instances_is_that_of_a_batch(n, J, p, batch, kw):
    """A launch with fewer blocks than SMs stores the products of the hemisphere
    nodes and adds them in a second kernel, in the order and with the bits of
    the launch that a batch takes; the first and the last instance, whose share
    of nodes per block differ with the batch."""
    L = 8.0
    _, g = workloads.batched_instances(n, L, batch=batch, seed=170 + n, noise=0.0)
    params = np.zeros((batch, 5))
    plan = lbo.Plan(n, L, 0.5, J, hemisphere_p=p, **kw)
    whole = apply(plan, params, g, quad=True)
    for i in (0, batch - 1):
        assert np.array_equal(apply(plan, params[i:i + 1], g[i:i + 1], quad=True)[0], whole[i])
    two = apply(plan, params[:2], g[:2], quad=True)
    assert np.array_equal(two, whole[:2])
