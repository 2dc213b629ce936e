"""The kernel sets that LBO_OPT_KERNEL = 1 and 2 select where the default is
fixed point: pairs of FP32 (FP32X2), FP64 in registers (N = 32) and FP64 in
shared memory, for L[g], its Maxwellian cache, groups in a graph, and Q(f,f)
with both loss multipliers.

Tolerances: L[g] 4 u rms(r), the stated bound of the FFT form (u = 2^-48 for
the pairs), and 1e-12 in FP64 on inputs g = M p; Q(f,f), which transforms f
itself, 2^10 u for the pairs and 1e-12 in FP64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.linearized import Tables, apply_linearized
from oracle.quadratic import apply_quadratic
from oracle.quadrature import hemisphere_rule
from paper_2503_09580_gb300 import lbo, workloads

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
L, OMEGA = 8.0, 0.5
U = {"fp64": 2.0 ** -53, "fp32x2": 2.0 ** -48}
_TAB = {}


def tables(n):
    if n not in _TAB:
        _TAB[n] = Tables(n, L, OMEGA, n)
    return _TAB[n]


def maxwellians(n, params):
    a = workloads.velocity_axis(n, L)
    out = []
    for rho, u1, u2, u3, th in params:
        d2 = (a[:, None, None] - u1) ** 2 + (a[None, :, None] - u2) ** 2 + (a[None, None, :] - u3) ** 2
        out.append(rho * (2 * np.pi * th) ** -1.5 * np.exp(-d2 / (2 * th)))
    return np.stack(out)


def linearized(plan, params, g):
    tp, tg = (params, g) if torch.is_tensor(g) else (torch.from_numpy(params).to(DEV), torch.from_numpy(g).to(DEV))
    out = plan.apply_linearized(tp, tg, torch.full_like(tg, 7.0))
    plan.sync()
    return out.cpu().numpy()


def quadratic(plan, f):
    tf = torch.from_numpy(f).to(DEV)
    out = plan.apply_quadratic(tf, torch.full_like(tf, 7.0))
    plan.sync()
    return out.cpu().numpy()


def errs(a, b):
    return np.array([np.abs(a[i] - b[i]).max() / np.abs(b[i]).max() for i in range(b.shape[0])])


@pytest.mark.parametrize("n,precision,kernel", [(16, "fp32x2", 1), (32, "fp32x2", 1), (16, "fp64", 1), (32, "fp64", 1),
                                                (32, "fp64", 2)])
def test_linearized_and_its_cache_match_the_oracle(n, precision, kernel):
    params, g = workloads.batched_instances(n, L, batch=3, seed=41, noise=0.0)
    plan = lbo.Plan(n, L, OMEGA, n, precision=precision, kernel=kernel)
    tp, tg = torch.from_numpy(params).to(DEV), torch.from_numpy(g).to(DEV)
    got = linearized(plan, tp, tg)
    r = g / maxwellians(n, params)
    r[np.abs(r) > 1e8] = 0.0  # beyond the cut-off
    rms = np.sqrt((r * r).mean(axis=(1, 2, 3)))
    e = errs(got, apply_linearized(tables(n), params, g))
    assert np.all(e <= (4 * U[precision] * rms if precision == "fp32x2" else 1e-12))
    # another kernel set than the default's, and the cache with the same arithmetic
    assert not np.array_equal(got, linearized(lbo.Plan(n, L, OMEGA, n, precision=precision), tp, tg))
    plan.cache_maxwellians(tp)
    assert np.array_equal(linearized(plan, tp, tg), got)


def test_register_kernels_agree_with_shared_memory_ones_and_over_their_tiles():
    n = 32
    params, g = workloads.batched_instances(n, L, batch=4, seed=7, noise=0.0)
    tp, tg = torch.from_numpy(params).to(DEV), torch.from_numpy(g).to(DEV)
    a = linearized(lbo.Plan(n, L, OMEGA, n, kernel=1), tp, tg)
    assert errs(linearized(lbo.Plan(n, L, OMEGA, n, kernel=2), tp, tg), a).max() <= 1e-13
    for planes in (2, 8):
        plan = lbo.Plan(n, L, OMEGA, n, kernel=1, planes=planes)
        assert np.array_equal(linearized(plan, tp, tg), a)
        plan.cache_maxwellians(tp)
        assert np.array_equal(linearized(plan, tp, tg), a)
    plan = lbo.Plan(n, L, OMEGA, n, kernel=1)
    assert plan.autotune(tp, tg, torch.empty_like(tg)) in (2, 4, 8)
    assert np.array_equal(linearized(plan, tp, tg), a)


@pytest.mark.parametrize("cached", [False, True])
def test_register_kernels_and_pairs_in_a_captured_group(cached):
    opts = ({"kernel": 1, "planes": 8}, {"kernel": 1, "precision": "fp32x2"})
    plans = [lbo.Plan(32, L, OMEGA, 32, **o) for o in opts]
    ps, gs = [], []
    for i in range(2):
        params, g = workloads.batched_instances(32, L, batch=3, seed=60 + i, noise=1e-4)
        ps.append(torch.from_numpy(params).to(DEV))
        gs.append(torch.from_numpy(g).to(DEV))
    if cached:
        for plan, tp in zip(plans, ps):
            plan.cache_maxwellians(tp)
    ref = [linearized(plan, tp, tg) for plan, tp, tg in zip(plans, ps, gs)]
    group = lbo.Group(plans, graph=True)
    outs = [torch.full_like(g, float("nan")) for g in gs]
    with torch.cuda.stream(torch.cuda.Stream()):
        for _ in range(3):  # eager, capture and launch, replay
            for o in outs:
                o.fill_(float("nan"))
            group.apply_linearized(ps, gs, outs)
            torch.cuda.synchronize()
            assert all(np.array_equal(o.cpu().numpy(), r) for o, r in zip(outs, ref))
    group.close()


@pytest.mark.parametrize("n,precision,kernel,sinc", [(16, "fp32x2", 1, 0), (16, "fp32x2", 1, 1), (32, "fp32x2", 1, 0),
                                                     (32, "fp32x2", 1, 1), (16, "fp64", 1, 0), (32, "fp64", 1, 0),
                                                     (32, "fp64", 1, 1), (32, "fp64", 2, 0)])
def test_quadratic_matches_the_oracle(n, precision, kernel, sinc):
    p = 2
    params, g = workloads.batched_instances(n, L, batch=2, seed=46, noise=0.0)
    f = maxwellians(n, params) + 0.3 * g
    opts = dict(hemisphere_p=p, precision=precision, q_sinc_quadrature=sinc)
    got = quadratic(lbo.Plan(n, L, OMEGA, n, kernel=kernel, **opts), f)
    sig, w = hemisphere_rule(p)
    ref = apply_quadratic(tables(n), f, sig, w, **({"mass_fix": "sinc_quadrature"} if sinc else {}))
    assert np.all(errs(got, ref) <= (1024 * U[precision] if precision == "fp32x2" else 1e-12))
    assert not np.array_equal(got, quadratic(lbo.Plan(n, L, OMEGA, n, **opts), f))
