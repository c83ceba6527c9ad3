"""Line contractions of the DG kernels in block fixed point: against the same
kernels' FP64 form, which an element takes as soon as a field of it is not finite,
over the orders and over fields of very different sizes; homogeneity over the range
of exponents; and steps with weak and strong filters against the oracle.

Tolerance of the box comparison: the FP64 form's error, at most 18 roundings of a
sum of |D u| (2^-53 each); the fixed-point one's is smaller."""
import numpy as np
import pytest

import ffe_workloads as W
from gpu_common import compare_state
from oracle.basis import Tables
from oracle.problem import Problem
from oracle.stepper import Stepper
from test_gpu_parity import ffe  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = {"equal": np.ones(9), "unequal": np.array([1e-5, 1e-5, 1e-4, 1, 1, 1, 1e-6, 1e2, 1e3])}


def _box(P):
    cfg = W.fast_wave(n=3, P=P)
    cfg.update(n=(3, 2, 2), hi=tuple(l + w for l, w in zip(cfg["lo"], (0.9, 0.2, 7.0))))
    cfg["params"]["eta"] = 7.0
    return cfg


def _state(ctx, sizes, seed):
    rng = np.random.default_rng(seed)
    n = ctx.P + 1
    dg = (rng.normal(size=(9, ctx.n_elem, n, n, n)) + 0.5) * sizes[:, None, None, None, None]
    return ctx.join(dg, np.zeros((9, ctx.n_elem) + (ctx.nc,) * 3))


def _rhs(ctx, host):
    ctx.set_initial()
    U = torch.from_numpy(host).cuda()
    ctx.set_state(U, torch.zeros(ctx.n_elem, dtype=torch.uint8, device="cuda"))
    out = torch.zeros_like(U)
    ctx.rhs(U, out)
    torch.cuda.synchronize()
    return ctx.split(out.cpu().numpy())[0].copy()


def _spoiled(ctx, host):
    """psi~ not a number at one interior node of every element."""
    h = host.copy()
    c = ctx.P // 2
    dg, fd = ctx.split(h)
    dg = dg.copy()
    dg[6, :, c, c, c] = np.nan
    return ctx.join(dg, fd)


@pytest.mark.parametrize("sizes", list(SIZES))
@pytest.mark.parametrize("P", [3, 4, 5, 6])
def test_box_volume(ffe, P, sizes):  # noqa: F811
    cfg = _box(P)
    ctx = ffe.Context(cfg)
    host = _state(ctx, SIZES[sizes], P)
    a, b = _rhs(ctx, host), _rhs(ctx, _spoiled(ctx, host))
    assert np.isfinite(a).all()
    c = P // 2
    lines = np.zeros(a.shape, bool)   # d psi~/dx^i in E~^i: the line along axis i
    lines[0, :, c, c, :] = lines[1, :, c, :, c] = lines[2, :, :, c, c] = True
    assert (np.isnan(b) == lines).all()
    D = np.abs(Tables(P).D).sum(1).max()
    rows = D * sum(2.0 * n / (hi - lo) for n, lo, hi in zip(cfg["n"], cfg["lo"], cfg["hi"]))
    dg = ctx.split(host)[0]
    E2, B2, EB = (dg[0:3] ** 2).sum(0), (dg[3:6] ** 2).sum(0), (dg[0:3] * dg[3:6]).sum(0)
    J = np.sqrt(E2 / B2) * np.abs(dg[8]) + 7.0 * (np.abs(EB) / B2 * np.sqrt(B2) + np.maximum(E2 / B2 - 1, 0) * np.sqrt(E2))
    top = lambda x: x.reshape(-1, ctx.n_elem, (P + 1) ** 3).max(axis=(0, 2))  # noqa: E731
    mE, mB = top(np.abs(dg[[0, 1, 2, 7]])), top(np.abs(dg[3:7]))
    for v in range(9):
        m = mB if v in (0, 1, 2, 7) else (mE if v < 8 else top(J[None]))
        err = np.where(lines[v], 0.0, np.abs(a[v] - b[v])).reshape(ctx.n_elem, -1).max(1)
        assert (err <= 2.0 ** -48 * rows * m).all(), (v, err / (rows * m))
    ctx.close()


@pytest.mark.parametrize("metric", ["flat", "kerr-schild"])
@pytest.mark.parametrize("P", [3, 4, 5])
def test_shell_volume(ffe, P, metric):  # noqa: F811
    cfg = W.pulsar(r_lc=3.0, chi=0.4, n_ang=1, n_rad=3, P=P, r_out=4.0) if metric == "flat" else W.wald(
        spin=0.7, n_ang=1, n_rad=3, P=P)
    ctx = ffe.Context(cfg)
    host = _state(ctx, SIZES["equal"], 20 + P)
    a, b = _rhs(ctx, host), _rhs(ctx, _spoiled(ctx, host))
    assert np.isfinite(a).all()
    ok = np.isfinite(b)
    assert ok.mean() > 0.6
    for v in range(9):
        scale = np.abs(a[v]).reshape(ctx.n_elem, -1).max(1)
        err = np.where(ok[v], np.abs(a[v] - b[v]), 0.0).reshape(ctx.n_elem, -1).max(1)
        assert (err <= 1e-12 * scale).all(), (v, err / scale)
    ctx.close()


def test_box_volume_exponents(ffe):  # noqa: F811
    """The right-hand side is homogeneous of degree 1 in the state: bit by bit under powers of two."""
    ctx = ffe.Context(_box(5))
    host = _state(ctx, SIZES["unequal"], 3)
    a = _rhs(ctx, host)
    for k in (-400, -3, 300):
        assert np.array_equal(_rhs(ctx, np.ldexp(host, k)), np.ldexp(a, k)), k
    ctx.close()


@pytest.mark.parametrize("P,b", [(3, 2.0), (4, 50.0), (5, 2.0), (6, 8.0)])
def test_filtered_step(ffe, P, b):  # noqa: F811
    """One step; b sets how many modes the filter damps (2: all but the mean)."""
    cfg = W.fast_wave(n=4, P=P)
    cfg["n"] = (4, 2, 2)
    cfg["params"].update(filter_on=1, filter_b=b, tci_on=0)
    pr = Problem(cfg)
    st = pr.initial_state()
    ctx = ffe.Context(cfg)
    ctx.set_initial()
    ctx.step(1)
    U, _ = ctx.download()
    compare_state(ctx, U, Stepper(pr).step(st), 1e-11)
    ctx.close()


# One component of B~ far above all others: it enters the equations of two components of E~ and of
# phi~ only, and the others have to be as accurate as without it.
GUIDE = np.array([1e-3, 1, 1e-3, 1e8, 1, 1, 1e-10, 1e-10, 1e-2])


def _terms(q, k):
    """Variable (9..11: J~) whose derivative along axis k enters equation q."""
    if q < 6:
        own = q % 3 == k
        return (6 if q < 3 else 7) if own else (3 if q < 3 else 0) + 3 - q % 3 - k
    return k if q == 6 else (3 + k if q == 7 else 9 + k)


def _component_bound(dg, eta, P, widths):
    """2^-49 of every line's |D u| bound, and of the equation's own variable on it (the lift), per
    equation and element: the box comparison's tolerance with each line's own variable and axis."""
    E, B = dg[0:3], dg[3:6]
    B2, EB = (B ** 2).sum(0), (E * B).sum(0)
    Jd = dg[8] * np.cross(E, B, axis=0) / B2
    J = Jd + eta * (EB / B2 * B + np.maximum((E ** 2).sum(0) / B2 - 1, 0) * E)
    top = lambda x: np.abs(x).reshape(len(x), x.shape[1], -1).max(2)  # noqa: E731
    m = np.concatenate([top(dg), top(J)])
    D = np.abs(Tables(P).D).sum(1).max()
    src = np.concatenate([top(Jd), np.zeros_like(m[:3]), m[8:9], np.zeros_like(m[:2])])
    return 2.0 ** -49 * np.array([sum(2.0 / widths[k] * D * (m[_terms(q, k)] + m[q]) for k in range(3)) + src[q] for q in range(9)])


@pytest.mark.parametrize("P", [2, 3, 5, 6])
def test_box_components(ffe, P):  # noqa: F811
    cfg = _box(P)
    cfg.update(hi=tuple(l + w for l, w in zip(cfg["lo"], (0.9, 0.002, 70.0))))
    cfg["params"]["tci_on"] = 0
    ctx = ffe.Context(cfg)
    host = _state(ctx, GUIDE, 40 + P)
    a, b = _rhs(ctx, host), _rhs(ctx, _spoiled(ctx, host))
    dg = ctx.split(host)[0]
    ctx.close()
    bound = _component_bound(dg, 7.0, P, [(hi - lo) / n for n, lo, hi in zip(cfg["n"], cfg["lo"], cfg["hi"])])
    for v in range(9):
        err = np.where(np.isfinite(b[v]), np.abs(a[v] - b[v]), 0.0).reshape(a.shape[1], -1).max(1)
        assert np.isfinite(b[v]).mean() > 0.5 and (err <= bound[v]).all(), (v, err / bound[v])


@pytest.mark.parametrize("P", [3, 5])
def test_shell_components(ffe, P):  # noqa: F811
    """As on a box, with the largest |d xi^k/d x^i| of the mesh for the widths, on elements off the
    boundaries (the star's state mixes components)."""
    cfg = W.pulsar(r_lc=3.0, chi=0.4, n_ang=1, n_rad=3, P=P, r_out=4.0)
    cfg["params"]["eta"] = 7.0
    ctx = ffe.Context(cfg)
    host = _state(ctx, GUIDE, 50 + P)
    a, b = _rhs(ctx, host), _rhs(ctx, _spoiled(ctx, host))
    dg = ctx.split(host)[0]
    ctx.close()
    disc = Problem(cfg).disc
    inner = (disc.nbr >= 0).all(1)
    g = np.abs(disc.ijac).reshape(3, 3, -1).max(2).sum()
    bound = _component_bound(dg, 7.0, P, [2.0 / g] * 3)
    for v in range(8):
        ok = np.isfinite(b[v][inner])
        err = np.where(ok, np.abs(a[v] - b[v])[inner], 0.0).reshape(inner.sum(), -1).max(1)
        assert ok.mean() > 0.3 and (err <= bound[v][inner]).all(), (v, err / bound[v][inner])


def test_box_volume_tiny(ffe):  # noqa: F811
    """Values below 2^-900 are differentiated as well as larger ones (J~ = 0 here)."""
    cfg = _box(5)
    cfg["params"]["eta"] = 0.0
    ctx = ffe.Context(cfg)
    host = _state(ctx, np.where(np.arange(9) == 8, 0.0, 1.0), 4)
    a, b = _rhs(ctx, host), _rhs(ctx, np.ldexp(host, -950))
    ctx.close()
    assert np.abs(np.ldexp(b, 950) - a).max() <= 1e-13 * np.abs(a).max()


def _filter_reference(u, P, a, b):
    """The filter of fields [..., k, j, i] in extended precision."""
    ld = np.longdouble
    x, n = Tables(P).x.astype(ld), P + 1

    def leg(t):
        p = [np.ones_like(t), t]
        for k in range(2, n):
            p.append(((2 * k - 1) * t * p[-1] - (k - 1) * p[-2]) / ld(k))
        return p
    for _ in range(3):   # Newton on (1 - x^2) P_P'(x), interior nodes
        p = leg(x[1:-1])
        dp = P * (p[P - 1] - x[1:-1] * p[P]) / (1 - x[1:-1] ** 2)
        x[1:-1] -= dp * (1 - x[1:-1] ** 2) / (2 * x[1:-1] * dp - P * (P + 1) * p[P])
    V = np.stack(leg(x), axis=1)
    w = 2 / (ld(P) * (P + 1) * V[:, P] ** 2)
    gamma = np.array([2 / ld(2 * m + 1) for m in range(P)] + [2 / ld(P)])
    sigma = np.exp(-ld(a) * (np.arange(n).astype(ld) / P) ** (2 * b))
    F = (V * sigma) @ (V * w[:, None] / gamma).T
    u = u.astype(ld)
    for ax in (-1, -2, -3):
        u = np.moveaxis(np.moveaxis(u, ax, -1) @ F.T, -1, ax)
    return u


@pytest.mark.parametrize("P,quanta", [(3, 1.0), (5, 1.6), (6, 3.9)])
def test_filter_corner(ffe, P, quanta):  # noqa: F811
    """A step of negligible length is the filter.  Fields that fall by 10^4 across an element, at the
    nodes of its low corner: root-mean-square error, in units of 2^-56 of the variable's largest value.
    Three axes of 2, 2 and 3 damped modes round values to one such unit (P = 6: two) and coefficients
    to 1, 2 and 2 of them, each uniformly: sqrt(3 n (1 + c^2)/12)."""
    cfg = W.fast_wave(n=3, P=P)
    cfg["n"] = (3, 2, 2)
    cfg["params"].update(eta=0.0, kappa_psi=0.0, kappa_phi=0.0, filter_on=1, tci_on=0, cfl=1e-40)
    ctx = ffe.Context(cfg)
    ctx.set_initial()
    n = P + 1
    s = 10.0 ** (-4.0 * np.add.outer(np.add.outer(np.arange(n), np.arange(n)), np.arange(n)) / (3 * P))
    dg = s * (1.0 + 0.3 * np.random.default_rng(P).normal(size=(9, ctx.n_elem, n, n, n)))
    ctx.set_state(torch.from_numpy(ctx.join(dg, np.zeros((9, ctx.n_elem) + (ctx.nc,) * 3))).cuda(),
                  torch.zeros(ctx.n_elem, dtype=torch.uint8, device="cuda"))
    ctx.step(1)
    got = ctx.split(ctx.download()[0])[0]
    ctx.close()
    err = np.abs(got - _filter_reference(dg, P, cfg["params"]["filter_a"], cfg["params"]["filter_b"])).astype(float)
    low = err[..., s < 0.1] / np.abs(dg).reshape(9, ctx.n_elem, -1).max(2)[..., None]
    rms = np.sqrt((low ** 2).mean())
    assert rms <= quanta * 2.0 ** -56, rms * 2.0 ** 56
