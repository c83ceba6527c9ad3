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
