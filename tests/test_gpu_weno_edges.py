"""WENO5-Z face values where the indicators are equal, vanish or differ by many
orders of magnitude: the line kernels (boxes, flat and Kerr-Schild shells, the
allocation-free entry point) on data of few heights, where b_0 - b_2 is exactly
zero beside a flat middle."""
import numpy as np
import pytest

import ffe_workloads as W
from oracle.fd import rhs_fd, weno5z
from oracle.problem import Problem
from test_gpu_parity import ffe  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GH = 3


def _plateaus(kind, shape, rng):
    """Fields [..., z, y, x] of two or three heights, or of plateaus whose middle cell is one
    rounding higher (along every axis every window of five cells is then symmetric or has a jump
    on one side only)."""
    if kind == "two":
        return rng.integers(1, 3, size=shape).astype(float)
    if kind == "three":
        return rng.integers(0, 3, size=shape).astype(float)
    z, y, x = np.meshgrid(*[np.arange(n) for n in shape[-3:]], indexing="ij")
    row = np.array([2.0, 1.0, 1.0 + 2.0 ** -52, 1.0])
    return np.broadcast_to(row[(x + y + 2 * z) % 4], shape).copy()


def _flux(u, k):
    """Flat flux along axis k of the first eight variables, J~ = 0."""
    i, j = (k + 1) % 3, (k + 2) % 3
    f = np.zeros_like(u)
    f[k], f[3 + k], f[6], f[7] = u[6], u[7], u[k], u[3 + k]
    f[i], f[j], f[3 + i], f[3 + j] = u[3 + j], -u[3 + i], -u[j], u[i]
    return f


def _block_rhs(ext, h, eps):
    """Right-hand side of extended blocks [9][E][ne^3] with eta = q~ = 0 and no corrector, in
    extended precision."""
    u = ext.astype(np.longdouble)
    n = ext.shape[-1] - 2 * GH
    out = np.zeros(u.shape[:2] + (n,) * 3, np.longdouble)
    for k in range(3):
        ax = 4 - k
        idx = [slice(None), slice(None)] + [slice(GH, GH + n)] * 3

        def cells(o):
            idx[ax] = slice(GH + o, GH + o + n + 1)
            return u[tuple(idx)]
        v = [cells(o) for o in range(-3, 3)]
        L, R = weno5z(*v[:5], np.longdouble(eps)), weno5z(*v[:0:-1], np.longdouble(eps))
        F = 0.5 * (_flux(L, k) + _flux(R, k)) - 0.5 * (R - L)
        out -= np.diff(F, axis=ax) * (np.longdouble(n) / h[k])
    return out


def _noalloc(ffe, P, ext, h, eps):  # noqa: F811
    out = torch.full(ext.shape[:2] + (2 * P + 1,) * 3, float("nan"), dtype=torch.float64, device="cuda")
    ffe.fd_rhs_noalloc(P, torch.from_numpy(ext).cuda(), h, 0.0, eps, 0, out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


H = (0.25, 0.5, 1.0)


@pytest.mark.parametrize("kind", ["two", "three", "ulp"])
def test_blocks_plateaus(ffe, kind):  # noqa: F811
    """Bound: 6 face fluxes of two values, each within 16 roundings of the largest cell."""
    P = 4
    rng = np.random.default_rng(3)
    ext = _plateaus(kind, (9, 2) + (2 * P + 7,) * 3, rng)
    ext[8] = 0.0
    err = np.abs(_noalloc(ffe, P, ext, H, 1e-40) - _block_rhs(ext, H, 1e-40)).max()
    assert err <= 2.0 ** -53 * 6 * 2 * 16 * 2.0 * (2 * P + 1) / min(H), err


@pytest.mark.parametrize("mesh", ["box", "shell", "kerr-schild"])
@pytest.mark.parametrize("kind", ["two", "three"])
def test_plateaus(ffe, mesh, kind):  # noqa: F811
    """Cells that reach only cells of their own element: the oracle's ghosts on a box carry an
    interpolation's rounding, which decides the weights of a plateau."""
    P = 5
    if mesh == "box":
        cfg = W.breakdown(nx=2, ny=2, nz=1, P=P, x_half=0.1)
    elif mesh == "shell":
        cfg = W.pulsar(r_lc=3.0, chi=0.4, n_ang=1, n_rad=2, P=P, r_out=4.0)
    else:
        cfg = W.wald(spin=0.7, n_ang=1, n_rad=2, P=P)
    cfg["params"].update(eta=0.0, recon=0, fd_corrector=0, tci_on=1)
    pr = Problem(cfg)
    E, n = pr.disc.E, 2 * P + 1
    u = _plateaus(kind, (9, E, n, n, n), np.random.default_rng(4))
    u[8] = 0.0
    u[3] += 3.0   # B~ does not vanish
    st = dict(mask=np.ones(E, np.uint8), udg=np.ones((9, E) + (P + 1,) * 3), ufd=u)
    ctx = ffe.Context(cfg)
    ctx.set_initial()
    U = torch.from_numpy(ctx.join(st["udg"], u)).cuda()
    ctx.set_state(U, torch.ones(E, dtype=torch.uint8, device="cuda"))
    out = torch.zeros_like(U)
    ctx.rhs(U, out)
    torch.cuda.synchronize()
    got = ctx.split(out.cpu().numpy())[1]
    ctx.close()
    own = (slice(None), slice(None)) + (slice(3, n - 3),) * 3
    ref = rhs_fd(st, pr.disc, pr.met, pr.prm)[own]
    assert np.abs(got[own] - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("h", [1e-6, 1e-12])
def test_blocks_beside_jump(ffe, h, axis):  # noqa: F811
    """Cells of size h beside cells of order one: away from the jump's own face, errors are roundings
    of h, not of the jump.  1e-12: a face value of random cells moves by up to 300 of its roundings
    with those of the indicators, two of which are subtracted."""
    P = 4
    n = 2 * P + 1
    rng = np.random.default_rng(8 + axis)
    shape = (9, 2) + (2 * P + 7,) * 3
    c = np.arange(2 * P + 7).reshape([-1 if a == 2 - axis else 1 for a in range(3)])
    ext = np.where(c < GH + 5, h * (1.0 + 0.1 * rng.normal(size=shape)), 2.0 + rng.random(shape))
    ext[8] = 0.0
    err = np.abs(_noalloc(ffe, P, ext, H, 1e-60) - _block_rhs(ext, H, 1e-60))
    low = np.moveaxis(err, 4 - axis, 0)[:4]   # the fifth cell's flux crosses the jump
    assert low.max() <= 1e-12 * 1.5 * h * n / min(H), low.max()


@pytest.mark.parametrize("eps", [1e-100, 1e-290])
def test_blocks_small_eps(ffe, eps):  # noqa: F811
    """Cells of 1e-28, whose indicators lie far below 1e-51, with an eps below those: the bound of
    test_blocks_plateaus, with 600 roundings for random cells as above."""
    P = 4
    ext = 1e-28 * (1.0 + 0.1 * np.random.default_rng(5).normal(size=(9, 2) + (2 * P + 7,) * 3))
    ext[8] = 0.0
    err = np.abs(_noalloc(ffe, P, ext, H, eps) - _block_rhs(ext, H, eps)).max()
    assert err <= 2.0 ** -53 * 6 * 2 * 600 * 2e-28 * (2 * P + 1) / min(H), err


def _fd_shell(ffe, weno_eps, scale):  # noqa: F811
    """rhs, its VJP and an adjoint step of a shell of two heights, all on FD; scale: of the state."""
    cfg = W.pulsar(r_lc=3.0, chi=0.4, n_ang=1, n_rad=2, P=4, r_out=4.0)
    cfg["params"].update(eta=0.0, recon=0, tci_on=0, weno_eps=weno_eps)
    ctx = ffe.Context(cfg)
    ctx.set_initial()
    rng = np.random.default_rng(6)
    u = _plateaus("two", (9, ctx.n_elem) + (ctx.nc,) * 3, rng)
    u[8] = 0.0
    U = torch.from_numpy(ctx.join(np.zeros((9, ctx.n_elem) + (ctx.P + 1,) * 3), u)).cuda() * scale
    nd = 9 * ctx.n_dg
    lam = torch.from_numpy(rng.normal(size=U.numel())).cuda()
    lam[:nd] = 0.0
    ctx.set_state(U, torch.ones(ctx.n_elem, dtype=torch.uint8, device="cuda"))
    out = [torch.zeros_like(U) for _ in range(3)]
    ctx.rhs(U, out[0])
    ctx.rhs_vjp(U, lam, out[1])
    ctx.adjoint_step(U, lam, out[2])
    torch.cuda.synchronize()
    ctx.close()
    return [x[nd:].cpu().numpy() for x in out]


def _close(a, b, tol):
    assert np.isfinite(a).all() and np.abs(a - b).max() <= tol * np.abs(b).max(), np.abs(a - b).max() / np.abs(b).max()


def test_shell_eps_scales_with_state(ffe):  # noqa: F811
    """With eta = q~ = 0 the right-hand side is of degree 1 in (state, sqrt(eps)) and its derivative of
    degree 0; the VJPs add contributions in any order."""
    s = 2.0 ** -93
    a, b = _fd_shell(ffe, 1e-40, 1.0), _fd_shell(ffe, 1e-40 * s * s, s)
    assert np.array_equal(a[0] * s, b[0])
    _close(b[1], a[1], 1e-12)
    _close(b[2], a[2], 1e-9)


def test_shell_zero_eps(ffe):  # noqa: F811
    """eps = 0 (allowed without the indicator): flat stencils take the ideal weights, in the step, its
    recomputation and its reverse."""
    a, b = _fd_shell(ffe, 1e-60, 1.0), _fd_shell(ffe, 0.0, 1.0)
    _close(b[0], a[0], 1e-12)
    _close(b[1], a[1], 1e-12)
    _close(b[2], a[2], 1e-9)
