"""FD face values from whole lines of cells (k_fd_flux, k_fd_states) against the
oracle, over the orders, reconstructions and the corrector, on meshes with
unequal element widths and every kind of neighbour (random masks)."""
import numpy as np
import pytest

import ffe_workloads as W
from oracle.problem import Problem
from test_gpu_parity import _rhs_parity, ffe  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


def _random_state(pr, P, seed):
    rng = np.random.default_rng(seed)
    E = pr.disc.E
    mask = (rng.random(E) < 0.6).astype(np.uint8)
    return dict(mask=mask, udg=rng.normal(size=(9, E) + (P + 1,) * 3) + 1.0,
                ufd=rng.normal(size=(9, E) + (2 * P + 1,) * 3) + 1.0)


@pytest.mark.parametrize("P", [3, 4, 6])
@pytest.mark.parametrize("recon", [0, 1])
@pytest.mark.parametrize("corr", [0, 1])
def test_box_lines(ffe, P, recon, corr):  # noqa: F811
    cfg = W.breakdown(nx=3, ny=2, nz=1, P=P, x_half=0.1)
    cfg.update(lo=(-0.16, -0.05, -0.2), hi=(0.14, 0.07, 0.1))
    cfg["params"].update(eta=7.0, recon=recon, fd_corrector=corr)
    pr = Problem(cfg)
    assert _rhs_parity(ffe, cfg, _random_state(pr, P, 10 * P + 2 * recon + corr), pr) <= 1e-11


@pytest.mark.parametrize("P,recon,corr", [(3, 0, 1), (4, 0, 0), (4, 1, 1), (5, 0, 1)])
def test_shell_lines(ffe, P, recon, corr):  # noqa: F811
    cfg = W.pulsar(r_lc=3.0, chi=0.4, n_ang=1, n_rad=3, P=P, r_out=4.0)
    cfg["params"].update(eta=7.0, recon=recon, fd_corrector=corr)
    pr = Problem(cfg)
    assert _rhs_parity(ffe, cfg, _random_state(pr, P, 77 + P), pr) <= 1e-11


@pytest.mark.parametrize("kind", ["constant", "spread", "steps", "large"])
def test_box_lines_indicators(ffe, kind):  # noqa: F811
    """Smoothness indicators that are equal, 1e-50 apart, zero next to order one, or of order 1e30."""
    cfg = W.breakdown(nx=3, ny=2, nz=1, P=4, x_half=0.1)
    cfg["params"].update(eta=0.0, recon=0, fd_corrector=0)
    pr = Problem(cfg)
    st = _random_state(pr, 4, 5)
    rng = np.random.default_rng(6)
    st["mask"][:] = 1
    u = st["ufd"]
    if kind == "constant":
        u[:] = np.arange(1.0, 10.0)[:, None, None, None, None]
    elif kind == "spread":
        u *= 10.0 ** rng.uniform(-25.0, 0.0, size=u.shape)
    elif kind == "steps":
        # heights at random, q~ = 0: between two heights, and in rounded values such as J~,
        # b_0 - b_2 cancels and the last bit of the values decides the weights
        u[:] = np.where(rng.random(u.shape) < 0.4, 1.0 + rng.random(u.shape), 1.0)
        u[8] = 0.0
    else:
        u *= 1e15
    assert _rhs_parity(ffe, cfg, st, pr) <= 1e-11
