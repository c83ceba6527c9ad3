"""Performance cases of the library: what its users run, through the public
entry points of paper_2404_01531_gb300.ffe, from the smallest meshes (launch
latency) to the largest of the workloads (FP64 throughput).

  rhs      ffe_rhs on a box: any mask of DG elements and FD subcells
  step     ffe_step on a box: IMEX steps, the mask fixed or the indicator on
  shell    ffe_step on a rotating-dipole shell (curved elements, flat metric)
  wald     ffe_step on a Kerr-Schild shell (the metric-general kernels)
  batch    ffe_step of many shells of different sizes and orders together
  adjoint  ffe_adjoint_step: one step backward on a shell
  vjp      ffe_rhs_vjp: the vector-Jacobian product of the right-hand side
  blocks   ffe_fd_rhs_noalloc on caller-built extended blocks

A stepping pass starts from the same state each time (ffe_set_state, then
ffe_step), as a restarted or a swept run does.  States are the closed-form data
of the workloads plus a smooth seeded perturbation of every variable, relaxed
to nearly force-free (E.B = 0) as every state behind a stiff solve is.

exact() restates the box operators and the IMEX step in plain torch, FP64 like
the library itself.  Shells, batches and the adjoint have no value there: their
plain form is a whole second solver (wedge maps, the 3+1 metric, the reverse
mode), and the tests compare them with one.
"""
import math
import random

import numpy as np
import torch

from paper_2404_01531_gb300 import ffe

DIRICHLET, PERIODIC = "dirichlet", "periodic"
AMP = (0.02, 0.02, 0.02, 0.02, 0.02, 0.02, 0.01, 0.01, 0.05)   # perturbation of each variable


def listed():
    return [
        # one right-hand side of a very small ragged box: an outer integrator's
        # smallest call, all launch latency
        dict(name="rhs_tiny_60", kind="rhs", flow="wave", n0=5, n1=4, n2=3, P=4, fd=0.0, recon=0, corr=0),
        # the paper's 1-D Alfven test at its second resolution: 64 elements,
        # thousands of short steps, so launches and latency count
        dict(name="step_alfven1d_64", kind="step", flow="alfven", n0=64, n1=1, n2=1, P=5, fd=0.0, recon=0, corr=1,
             tci=1, mode=0, steps=4),
        # the smooth wave in a periodic cube, every element on DG: the DG
        # substep at a size that fills the chip
        dict(name="step_wave_4096", kind="step", flow="wave", n0=16, n1=16, n2=16, P=5, fd=0.0, recon=0, corr=0,
             tci=1, mode=0, steps=2),
        # the current sheet of the benchmark at full size: DG with a slab of FD
        # subcells, indicator and switching on
        dict(name="step_breakdown_4096", kind="step", flow="breakdown", n0=64, n1=8, n2=8, P=5, fd=0.07, recon=0,
             corr=1, tci=1, mode=0, steps=2),
        # the same sheet on an odd mesh with the MP5 reconstruction and the
        # algebraic constraint clamp
        dict(name="step_hard_mp5_775", kind="step", flow="breakdown", n0=31, n1=5, n2=5, P=5, fd=0.16, recon=1,
             corr=1, tci=0, mode=1, steps=1),
        # DG/FD split of a stationary wave at order 4: half the right-hand side's
        # elements on FD, odd sizes
        dict(name="rhs_split_441", kind="rhs", flow="alfven", n0=9, n1=7, n2=7, P=4, fd=0.5, recon=0, corr=1),
        # rotating-dipole shell, the innermost layers on FD subcells: curved DG
        # and FD kernels and the ghosts between wedges
        dict(name="step_shell_1200", kind="shell", n_ang=5, n_rad=8, P=5, layers=2, corr=0, steps=1),
        # black-hole shell in Kerr-Schild coordinates, all DG
        dict(name="step_wald_1536", kind="wald", n_ang=4, n_rad=16, P=5, spin=0.9, spheroidal=1, steps=1),
        # a parameter sweep: pulsars of different orders and sizes in one context
        dict(name="step_batch_8", kind="batch", count=8, n_ang=4, n_rad=10, mix=1, steps=2),
        # one step of the adjoint run of a luminosity gradient, hybrid mask
        dict(name="adjoint_shell_324", kind="adjoint", n_ang=3, n_rad=6, P=5, layers=1, corr=0),
        # right-hand side of caller-owned FD blocks, the most one call takes
        dict(name="blocks_19", kind="blocks", P=5, count=19, corr=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rhs", "rhs", "step", "step", "step", "shell", "wald", "batch", "adjoint", "vjp", "blocks"])
    if kind in ("rhs", "step"):
        flow = rng.choice(["wave", "alfven", "breakdown"])
        P = rng.choice([3, 4, 5, 5, 5, 6])
        E = _log_int(rng, 24, 2000 if P < 6 else 1000)
        n1 = rng.randint(1, max(1, min(9, int(E ** (1 / 3)))))
        n2 = rng.randint(1, max(1, min(9, int(E ** (1 / 3)))))
        n0 = max(4, min(96, E // (n1 * n2)))
        E = n0 * n1 * n2
        # FD elements cost some thirty times a DG element: at most 150 of them
        fd = rng.choice([0.0, rng.uniform(0.02, 1.0)]) * min(1.0, 150.0 / E)
        c = dict(kind=kind, flow=flow, n0=n0, n1=n1, n2=n2, P=P, fd=round(fd, 4), recon=rng.choice([0, 0, 0, 1]),
                 corr=rng.randint(0, 1))
        if kind == "step":
            c.update(tci=rng.randint(0, 1), mode=rng.choice([0, 0, 1, 2]), steps=rng.randint(1, 2))
        return c
    if kind == "shell":
        return dict(kind=kind, n_ang=rng.randint(1, 6), n_rad=rng.randint(4, 10), P=rng.choice([3, 4, 5]),
                    layers=rng.randint(0, 1), corr=rng.randint(0, 1), steps=rng.randint(1, 2))
    if kind == "wald":
        return dict(kind=kind, n_ang=rng.choice([1, 2, 3, 4, 5]), n_rad=rng.randint(4, 16), P=rng.choice([3, 4, 5]),
                    spin=round(rng.uniform(0.0, 0.95), 3), spheroidal=rng.randint(0, 1), steps=rng.randint(1, 2))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 10), n_ang=rng.randint(3, 5), n_rad=rng.randint(10, 12),
                    mix=rng.randint(1, 10 ** 6), steps=1)
    if kind == "blocks":
        P = rng.choice([3, 4, 5, 6])
        return dict(kind=kind, P=P, count=rng.randint(1, _blocks_cap(P)), corr=rng.randint(0, 1))
    return dict(kind=kind, n_ang=rng.randint(1, 3), n_rad=rng.randint(4, 8), P=rng.choice([3, 4, 5]),
                layers=rng.randint(0, 1), corr=rng.randint(0, 1))


def _blocks_cap(P):
    nc = 2 * P + 1
    return (1 << 20) // (3 * (nc + 6) ** 3 + 27 * (nc + 1) * nc * nc)


# ---- 1-D tables ------------------------------------------------------------------

def _lgl(N):
    """Legendre-Gauss-Lobatto nodes and weights of order N."""
    c = np.zeros(N + 1)
    c[N] = 1.0
    dc = np.polynomial.legendre.legder(c)
    d2c = np.polynomial.legendre.legder(dc)
    x = np.concatenate([[-1.0], np.sort(np.polynomial.legendre.legroots(dc).real), [1.0]])
    for _ in range(4):
        x[1:-1] -= np.polynomial.legendre.legval(x[1:-1], dc) / np.polynomial.legendre.legval(x[1:-1], d2c)
    x = 0.5 * (x - x[::-1])
    return x, 2.0 / (N * (N + 1) * np.polynomial.legendre.legval(x, c) ** 2)


def _lagrange(xs, y):
    """Rows: the Lagrange polynomials through xs at each point of y."""
    out = np.ones((len(y), len(xs)))
    for j in range(len(xs)):
        for m in range(len(xs)):
            if m != j:
                out[:, j] *= (y - xs[m]) / (xs[j] - xs[m])
    return out


def _centres(nc):
    return -1.0 + (np.arange(nc) + 0.5) * 2.0 / nc


def _fd2dg(P):
    """6-point Lagrange through the nearest subcell centres, the stencil kept inside."""
    nc = 2 * P + 1
    x, xc = _lgl(P)[0], _centres(nc)
    out = np.zeros((P + 1, nc))
    for i in range(P + 1):
        lo = min(max(int(math.floor((x[i] + 1.0) * nc / 2.0 - 0.5)) - 2, 0), nc - 6)
        out[i, lo:lo + 6] = _lagrange(xc[lo:lo + 6], x[i:i + 1])[0]
    return out


# ---- boxes -----------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


class _Box:
    """Mesh, flow and perturbation of a box case; arrays are [..., z, y, x, k, j, i]."""

    def __init__(self, case, seed):
        self.c = case
        self.P, self.np1, self.nc = case["P"], case["P"] + 1, 2 * case["P"] + 1
        self.n = (case["n0"], case["n1"], case["n2"])
        self.E = self.n[0] * self.n[1] * self.n[2]
        h = {"wave": 2.0, "alfven": 3.0}.get(case["flow"], case["n0"] / 16.0) / case["n0"]
        self.h = h
        self.lo = tuple(-0.5 * h * k for k in self.n)
        self.hi = tuple(0.5 * h * k for k in self.n)
        self.bc = (PERIODIC if case["flow"] == "wave" else DIRICHLET, PERIODIC, PERIODIC)
        self.x1, self.w1 = _lgl(self.P)
        self.dt = 0.3 * 0.4186 * h * float(self.x1[1] - self.x1[0]) / 2.0
        # the conductivity of the workloads: 1e6 where the Alfven layer is resolved (the 1-D tests)
        self.driver = 1e3 if case["flow"] != "alfven" else 1e6 if case["n0"] >= 32 else 1e5
        self.eta = 0.0 if case.get("mode") == 1 else self.driver
        r = random.Random(seed)
        self.modes = [[(r.randint(-2, 2), r.randint(-1, 1), r.randint(-1, 1), r.uniform(0.0, 2.0 * math.pi),
                        AMP[v] * r.uniform(0.4, 1.0)) for _ in range(2)] for v in range(9)]
        # FD slab: the columns of elements nearest the middle of the x range
        k = int(round(case["fd"] * self.n[0]))
        k = max(k, 1) if case["fd"] > 0 else 0
        first = (self.n[0] - k) // 2
        col = torch.zeros(self.n[0], dtype=torch.uint8)
        col[first:first + k] = 1
        self.mask = col.repeat(self.n[1] * self.n[2])

    def config(self):
        c = self.c
        prm = dict(eta=self.driver, kappa_psi=1.0, kappa_phi=1.0, cfl=0.3, c_over_D=0.4186, dt=self.dt,
                   filter_on=1, filter_a=36.0, filter_b=50.0, tci_on=c.get("tci", 0), tci_M=3, tci_alpha=4.0,
                   weno_eps=1e-40, fd_corrector=c["corr"], constraint_mode=c.get("mode", 0), omega_star=0.0,
                   recon=c["recon"])
        initial = {"wave": ("fast_wave", dict(amp=0.5)), "alfven": ("alfven", {}), "breakdown": ("breakdown", {})}
        return dict(kind="box", lo=self.lo, hi=self.hi, n=self.n, bc=self.bc, P=self.P,
                    metric=("minkowski", 0.0, 0.0), params=prm, initial=initial[c["flow"]])

    def points(self, ref):
        """Coordinates per axis at the reference points `ref` of every element, broadcastable to [z, y, x, k, j, i]."""
        out = []
        for a in range(3):
            e = torch.arange(self.n[a], dtype=torch.float64, device=_device())
            t = torch.as_tensor(ref, dtype=torch.float64, device=_device())
            x = self.lo[a] + self.h * (e[:, None] + 0.5 * (t[None, :] + 1.0))
            shape = [1] * 6
            shape[2 - a], shape[5 - a] = self.n[a], len(ref)
            out.append(x.reshape(shape))
        return out

    def flow(self, x):
        """The workload's closed form (9 variables) at x (any shape)."""
        U = torch.zeros((9,) + tuple(x.shape), dtype=torch.float64, device=x.device)
        U[3] = 1.0
        if self.c["flow"] == "wave":
            b = 1.0 + 0.5 * torch.sin(math.pi * x)
            U[4], U[2] = b, -b
        elif self.c["flow"] == "alfven":
            inside = x.abs() < 0.1
            b = torch.where(inside, 1.15 + 0.15 * torch.sin(5.0 * math.pi * x), 1.0 + 0.3 * (x > 0).to(x.dtype))
            U[0], U[2], U[4], U[5] = -b, 1.0, 1.0, b
            U[8] = torch.where(inside, -0.75 * math.pi * torch.cos(5.0 * math.pi * x), 0.0)
        else:
            U[4] = torch.where(x < -0.1, 1.0, torch.where(x > 0.1, -1.0, -10.0 * x))
            U[2] = torch.where(x.abs() < 0.1, 0.5, 1.0)
        return U

    def state_at(self, ref):
        xs = self.points(ref)
        U = self.flow(xs[0]).expand(9, *torch.broadcast_shapes(*(x.shape for x in xs))).clone()
        ph = [2.0 * math.pi * (x - l) / (h - l) for x, l, h in zip(xs, self.lo, self.hi)]
        window = 1.0 if self.bc[0] == PERIODIC else torch.sin(0.5 * ph[0]) ** 2
        for v in range(9):
            for kx, ky, kz, shift, amp in self.modes[v]:
                U[v] += amp * window * torch.cos(kx * ph[0] + ky * ph[1] + kz * ph[2] + shift)
        return _relaxed(U)

    def state(self):
        """(U, mask): the state vector, zero in the blocks an element does not use."""
        dg = self.state_at(self.x1).reshape(9, self.E, -1)
        fd = self.state_at(_centres(self.nc)).reshape(9, self.E, -1)
        m = self.mask.to(dg.device)
        dg[:, m != 0] = 0.0
        fd[:, m == 0] = 0.0
        return torch.cat([dg.reshape(-1), fd.reshape(-1)]), m


def _relaxed(U):
    """E with all but a thousandth of its part along B taken out, as behind a stiff solve."""
    E, B = U[0:3], U[3:6]
    U[0:3] = E - 0.999 * ((E * B).sum(0) / (B * B).sum(0)) * B
    return U


# ---- shells ----------------------------------------------------------------------

def _shell_config(case, r_lc=6.0, chi=math.pi / 4, mu=1.0, n_ang=None, n_rad=None, P=None, r_out=24.0):
    prm = dict(eta=1e5, kappa_psi=1.0, kappa_phi=1.0, cfl=0.25, c_over_D=0.4186, filter_on=1, filter_a=36.0,
               filter_b=50.0, tci_on=1 if case["kind"] == "batch" else 0, tci_M=3, tci_alpha=4.0, weno_eps=1e-40,
               fd_corrector=case.get("corr", 0), constraint_mode=0, omega_star=1.0 / r_lc)
    return dict(kind="shell", r_in=1.0, r_out=r_out, n_ang=n_ang or case["n_ang"], n_rad=n_rad or case["n_rad"],
                bc_inner="star", bc_outer="no_incoming", P=P or case["P"], metric=("minkowski", 0.0, 0.0), params=prm,
                initial=("dipole", dict(mu=mu, delta=0.1, chi=chi)))


def _perturb_shell(U, ctx, rng):
    """Smooth relative perturbation of a single shell's state (U changed in place)."""
    xd, xf = ctx.coords()
    cut = 9 * ctx.n_dg
    for x, u in ((xd, U[:cut].view(9, -1)), (xf, U[cut:].view(9, -1))):
        r = x.square().sum(0).sqrt()
        scale = u[3:6].square().sum(0).sqrt()
        n = x / r
        for v in range(9):
            k = [rng.uniform(-2.0, 2.0) for _ in range(3)]
            rad, shift = rng.uniform(0.5, 1.5), rng.uniform(0.0, 2.0 * math.pi)
            u[v] += AMP[v] * scale * torch.cos(k[0] * n[0] + k[1] * n[1] + k[2] * n[2] + rad * r.log() + shift)
        _relaxed(u)


def _shell_state(case, seed):
    """Context on the rotating-dipole shell with its innermost layers on FD, and the state of the pass."""
    r = random.Random(seed)
    ctx = ffe.Context(_shell_config(case, chi=r.uniform(0.3, 1.2), mu=r.uniform(0.8, 1.2)))
    layer = torch.arange(ctx.n_elem, device="cuda") % (case["n_rad"] * case["n_ang"] ** 2) // case["n_ang"] ** 2
    mask = (layer < case["layers"]).to(torch.uint8)
    ctx.set_state(torch.zeros(ctx.n_state, dtype=torch.float64, device="cuda"), mask)
    ctx.set_initial(keep_mask=True)
    U = ctx.state()[0].clone()
    # one perturbation for both representations: the same numbers for the nodes and the cells
    _perturb_shell(U, ctx, _Repeat(r))
    on_fd = mask != 0
    cut = 9 * ctx.n_dg
    U[:cut].view(9, ctx.n_elem, -1)[:, on_fd] = 0.0
    U[cut:].view(9, ctx.n_elem, -1)[:, ~on_fd] = 0.0
    return ctx, U, mask, r


class _Repeat:
    """A stream of uniform numbers that starts again after the 45 one representation's perturbation takes."""

    def __init__(self, rng):
        self.u, self.i = [rng.random() for _ in range(45)], 0

    def uniform(self, a, b):
        self.i += 1
        return a + (b - a) * self.u[(self.i - 1) % 45]


def _batch_configs(case, seed):
    shape, r = random.Random(case["mix"]), random.Random(seed)
    out = []
    for _ in range(case["count"]):
        r_lc = shape.uniform(3.0, 5.0)   # with 10 radial elements or more, the dipole's profile stays on DG
        out.append(_shell_config(case, r_lc=r_lc, chi=r.uniform(0.0, math.pi / 3), mu=r.uniform(0.8, 1.2),
                                 n_ang=max(3, case["n_ang"] - shape.randint(0, 2)),
                                 n_rad=case["n_rad"] + shape.randint(0, 4), P=shape.choice([4, 5]),
                                 r_out=4.0 * r_lc))
    return out


# ---- preparing and running ----------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("rhs", "step"):
        box = _Box(case, seed)
        ctx = ffe.Context(box.config())
        ctx.set_initial()
        U, mask = box.state()
        ctx.set_state(U, mask)
        return _with_view(dict(case=case, ctx=ctx, U=U, mask=mask, out=torch.zeros_like(U)))
    if kind == "blocks":
        U = _block_state(case, seed).contiguous()
        nc = 2 * case["P"] + 1
        return dict(case=case, U=U, out=torch.zeros(9, case["count"], nc ** 3, dtype=torch.float64, device="cuda"))
    if kind == "wald":
        r = random.Random(seed)
        prm = dict(eta=0.0, kappa_psi=1.0, kappa_phi=1.0, cfl=0.25, c_over_D=0.4186, filter_on=1, filter_a=36.0,
                   filter_b=50.0, tci_on=0, tci_M=3, tci_alpha=4.0, weno_eps=1e-40, fd_corrector=0,
                   constraint_mode=0, omega_star=0.0)
        ks = bool(case["spheroidal"])
        ctx = ffe.Context(dict(kind="shell", r_in=1.0 if ks else 1.9, r_out=125.0 if ks else 50.0,
                               n_ang=case["n_ang"], n_rad=case["n_rad"], bc_inner="outflow" if ks else DIRICHLET,
                               bc_outer="no_incoming" if ks else DIRICHLET, P=case["P"],
                               metric=("kerr_schild", 1.0, case["spin"]), shell_ks=ks, params=prm,
                               initial=("wald", dict(M=1.0, a=case["spin"], B0=r.uniform(0.8, 1.2),
                                                     e=r.uniform(0.0, 1.0)))))
        ctx.set_initial()
    elif kind == "batch":
        cfgs = _batch_configs(case, seed)
        E = sum(6 * c["n_ang"] ** 2 * c["n_rad"] for c in cfgs)
        ctx = ffe.BatchContext(cfgs, fd_capacity=max(16, E // 4))
        ctx.set_initial()
        ctx.freeze_mask(True)
    else:
        ctx, U, mask, r = _shell_state(case, seed)
        if kind == "shell":
            return _with_view(dict(case=case, ctx=ctx, U=U, mask=mask))
        ctx.freeze_mask(True)
        ctx.set_state(U, mask)
        g = torch.Generator(device="cuda").manual_seed(seed)
        lam = torch.randn(ctx.n_state, dtype=torch.float64, device="cuda", generator=g)
        on_fd, cut = mask != 0, 9 * ctx.n_dg
        lam[:cut].view(9, ctx.n_elem, -1)[:, on_fd] = 0.0
        lam[cut:].view(9, ctx.n_elem, -1)[:, ~on_fd] = 0.0
        return dict(case=case, ctx=ctx, U=U, mask=mask, lam=lam, out=torch.zeros_like(lam))
    U, mask = (t.clone() for t in ctx.state())
    return _with_view(dict(case=case, ctx=ctx, U=U, mask=mask))


def _with_view(state):
    """The library's state and mask, borrowed for the life of the context: each
    view holds the context, so that what run() returns outlives the state."""
    state["view"] = list(state["ctx"].state())
    for t in state["view"]:
        t.context = state["ctx"]
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "blocks":
        ffe.fd_rhs_noalloc(case["P"], state["U"], (0.0625, 0.0625, 0.0625), 1e3, 1e-40, case["corr"], state["out"])
        return state["out"]
    ctx = state["ctx"]
    if kind == "rhs":
        ctx.rhs(state["U"], state["out"])
        return state["out"]
    if kind == "adjoint":
        return [state["out"], ctx.adjoint_step(state["U"], state["lam"], state["out"])]
    if kind == "vjp":
        return [state["out"], ctx.rhs_vjp(state["U"], state["lam"], state["out"])]
    ctx.set_state(state["U"], state["mask"])
    ctx.step(case["steps"])
    return state["view"]


# ---- what a pass cannot do without ----------------------------------------------------

def _elements(case):
    """[(elements on DG, elements on FD, order)]"""
    kind = case["kind"]
    if kind == "batch":
        return [(6 * c["n_ang"] ** 2 * c["n_rad"], 0, c["P"]) for c in _batch_configs(case, 0)]
    if kind == "blocks":
        return [(0, case["count"], case["P"])]
    if kind in ("rhs", "step"):
        fd = int(_Box(case, 0).mask.sum())
        return [(case["n0"] * case["n1"] * case["n2"] - fd, fd, case["P"])]
    fd = 6 * case["n_ang"] ** 2 * case.get("layers", 0)
    return [(6 * case["n_ang"] ** 2 * case["n_rad"] - fd, fd, case["P"])]


def work(case):
    """State read and written once; flops (an FMA is 2) of the method: per DG
    node 54 (P+1) for the 27 line contractions of the volume term (162 (P+1) of
    the metric-general one) and 60 for its combination, sources, lift and
    stage, with the filter's two modes and the pointwise solves in a step; per
    FD cell and axis 10 reconstructed values (12 on a shell) at 75 flops, both
    sides of a cell from one set of indicators, and 60 for the flux and its
    difference."""
    kind = case["kind"]
    curved = kind in ("shell", "wald", "batch", "adjoint", "vjp")
    rhs = {"rhs": 1, "blocks": 1, "vjp": 2, "adjoint": 9}.get(kind, 3 * case.get("steps", 1))
    stages = 0 if kind in ("rhs", "blocks", "vjp") else rhs
    flops = values = 0
    for dg, fd, P in _elements(case):
        nodes, cells = dg * (P + 1) ** 3, fd * (2 * P + 1) ** 3
        node = (162 if kind == "wald" else 54) * (P + 1) + 60
        cell = 3 * ((12 if curved else 10) * 75 + 60)
        flops += rhs * (nodes * node + cells * cell) + stages * (nodes * (36 * (P + 1) + 120) + cells * 120)
        values += 9 * (nodes + cells)
    return {"bytes": 8 * values * (3 if kind in ("vjp", "adjoint") else 2), "flops": flops}


# ---- the same in plain torch ------------------------------------------------------------

def _along(M, f, axis):
    """Matrix M applied along the point index of `axis` (0 = x, the last dimension)."""
    return (f.movedim(-1 - axis, -1) @ torch.as_tensor(M, dtype=f.dtype, device=f.device).T).movedim(-1, -1 - axis)


def _tensor3(M, f):
    for a in range(3):
        f = _along(M, f, a)
    return f


def _current(U, eta):
    """(drift, full) current; zero where B = 0."""
    E, B = U[0:3], U[3:6]
    B2 = (B * B).sum(0)
    ib = torch.where(B2 > 0, 1.0 / torch.where(B2 > 0, B2, 1.0), 0.0)
    drift = U[8] * ib * torch.linalg.cross(E, B, dim=0)
    extra = ((E * E).sum(0) - B2).clamp_min(0.0)
    return drift, drift + eta * ib * ((E * B).sum(0) * B + extra * E)


def _flux(U, J, a):
    """Flux along axis a of (U, J)."""
    b, c = (a + 1) % 3, (a + 2) % 3
    F = torch.empty_like(U)
    F[a], F[b], F[c] = U[6], U[3 + c], -U[3 + b]
    F[3 + a], F[3 + b], F[3 + c] = U[7], -U[c], U[b]
    F[6], F[7], F[8] = U[a], U[3 + a], J[a]
    return F


def _weno(v):
    """WENO5-Z value at the right face of v[2] (point values; weights 1, 10, 5)."""
    v0, v1, v2, v3, v4 = v
    p = ((3 * v0 - 10 * v1 + 15 * v2) / 8, (-v1 + 6 * v2 + 3 * v3) / 8, (3 * v2 + 6 * v3 - v4) / 8)
    b = [13 / 12 * s * s + 0.25 * e * e + 1e-40 for s, e in ((v0 - 2 * v1 + v2, v0 - 4 * v1 + 3 * v2),
                                                             (v1 - 2 * v2 + v3, v1 - v3),
                                                             (v2 - 2 * v3 + v4, 3 * v2 - 4 * v3 + v4))]
    w = [d * (1.0 + ((b[0] - b[2]) / bk) ** 2) for d, bk in zip((1.0, 10.0, 5.0), b)]
    return sum(wk * pk for wk, pk in zip(w, p)) / sum(w)


def _minmod(*t):
    t = torch.stack(t)
    return torch.where((t > 0).all(0), t.amin(0), torch.where((t < 0).all(0), t.amax(0), 0.0))


def _mp5(v):
    """Suresh and Huynh's limiter on the 5-point interpolant at the right face of v[2]."""
    v0, v1, v2, v3, v4 = v
    u = (3 * v0 - 20 * v1 + 90 * v2 + 60 * v3 - 5 * v4) / 128
    mp = v2 + _minmod(v3 - v2, 4 * (v2 - v1))
    d1, d2, d3 = v0 - 2 * v1 + v2, v1 - 2 * v2 + v3, v2 - 2 * v3 + v4
    dp, dm = _minmod(4 * d2 - d3, 4 * d3 - d2, d2, d3), _minmod(4 * d2 - d1, 4 * d1 - d2, d2, d1)
    ul, md, lc = v2 + 4 * (v2 - v1), 0.5 * (v2 + v3) - 0.5 * dp, v2 + 0.5 * (v2 - v1) + 4 / 3 * dm
    lo = torch.maximum(torch.minimum(torch.minimum(v2, v3), md), torch.minimum(torch.minimum(v2, ul), lc))
    hi = torch.minimum(torch.maximum(torch.maximum(v2, v3), md), torch.maximum(torch.maximum(v2, ul), lc))
    return torch.where((u - v2) * (u - mp) <= 0, u, u + _minmod(lo - u, hi - u))


def _face_flux(ext, a, recon, corr):
    """Rusanov flux (with the 4th-order corrector) at every face along axis a of
    cells [12, z, y, x] that carry 3 ghost layers along that axis."""
    d = 3 - a
    N = ext.shape[d] - 6
    v = [ext.narrow(d, i, N + 1) for i in range(6)]
    value = _mp5 if recon else _weno
    L, R = value(v[:5]), value(v[:0:-1])
    FL, FR, Fm, Fp = (_flux(s[:9], s[9:], a) for s in (L, R, v[2], v[3]))
    F = 0.5 * (FL + FR) - 0.5 * (R[:9] - L[:9])
    return F - (Fm - 2 * F + Fp) / 6 if corr else F


def _box_rhs(box, dg, fd):
    """Right-hand side (DG blocks, FD blocks) of a box under its mask; the blocks
    of the other representation are not meaningful."""
    P, nc, n, h = box.P, box.nc, box.n, box.h
    on_fd = box.mask.to(dg.device).reshape(n[2], n[1], n[0], 1, 1, 1) != 0
    Jd, Jf = _current(dg, box.eta)
    Kd, Kf = _current(fd, box.eta)
    dg12, fd12 = torch.cat([dg, Jf]), torch.cat([fd, Kf])
    # what the neighbours see: an FD element's nodes, a DG element's cells
    nodes = torch.where(on_fd, _tensor3(_fd2dg(P), fd12), dg12)
    cells = torch.where(on_fd, fd12, _tensor3(_lagrange(box.x1, _centres(nc)), dg12))
    L = _lagrange(box.x1, box.x1)
    D = np.zeros_like(L)
    w = 1.0 / np.array([np.prod([xi - xj for xj in box.x1 if xj != xi]) for xi in box.x1])
    for i in range(P + 1):
        for j in range(P + 1):
            if i != j:
                D[i, j] = w[j] / w[i] / (box.x1[i] - box.x1[j])
        D[i, i] = -D[i].sum()
    du = torch.zeros_like(dg)
    du[0:3] -= Jd
    du[6] += dg[8]
    for a in range(3):
        du -= 2.0 / h * _along(D, _flux(dg, Jf, a), a)
        el, pt = dg.dim() - 4 - a, dg.dim() - 1 - a
        for side in (0, 1):
            own = dg12.select(pt, P if side else 0)
            # the element dimension keeps its number: the point dimensions follow it
            other = torch.roll(nodes.select(pt, 0 if side else P), -1 if side else 1, el)
            if box.bc[a] == DIRICHLET:
                ends = torch.tensor([box.hi[0] if side else box.lo[0]], dtype=dg.dtype, device=dg.device)
                U = box.flow(ends)
                out = torch.cat([U, _current(U, box.eta)[1]]).reshape(12, *([1] * (other.dim() - 1)))
                at = n[0] - 1 if side else 0
                other = other.clone()
                other.narrow(el, at, 1).copy_(out.expand_as(other.narrow(el, at, 1)))
            jump = other - own
            sign = 1.0 if side else -1.0
            du.select(pt, P if side else 0).sub_((sign * _flux(jump[:9], jump[9:], a) - jump[:9]) / (h * box.w1[0]))
    grid = cells.permute(0, 1, 4, 2, 5, 3, 6).reshape(12, n[2] * nc, n[1] * nc, n[0] * nc)
    df = torch.zeros_like(grid[:9])
    df[0:3] -= Kd.permute(0, 1, 4, 2, 5, 3, 6).reshape_as(df[0:3])
    df[6] += grid[8]
    for a in range(3):
        d = 3 - a
        N = grid.shape[d]
        reach = torch.arange(-3, N + 3, device=grid.device) % N
        ext = grid.index_select(d, reach)
        if box.bc[a] == DIRICHLET:
            for first, x0 in ((0, box.lo[0] - 3 * h / nc), (N + 3, box.hi[0])):
                x = x0 + (torch.arange(3, dtype=grid.dtype, device=grid.device) + 0.5) * h / nc
                U = box.flow(x)
                out = torch.cat([U, _current(U, box.eta)[1]])[:, None, None, :]
                ext.narrow(d, first, 3).copy_(out.expand_as(ext.narrow(d, first, 3)))
        F = _face_flux(ext, a, box.c["recon"], box.c["corr"])
        df -= nc / h * (F.narrow(d, 1, N) - F.narrow(d, 0, N))
    df = df.reshape(9, n[2], nc, n[1], nc, n[0], nc).permute(0, 1, 3, 5, 2, 4, 6)
    return du, df


def _clamp(U):
    E, B = U[0:3], U[3:6]
    B2 = (B * B).sum(0)
    safe = torch.where(B2 > 0, B2, 1.0)
    E = torch.where(B2 > 0, E - (E * B).sum(0) / safe * B, 0.0)
    E2 = (E * E).sum(0)
    return torch.cat([torch.where(E2 > B2, E * (B2 / torch.where(E2 > 0, E2, 1.0)).sqrt(), E), U[3:]])


def _solve(U, box, c):
    """U = R + dt a G(U), pointwise: the cleaning damping and the parallel current."""
    U = U.clone()
    U[6:8] /= 1.0 + box.dt * 0.24169426078821
    if box.eta > 0:
        E, B = U[0:3], U[3:6]
        B2 = (B * B).sum(0)
        safe = torch.where(B2 > 0, B2, 1.0)
        par = (E * B).sum(0) / safe * B
        perp = E - par
        p2, a2 = (perp * perp).sum(0), (par * par).sum(0)
        s = torch.zeros_like(B2)
        for _ in range(80):
            g = c * (p2 / (1 + s) ** 2 + a2 / (1 + c + s) ** 2 - B2) / safe - s
            dg = -2 * c * (p2 / (1 + s) ** 3 + a2 / (1 + c + s) ** 3) / safe - 1.0
            s = torch.where(g > 0, s - g / dg, s)
        U[0:3] = torch.where(B2 > 0, perp / (1 + s) + par / (1 + c + s), E)
    return _clamp(U) if box.c["mode"] else U


def _implicit(U, box):
    drift, full = _current(U, box.eta)
    return torch.cat([drift - full, torch.zeros_like(U[3:6]), -U[6:8], torch.zeros_like(U[8:9])])


def _box_steps(box, dg, fd):
    a, b, e = 0.24169426078821, 0.06042356519705, 0.12915286960590
    z, dt = 0.5 - a - b - e, box.dt
    V = np.polynomial.legendre.legvander(box.x1, box.P)
    sigma = np.exp(-36.0 * (np.arange(box.P + 1) / box.P) ** 100.0)
    F = V @ np.diag(sigma) @ np.linalg.inv(V)
    both = lambda fn, *p: tuple(fn(*(q[k] for q in p)) for k in (0, 1))  # noqa: E731
    solve = lambda p: both(lambda u: _solve(u, box, box.eta * dt * a), p)  # noqa: E731
    imp = lambda p: both(lambda u: _implicit(u, box), p)  # noqa: E731
    filt = lambda p: (_tensor3(F, p[0]), p[1])  # noqa: E731
    un = (dg, fd)
    for _ in range(box.c["steps"]):
        G1 = imp(solve(un))
        U2 = solve(both(lambda u, g: u - dt * a * g, un, G1))
        F2, G2 = _box_rhs(box, *U2), imp(U2)
        U3 = solve(filt(both(lambda u, f, g: u + dt * (f + (1 - a) * g), un, F2, G2)))
        F3, G3 = _box_rhs(box, *U3), imp(U3)
        U4 = solve(filt(both(lambda u, f2, f3, g1, g2, g3: u + dt * (0.25 * (f2 + f3) + b * g1 + e * g2 + z * g3),
                             un, F2, F3, G1, G2, G3)))
        F4, G4 = _box_rhs(box, *U4), imp(U4)
        un = filt(both(lambda u, f2, f3, f4, g2, g3, g4: u + dt * ((f2 + f3 + g2 + g3) / 6 + 2 / 3 * (f4 + g4)),
                       un, F2, F3, F4, G2, G3, G4))
        if box.c["mode"]:
            un = both(_clamp, un)
    return un


def _block_state(case, seed):
    """Extended blocks [9][count][ne^3]: smooth data with a steep front in a third of them."""
    r = random.Random(seed)
    ne, nb = 2 * case["P"] + 7, case["count"]
    t = (torch.arange(ne, dtype=torch.float64, device=_device()) - 0.5 * ne) / ne
    z, y, x = t[:, None, None], t[None, :, None], t[None, None, :]
    U = torch.empty(9, nb, ne, ne, ne, dtype=torch.float64, device=_device())
    base = (0.0, 0.0, -0.8, 1.0, 0.9, 0.3, 0.0, 0.0, 0.2)
    for e in range(nb):
        for v in range(9):
            k = [r.uniform(-3.0, 3.0) for _ in range(3)]
            U[v, e] = base[v] + 3.0 * AMP[v] * torch.cos(k[0] * x + k[1] * y + k[2] * z + r.uniform(0.0, 6.28))
        if e % 3 == 0:
            U[4, e] -= torch.tanh(25.0 * (x + 0.2 * y))
    return _relaxed(U).reshape(9, nb, -1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "blocks":
        ne, nc, nb = 2 * case["P"] + 7, 2 * case["P"] + 1, case["count"]
        U = _block_state(case, seed).reshape(9, nb, ne, ne, ne)
        J = _current(U, 1e3)
        out = torch.zeros(9, nb, nc, nc, nc, dtype=torch.float64, device=U.device)
        core = (slice(None), slice(3, -3), slice(3, -3), slice(3, -3))
        for e in range(nb):
            ext = torch.cat([U[:, e], J[1][:, e]])
            out[0:3, e] = -J[0][:, e][core]
            out[6, e] = U[8:9, e][core][0]
            for a in range(3):
                d, s = 3 - a, list(core)
                s[d] = slice(None)
                F = _face_flux(ext[tuple(s)], a, 0, case["corr"])
                out[:, e] -= nc / 0.0625 * (F.narrow(d, 1, nc) - F.narrow(d, 0, nc))
        return out.reshape(9, nb, -1)
    # with the indicator on, the mask is the run's own choice
    if kind not in ("rhs", "step") or (case.get("tci") and case["flow"] != "wave"):
        return None
    box = _Box(case, seed)
    U, m = box.state()
    cut = 9 * box.E * box.np1 ** 3
    n = box.n
    dg = U[:cut].reshape(9, n[2], n[1], n[0], box.np1, box.np1, box.np1)
    fd = U[cut:].reshape(9, n[2], n[1], n[0], box.nc, box.nc, box.nc)
    if kind == "step" and case.get("tci") and int(m.sum()):
        return None
    dg, fd = _box_rhs(box, dg, fd) if kind == "rhs" else _box_steps(box, dg, fd)
    dg, fd = dg.reshape(9, box.E, -1).clone(), fd.reshape(9, box.E, -1).clone()
    dg[:, m != 0] = 0.0
    fd[:, m == 0] = 0.0
    out = torch.cat([dg.reshape(-1), fd.reshape(-1)])
    return out if kind == "rhs" else [out, None]
