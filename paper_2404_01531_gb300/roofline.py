"""Operation counts of the hot kernels, two kinds.

*_flops: the method's FP64 work (FMA = 2 flops, add/mul/div/sqrt = 1), counted
from the operations the method defines.  The kernels share work between
neighbouring face values and run line contractions and WENO5-Z weights on the
integer pipes, so this divided by the launch time can exceed the FP64 peak.

*_fp64_ops: FP64 operations the kernels issue.  Each takes one FMA slot of the
FP64 pipe, the pipe with the highest use, so 2 x ops / time over the peak is
the fraction of that bound (at most 1)."""
import math


def fp64_peak_tflops(n_sm, sm_mhz):
    """FP64 peak from the unit counts and the clock: 2 FMA lanes per clock per
    SM x 2 flops x SMs x clock (152 SMs at 2070 MHz: the GB300's nominal
    1.25 TFLOP/s FP64)."""
    return 2 * 2 * n_sm * sm_mhz * 1e6 / 1e12


FP64_PEAK_TFLOPS = fp64_peak_tflops(152, 2070.0)   # the GB300's nominal figure


def filter_rank(P, a=36.0, b=50.0):
    """Modes the exponential filter sigma_m = exp(-a (m/P)^(2b)) damps by more
    than 1e-20: the rank of I - F along one axis as the DG kernels apply it."""
    return sum(1 for m in range(P + 1) if -math.expm1(-a * (m / P) ** (2 * b)) > 1e-20)


def dg_flops_per_node(P, sub, filter_on=True, tci_on=True, solve=True, a=36.0, b=50.0):
    """One DG node through k_dg_substep: volume term (27 directional (P+1)-point
    contractions), derivative combination and explicit sources, the lifted
    Rusanov correction (6 (P+1)^2 face nodes per (P+1)^3 nodes), the IMEX stage
    combination, the pointwise stiff solve and implicit operator (substeps A, B),
    the filter of 9 variables in its low-rank form (per axis and kept mode one
    (P+1)-point dot product per line and one FMA per node) and the indicator
    (|B|, 3 low-pass contractions, two sums).  sub: 0 (A), 1 (B), 2 (C)."""
    n = P + 1
    f = 27 * n * 2              # volume contractions
    f += 22                     # combination + sources
    f += 39 * 6 / n             # lift per face node, averaged per node
    f += (28, 57, 84)[sub]      # stage combination
    if sub != 2 and solve:
        f += 38 + 30            # stiff solve + implicit operator
    if filter_on:
        f += 3 * 2 * 2 * 9 * filter_rank(P, a, b)
    if tci_on:
        f += 6 + 3 * n * 2 + 5
    return f


WENO_FLOPS = 75                  # both WENO5-Z face values of a cell (one set of indicators, 2 divisions)
# MP5: both values on their unlimited path, the 5-point interpolant (9), v_MP (4) and
# the bracketing test (3) each; the limited path adds data-dependent work not counted
MP5_FLOPS = 32
FLUX_FLOPS = 60                  # Rusanov flux, corrector and flux difference


def fd_flux_flops(recon, quantities=10):
    """Algorithmic flops of one face of the FD flux kernel for the reconstruction
    (0 WENO5-Z, 1 MP5): 10 of the 12 quantities enter the flux along a direction of
    a box, all of them a face of a shell."""
    return quantities * (MP5_FLOPS if recon == 1 else WENO_FLOPS) + FLUX_FLOPS


def fd_faces_per_element(P):
    nc = 2 * P + 1
    return 3 * (nc + 1) * nc * nc


def fd_flux_fp64_ops(recon, P, quantities=10, corrector=True):
    """FP64 operations per face that k_fd_flux (a box: 10 quantities a direction) or
    k_fd_states (a flat shell: 12) issues: a line of nc cells takes nc two-sided
    reconstructions, two one-sided ones and 5 differences (MP5: its unlimited path),
    a face the flux of 5 pairs of quantities, or the states of 6.  ncu counts
    the same 308.3 for k_fd_flux at P = 5 with the corrector."""
    nc = 2 * P + 1
    both, one = (14, 8) if recon == 1 else (25, 15)
    line = quantities * (nc * both + 2 * one + 5) / (nc + 1)
    if quantities == 12:
        return line + (66 if corrector else 42)
    return line + (50 if corrector else 30)


# FP64 operations a thread of k_dg_substep issues per node in substeps A, B and C at
# P = 5, flat metric, filter (a = 36, b = 50) and indicator on: FP64-pipe instructions
# (ncu sm__inst_executed_pipe_fp64) over 28672 warps of 4096 elements
DG_FP64_OPS_P5 = (138.1, 157.1, 122.1)


def dg_fp64_ops_per_element(P):
    """Mean over the substeps, for the threads of an element's CTA; None at other orders."""
    return sum(DG_FP64_OPS_P5) / 3.0 * 224 if P == 5 else None
