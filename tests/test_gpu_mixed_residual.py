"""The outer residual that the mixed form's solves compute, cell by cell: one outer iteration
from a rough potential in the mixed form and in FP64.

Both take the same V-cycles on their residual; the FP64 one's residual is compared with the
oracle elsewhere (ferrox_residual).  The mixed correction e differs by FP32 arithmetic: its
right-hand side, shifts and diagonals are rounded once (2^-24 of them) and a cell sees under
200 roundings a V-cycle, so |e_mixed - e_fp64| <= 2 x 400 x 2^-24 max|e| = 5e-5 max|e| with
two V-cycles, every rounding taken at full size.  An error in the residual of one cell
shows as that error over the cell's diagonal at least.  Stacks: without carriers, Boltzmann
ones (double-float beside the stencil), Fermi-Dirac ones in one chunk rule and the other,
both kinds; odd plane counts, ragged and one-cell-wide sides (a grid that the mixed form holds
whole in the tail takes other V-cycles).
"""
import numpy as np
import pytest

from paper_2210_15668_gb300 import inputs as I

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


def _sc(n, fd):
    return I.sc_layer(n, N_A=1e24, stats=I.STATS_FERMI_DIRAC if fd else I.STATS_BOLTZMANN)


STACKS = {
    "none": lambda nz: I.mfim_stack(nz, n_fe=6),
    "boltzmann": lambda nz: [_sc(nz - 8, False), I.de_layer(2), I.fe_layer(6)],
    "fermi": lambda nz: [_sc(nz - 8, True), I.de_layer(2), I.fe_layer(6)],
    "both": lambda nz: [_sc(nz // 4, True), _sc(nz // 4, False), I.de_layer(2), I.fe_layer(nz - 2 * (nz // 4) - 2)],
}


@pytest.mark.parametrize("shape", [(64, 64, 32), (48, 40, 24), (24, 36, 21), (1, 512, 20), (160, 96, 48)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("stack", list(STACKS))
def test_one_outer_iteration_agrees_with_fp64(stack, shape):
    from paper_2210_15668_gb300 import ferrox
    nx, ny, nz = shape
    geom = I.make_geometry(nx, ny, STACKS[stack](nz))
    P = I.random_polarization(geom, seed=8, amp=0.05)
    phi0 = np.random.default_rng(9).uniform(-0.05, 0.05, P.shape[1:])
    e = []
    for precision in (ferrox.FP64, ferrox.MIXED):
        num = ferrox.make_numerics(4e-13, tol=1e-14, max_cycles=1, precision=precision, inner=2)
        d = ferrox.Device(geom, P, numerics=num, phi0=phi0)
        d.set_bias(0.02, 0.3)
        d.solve_poisson()
        e.append(d.phi.cpu().numpy() - phi0)   # the state entry would report the solve as not converged
        assert d.stats(check=False)["cycles"] == 1
        d.close()
    assert np.abs(e[0]).max() > 1e-2
    assert np.abs(e[1] - e[0]).max() <= 5e-5 * np.abs(e[0]).max()
