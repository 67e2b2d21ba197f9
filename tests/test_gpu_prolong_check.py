"""The FP64 transfers that only touch the colour that is read again: prolongation of the
black cells alone, and the residual, norm and restriction of the red ones.

A solve must reach the potential of the oracle's exact solve, where tiles are ragged, one
coarse column wide, shorter than a block's planes, or single cells; with and without
post-smoothing (without it every cell is wanted unless pre-smoothing follows at once, as
with one V-cycle per check).  Solves to 1e-12 agree to 1e-10 relative (L2), the factor
between tolerance and error of the other solver tests.
"""
import numpy as np
import pytest

import oracle
from oracle import poisson
from paper_2210_15668_gb300 import inputs as I

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

SHAPES = [(4, 4, 4), (2, 64, 8), (68, 12, 10), (64, 64, 16), (72, 40, 6), (132, 20, 34), (64, 64, 37), (2, 2, 12)]


@pytest.mark.parametrize("inner", [1, 2])
@pytest.mark.parametrize("nu", [(2, 2), (1, 0), (1, 3)], ids=lambda n: f"nu{n[0]}{n[1]}")
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_solve_matches_oracle(shape, nu, inner):
    from paper_2210_15668_gb300 import ferrox
    nx, ny, nz = shape
    if nz % 2 and nu[1] == 0:
        pytest.skip("planes that never halve: one sweep a V-cycle needs more than 400")
    geom = I.make_geometry(nx, ny, [I.de_layer(nz // 2), I.fe_layer(nz - nz // 2)])
    pl = oracle.planes(geom)
    P = I.random_polarization(geom, seed=71, amp=0.2)
    d = ferrox.Device(geom, P, numerics=ferrox.make_numerics(4e-13, tol=1e-12, nu1=nu[0], nu2=nu[1], max_cycles=400,
                                                               inner=inner))
    d.set_bias(-0.2, 0.6)
    d.solve_poisson()
    st = d.stats()
    phig = d.get_state()[1]
    d.close()
    phio = poisson.solve_linear(P, pl, geom["h"], -0.2, 0.6)
    assert st["status"] == 0 and st["last_rel_res"] <= 1e-12
    assert np.linalg.norm(phig - phio) <= 1e-10 * np.linalg.norm(phio)
