"""The FP64 restriction of the red children with a Newton shift: levels halved in all three
directions that are two cells wide, ragged against the blocks, or large enough for whole
blocks, against the oracle's Newton solve.  Solves to 1e-12 agree to 1e-9 relative (L2), the
bound of the other carrier tests."""
import numpy as np
import pytest

import oracle
from oracle import carriers, poisson
from paper_2210_15668_gb300 import inputs as I

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


@pytest.mark.parametrize("stats", [I.STATS_BOLTZMANN, I.STATS_FERMI_DIRAC])
@pytest.mark.parametrize("shape", [(2, 64, 32), (4, 4, 24), (72, 20, 32), (64, 48, 16), (64, 64, 64)],
                         ids=lambda s: "x".join(map(str, s)))
def test_solve_with_carriers(shape, stats):
    from paper_2210_15668_gb300 import ferrox
    nx, ny, nz = shape
    geom = I.make_geometry(nx, ny, [I.sc_layer(nz // 2, N_A=1e24, stats=stats), I.de_layer(nz // 8),
                                    I.fe_layer(nz - nz // 2 - nz // 8)])
    pl = oracle.planes(geom)
    P = I.random_polarization(geom, seed=91, amp=0.2)
    d = ferrox.Device(geom, P, numerics=ferrox.make_numerics(4e-13, tol=1e-12))
    d.set_bias(0.0, 0.8)
    d.solve_poisson()
    st = d.stats()
    phig = d.get_state()[1]
    d.close()
    phio, _ = carriers.newton_solve(poisson.rhs(P, pl, geom["h"], 0.0, 0.8), np.zeros(P.shape[1:]), pl, geom["h"], tol=1e-13)
    assert st["status"] == 0 and st["last_rel_res"] <= 1e-12
    assert np.linalg.norm(phig - phio) <= 1e-9 * np.linalg.norm(phio)
