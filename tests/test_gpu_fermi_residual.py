"""The Fermi-Dirac charge of the FP64 residual over the whole range of the reduced
potential, cell by cell against the oracle.

phi is drawn so that u = phi / V_T covers [-45, 45] (both carriers from far below the band
edge to deep inside the band, across every place where a term of the approximation is left
out), and beyond |u| = 300, where the general form is taken.  Each side rounds eta =
eta_0 + u and u itself, so e^-eta carries about (|u| + |eta|) 2^-53, and a handful of
operations more: 512 2^-53 of the charges bounds the difference for |u| <= 45, and the
stencil's terms are rounded to 2^-53 of the largest.
"""
import numpy as np
import pytest

import oracle
from oracle import carriers, poisson
from paper_2210_15668_gb300 import inputs as I

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

DOPING = {"undoped": dict(N_A=0.0), "p": dict(N_A=1e24), "n+": dict(N_A=0.0, N_D=5e26)}


@pytest.mark.parametrize("doping", list(DOPING))
@pytest.mark.parametrize("span", [45.0, 800.0])
def test_residual_matches_oracle(doping, span):
    from paper_2210_15668_gb300 import ferrox
    geom = I.make_geometry(32, 16, [I.sc_layer(20, stats=I.STATS_FERMI_DIRAC, **DOPING[doping]), I.de_layer(2),
                                    I.fe_layer(10)])
    pl = oracle.planes(geom)
    P = I.random_polarization(geom, seed=81, amp=0.1)
    vt = carriers.K_B * 300.0 / carriers.Q_E
    phi = np.random.default_rng(82).uniform(-span, span, P.shape[1:]) * vt
    h = geom["h"]
    scale = h * h / oracle.EPS0
    d = ferrox.Device(geom, P, numerics=ferrox.make_numerics(4e-13), phi0=phi)
    d.set_bias(0.0, 0.3)
    d.tdgl_update()
    P1 = d.get_state()[0]
    r = d.residual()
    d.close()
    rho, _ = carriers.charge(phi, pl)
    b = poisson.rhs(P1, pl, h, 0.0, 0.3)
    ro = poisson.residual(phi, b, pl, h, rho=rho) * scale
    eps = 2.0 ** -53
    terms = 12.0 * (pl["eps"] / oracle.EPS0).max() * np.abs(phi).max() + np.abs(b).max() * scale
    weight = 512.0 if span < 100 else 16.0 * span
    assert np.all(np.abs(r - ro) <= 32 * eps * terms + weight * eps * (np.abs(rho) * scale + 1.0))
