"""The FP64 polarization update with face values shared along the column, against the
oracle: stacks that start and end the march (every remainder of the chunks,
ferroelectric layers apart and side by side with different materials, electrodes on either
side) through the context entry and through the one that allocates nothing, which takes its
tables by value up to 16 layers and by copy beyond.

Tolerances: the update is the oracle's FP64 arithmetic in another order, <= 1e-12 max|P|;
the right-hand side shows through a solve to 1e-13, <= 1e-11 relative on the potential.
"""
import numpy as np
import pytest

import oracle
from oracle import poisson, tdgl
from paper_2210_15668_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

STACKS = {
    "two": [I.fe_layer(2), I.de_layer(6)],
    "three": [I.de_layer(5), I.fe_layer(3)],
    "five_all": [I.fe_layer(5)],
    "six": [I.de_layer(2), I.fe_layer(6), I.de_layer(4)],
    "thirteen": [I.de_layer(3), I.fe_layer(13)],
    "apart": [I.fe_layer(3), I.de_layer(1), I.fe_layer(2), I.de_layer(2, 10.0), I.fe_layer(5)],
    "side_by_side": [I.de_layer(2), I.fe_layer(2), I.fe_layer(3, g=5e-10, eps_r=40.0, Gamma=60.0), I.fe_layer(1)],
    "sixteen_layers": [I.fe_layer(2, g=2e-10), I.de_layer(1)] * 8,
    "eighteen_layers": [I.de_layer(1, 10.0), I.fe_layer(2)] * 9,
}


@pytest.mark.parametrize("ncomp", [1, 3])
@pytest.mark.parametrize("name", list(STACKS))
def test_update_and_rhs_match_oracle(name, ncomp):
    from paper_2210_15668_gb300 import ferrox
    geom = I.make_geometry(34, 6, STACKS[name], pbc=I.PBC_LAMBDA, ncomp=ncomp)
    pl = oracle.planes(geom)
    P = I.random_polarization(geom, seed=61, amp=0.15)
    phi = np.random.default_rng(62).uniform(-0.5, 0.5, P.shape[1:])
    dt, vb, vt = 4e-13, 0.1, 0.7
    Pexp = P + dt * tdgl.force(P, phi, pl, geom, vb, vt)
    d = ferrox.Device(geom, P, numerics=ferrox.make_numerics(dt, tol=1e-13), phi0=phi)
    d.set_bias(vb, vt)
    d.tdgl_update()
    Pg, phig = d.get_state()
    assert np.abs(Pg - Pexp).max() <= 1e-12 * np.abs(P).max()
    assert np.array_equal(phig, phi)
    d.solve_poisson()
    phio = poisson.solve_linear(Pexp, pl, geom["h"], vb, vt)
    phig = d.get_state()[1]
    assert np.linalg.norm(phig - phio) <= 1e-11 * np.linalg.norm(phio)
    d.close()
    Ps, ps = torch.as_tensor(P, device="cuda").clone(), torch.as_tensor(phi, device="cuda").clone()
    ferrox.tdgl_update_static(geom, dt, vb, vt, Ps, ps)
    torch.cuda.synchronize()
    assert np.abs(Ps.cpu().numpy() - Pexp).max() <= 1e-12 * np.abs(P).max()
    assert np.array_equal(ps.cpu().numpy(), phi)
