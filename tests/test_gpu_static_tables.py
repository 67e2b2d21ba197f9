"""The allocation-free update's tables do not depend on how they are made: by a kernel from up
to 16 layers, by the host from more, or by a context.  The same planes given as one layer
and as one layer a plane, and to a context, lead to the same bits."""
import numpy as np
import pytest

from paper_2210_15668_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ncomp", [1, 3])
@pytest.mark.parametrize("pbc, lam", [(I.PBC_LAMBDA, 3e-9), (I.PBC_LAMBDA, 0.7e-9), (I.PBC_LAMBDA, 1.3e-10), (I.PBC_FREE, 0.0),
                                      (I.PBC_ZERO, 0.0)])
@pytest.mark.parametrize("g, h", [(1e-10, 0.5e-9), (3e-9, 0.37e-9)])
def test_layers_planes_and_context_agree(g, h, pbc, lam, ncomp):
    from paper_2210_15668_gb300 import ferrox
    run = [(I.de_layer, 2, 3.9, {}), (I.fe_layer, 7, g, dict(Gamma=90.0)), (I.de_layer, 1, 10.0, {}),
           (I.fe_layer, 9, 1.7 * g, dict(eps_r=33.0))]
    whole = [f(n, v, **kw) for f, n, v, kw in run]
    split = [f(1, v, **kw) for f, n, v, kw in run for _ in range(n)]
    assert len(whole) <= 16 < len(split)
    geoms = [I.make_geometry(36, 10, l, h=h, pbc=pbc, lam=lam, ncomp=ncomp) for l in (whole, split)]
    P = I.random_polarization(geoms[0], seed=5, amp=0.2)
    phi = np.random.default_rng(6).uniform(-0.5, 0.5, P.shape[1:])
    dt, vb, vt = 4e-13, 0.15, 0.6
    got = []
    for geom in geoms:
        Ps, ps = torch.as_tensor(P, device="cuda").clone(), torch.as_tensor(phi, device="cuda").clone()
        ferrox.tdgl_update_static(geom, dt, vb, vt, Ps, ps)
        torch.cuda.synchronize()
        got.append(Ps.cpu().numpy())
    d = ferrox.Device(geoms[0], P, numerics=ferrox.make_numerics(dt), phi0=phi)
    d.set_bias(vb, vt)
    d.tdgl_update()
    got.append(d.get_state()[0])
    d.close()
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
