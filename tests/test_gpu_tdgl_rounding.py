"""The FP64 polarization update rounds relative to its gradient terms, not to g/h^2 P.

In smooth domains the terms of d2/dx2, d2/dy2 and d2/dz2 nearly cancel: the sums of their
neighbours are larger than the differences by orders of magnitude.  P is given on a grid of
2^-20, so that every difference of neighbours is exact, and the Landau coefficients vanish.
Then P_new differs from the exact value (extended precision) by its own rounding, 2^-53 |P_new|,
and by the roundings of the force's terms, at most 16 of 2^-53 Gamma dt times the sum S of the
terms' sizes (three or four operations a term and its coefficients).  S is about 0.02 P
inside a layer; coefficients of P collected over the neighbours would add 6 g/h^2 Gamma dt P =
0.96 P (and its fourfold) instead.
"""
import numpy as np
import pytest

from paper_2210_15668_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -53
EPS0 = 8.8541878128e-12


def _exact(geom, P, dt, g, Gamma):
    """P_new and the sum of the terms' sizes, potential and electrodes zero."""
    L = np.longdouble
    h, lam = L(geom["h"]), L(geom["lam"])
    kappa = lam / (3 * h + 8 * lam)
    eps = np.array([l["eps_r"] for l in geom["layers"] for _ in range(l["ncells"])], dtype=L)
    fe = I.fe_plane_mask(geom)
    q, nz = P.astype(L), len(eps)
    lap = np.roll(q, 1, 1) + np.roll(q, -1, 1) + np.roll(q, 1, 2) + np.roll(q, -1, 2) - 4 * q
    face = np.zeros((nz + 1,) + q.shape[1:], dtype=L)
    for k in range(1, nz):
        face[k] = -h * (q[k] - q[k - 1]) / (2 * L(EPS0) * (eps[k] + eps[k - 1]))
    out, size = q.copy(), np.zeros_like(q)
    for k in np.nonzero(fe)[0]:
        dn, up = k > 0 and fe[k - 1], k + 1 < nz and fe[k + 1]
        if dn and up:
            terms = [q[k + 1] - q[k], q[k - 1] - q[k]]
        else:
            o = q[k + 1] if up else q[k - 1]
            terms = [4 * (18 * kappa - 3) / 3 * q[k], 4 * (1 - 2 * kappa) / 3 * o]
        grad = [-g * lap[k] / h ** 2] + [-g * t / h ** 2 for t in terms] + [face[k + 1] / h, -face[k] / h]
        out[k] = q[k] - Gamma * dt * sum(grad)
        size[k] = Gamma * dt * sum(np.abs(t) for t in grad)
    return out, size


@pytest.mark.parametrize("g", [1e-9, 4e-9])
@pytest.mark.parametrize("layers", [(3, 10), (0, 9), (2, 2)])
def test_update_rounds_relative_to_its_terms(layers, g):
    from paper_2210_15668_gb300 import ferrox
    n, dt, Gamma = 64, 4e-13, 100.0
    de, nf = layers
    stack = ([I.de_layer(de)] if de else []) + [I.fe_layer(nf, g=g, alpha=0.0, beta=0.0, gamma=0.0, Gamma=Gamma)]
    geom = I.make_geometry(n, n, stack)
    k, j, i = np.meshgrid(np.arange(de + nf), np.arange(n), np.arange(n), indexing="ij")
    P = 0.2 * (1.5 + np.sin(2 * np.pi * i / n) * np.cos(2 * np.pi * j / n)) * (1 + 1e-3 * k)
    P = np.round(P * 2.0 ** 20) / 2.0 ** 20
    P[~I.fe_plane_mask(geom)] = 0.0
    exact, size = _exact(geom, P, np.longdouble(dt), np.longdouble(g), np.longdouble(Gamma))
    d = ferrox.Device(geom, P[None], numerics=ferrox.make_numerics(dt), phi0=np.zeros_like(P))
    d.set_bias(0.0, 0.0)
    d.tdgl_update()
    ctx = d.get_state()[0][0]
    d.close()
    Ps, ps = torch.as_tensor(P[None], device="cuda").clone(), torch.zeros(P.shape, dtype=torch.float64, device="cuda")
    ferrox.tdgl_update_static(geom, dt, 0.0, 0.0, Ps, ps)
    torch.cuda.synchronize()
    for got in (ctx, Ps.cpu().numpy()[0]):
        off = np.abs(got.astype(np.longdouble) - exact)
        assert (off <= U * (np.abs(exact) * (1 + 1e-6) + 16 * size)).all()
