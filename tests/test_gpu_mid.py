"""The middle levels and the tail of a V-cycle in one cluster launch against the
launches they replace.

Every cell sees the same operations in the same order, so whole runs are bit-identical with
either path (FERROX_RB_SWEEPS=0, read when a context is created, keeps the separate
launches): one to three middle levels, sides of 4 and up, planes that halve, stay odd or do
not fill the CTAs' parts, tails solved by their inverse and by a V-cycle, with and without
carriers, one and two smoothing sweeps, levels that are halved in one lateral direction
only, FP64 and mixed.
"""
import numpy as np
import pytest

from paper_2210_15668_gb300 import inputs as I

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

SHAPES = [(64, 64, 16), (48, 80, 12), (128, 16, 9), (8, 512, 10), (32, 32, 32), (64, 48, 24), (64, 32, 37),
          (256, 192, 16), (64, 64, 64), (96, 80, 37), (80, 96, 21), (48, 20, 30)]
FORMS = {"plain": dict(), "one_sweep": dict(nu1=1, nu2=1), "inner2": dict(inner=2), "order2": dict(order=2)}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("stack", ["mfim", "mfism", "fermi"])
def test_middle_levels_bit_identical(stack, shape, form, precision, monkeypatch):
    from paper_2210_15668_gb300 import ferrox
    nx, ny, nz = shape
    layers = I.mfim_stack(nz, n_fe=4) if stack == "mfim" else I.mfism_stack(nz, n_fe=3, n_ox=1)
    if stack == "fermi":
        layers[0] = I.sc_layer(nz - 4, stats=I.STATS_FERMI_DIRAC)
    geom = I.make_geometry(nx, ny, layers)
    P0 = I.random_polarization(geom, seed=6, amp=0.05)
    num = ferrox.make_numerics(4e-13, tol=1e-10, precision=precision, **FORMS[form])
    out = {}
    for env in ("0", "1"):
        monkeypatch.setenv("FERROX_RB_SWEEPS", env)
        d = ferrox.Device(geom, P0, numerics=num)
        d.set_bias(0.0, 0.6)
        d.solve_poisson()
        d.step(2)
        out[env] = d.get_state() + (d.stats(),)
        d.close()
    (Pa, pa, sa), (Pb, pb, sb) = out["0"], out["1"]
    assert sb["status"] == sa["status"] and sa["vcycles"] == sb["vcycles"]
    assert np.array_equal(Pa, Pb) and np.array_equal(pa, pb)
    assert sb["launches"] <= sa["launches"]
