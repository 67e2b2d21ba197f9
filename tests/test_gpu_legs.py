"""V-cycle legs (one launch per level and direction) against the launches they replace.

A leg relaxes, restricts and prolongates with the operations of the colour sweeps and
transfers in the same order, so whole runs are bit-identical with either path
(FERROX_RB_SWEEPS=0, read when a context is created, keeps the separate launches), on
grids that leave ragged tiles, wrap the halo around short sides, cut the planes into
chunks and end in odd plane counts.
"""
import numpy as np
import pytest

from paper_2210_15668_gb300 import inputs as I

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

SHAPES = [(36, 20, 9), (16, 40, 12), (4, 300, 8), (132, 68, 16), (48, 80, 37), (96, 64, 40), (256, 144, 34),
          (288, 576, 36)]
FORMS = {"plain": dict(), "inner3": dict(inner=3, guess=1), "adaptive": dict(inner=-8, guess=1)}


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("stack", ["mfim", "mfism"])
def test_legs_bit_identical(stack, shape, form, monkeypatch):
    from paper_2210_15668_gb300 import ferrox
    nx, ny, nz = shape
    layers = I.mfim_stack(nz, n_fe=4) if stack == "mfim" else I.mfism_stack(nz, n_fe=3, n_ox=1)
    geom = I.make_geometry(nx, ny, layers)
    P0 = I.random_polarization(geom, seed=5, amp=0.05)
    num = ferrox.make_numerics(4e-13, tol=1e-10, precision=ferrox.MIXED, **FORMS[form])
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
    assert np.array_equal(Pa, Pb) and np.array_equal(pa, pb)
    assert sa["vcycles"] == sb["vcycles"] and sa["cycles"] == sb["cycles"]
    assert sb["launches"] < sa["launches"]


def test_batched_legs_equal_the_persistent_launch():
    """The graph engine's legs against the persistent launch's colour sweeps: a batch with
    and without carriers, with short, ragged and odd instances."""
    from paper_2210_15668_gb300 import ferrox
    geoms = [I.make_geometry(nx, ny, I.mfim_stack(nz, n_fe=4) if k == 0 else I.mfism_stack(nz, n_fe=3, n_ox=1))
             for nx, ny, nz, k in [(64, 48, 16, 0), (36, 20, 9, 1), (112, 80, 14, 1), (16, 144, 12, 0), (96, 96, 21, 1)]]
    P0 = [I.random_polarization(g, seed=40 + i, amp=0.05) for i, g in enumerate(geoms)]
    out = []
    for engine in (0, 1):
        b = ferrox.Batch(geoms, P0, ferrox.make_numerics(4e-13, tol=1e-10, precision=ferrox.MIXED))
        b.set_engine(engine)
        b.set_bias(0.0, [0.5, -0.4, 0.2, 1.0, -0.1])
        b.solve_poisson()
        b.step(2)
        out.append(([b.state(i) for i in range(len(geoms))], [s["cycles"] for s in b.stats()]))
        b.close()
    (sa, ca), (sb, cb) = out
    assert ca == cb
    for (Pa, pa), (Pb, pb) in zip(sa, sb):
        assert np.array_equal(Pa, Pb) and np.array_equal(pa, pb)
