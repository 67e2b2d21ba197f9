"""The cluster launch of the middle levels takes the levels it is meant for, so that the bit
comparisons with the separate launches compare two paths: from the first level below the
fine one of at most 16384 cells on, stacks solved in FP64 and mixed ones whose tail is
relaxed.  The levels above it show one restriction (one way down) each per V-cycle in an
eagerly run step, none of the FP64 ones below a colour sweep of their own."""
import pytest

from paper_2210_15668_gb300 import inputs as I

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

# stack, shape, precision, levels between the fine one and the cluster
CASES = [("mfim", (64, 64, 16), 0, 0), ("mfim", (48, 80, 12), 0, 0), ("mfim", (64, 48, 24), 0, 0), ("mfim", (64, 64, 64), 0, 1),
         ("mfim", (256, 192, 16), 0, 1), ("mfism", (64, 48, 24), 1, 0), ("mfism", (64, 64, 64), 1, 1), ("mfism", (96, 80, 37), 1, 2)]


@pytest.mark.parametrize("stack, shape, precision, above", CASES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_levels_taken_by_the_cluster(stack, shape, precision, above, monkeypatch):
    from paper_2210_15668_gb300 import ferrox
    nx, ny, nz = shape
    geom = I.make_geometry(nx, ny, I.mfim_stack(nz, n_fe=4) if stack == "mfim" else I.mfism_stack(nz, n_fe=3, n_ox=1))
    P0 = I.random_polarization(geom, seed=6, amp=0.05)
    seen = {}
    for env in ("0", "1"):
        monkeypatch.setenv("FERROX_RB_SWEEPS", env)
        d = ferrox.Device(geom, P0, numerics=ferrox.make_numerics(4e-13, tol=1e-10, precision=precision))
        d.set_bias(0.0, 0.6)
        d.solve_poisson()
        prof = d.profile_step()
        d.close()
        assert prof["tail"][1] > 0
        seen[env] = {k: prof[k][1] / prof["tail"][1] for k in ("restrict", "smooth_coarse")}
    assert seen["1"]["restrict"] == above < seen["0"]["restrict"]
    assert seen["1"]["smooth_coarse"] <= seen["0"]["smooth_coarse"] and (above or not seen["1"]["smooth_coarse"])
