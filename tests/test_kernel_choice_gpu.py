"""Which kernel a grid takes, on both sides of each rule: FP64 2D grids of
small and of large tiles, anisotropic problems of four phases in 3D (the
extended kernels), 3D grids whose liquid path marches two segments at a time,
and handles whose buffers hold an older state's liquid planes."""
import copy

import numpy as np
import pytest

from paper_2608_26908_gb300 import gpflbm, inputs, slabs
from parity import device_run, reference, rel_err

pytestmark = pytest.mark.gpu

TOL = {"fp64": {"phi": 1e-10, "mu": 1e-10, "c": 1e-10, "rho": 1e-10, "u": 1e-8, "dev": 1e-8},
       "fp32": dict.fromkeys(("phi", "mu", "c", "rho", "u", "dev"), 1e-5)}


def _check(sc, steps):
    ref = reference(sc, steps)
    sim, got = device_run(sc, steps)
    sim.close()
    for k, tol in TOL[sc["precision"]].items():
        assert rel_err(got[k], ref[k]) <= tol, (k, rel_err(got[k], ref[k]))


@pytest.mark.parametrize("name,nx,ny", [
    ("dendrite2d", 64, 56),     # small tiles
    ("dendrite2d", 225, 203),   # the last grid of small tiles ...
    ("dendrite2d", 300, 191),   # ... and grids of large ones, ragged
    ("eutectic2d", 301, 200),
])
def test_fp64_2d_tiles_on_both_sides_of_the_rule(name, nx, ny):
    sc = inputs.scenario(name, nx=nx, ny=ny, precision="fp64")
    sc["params"]["gbeta_c"] = [2e-3, 0.0]
    _check(sc, 20)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_anisotropic_four_phases_in_3d(prec):
    sc = inputs.scenario("eutectic3d", nx=36, ny=34, nz=40, precision=prec)
    sc["init"]["height"] = 12
    for a in range(1, 4):
        sc["params"]["delta"][0][a] = sc["params"]["delta"][a][0] = 0.03
    _check(sc, 30)


def test_two_segments_a_march_match_the_slabs():
    """FP16 populations: 2052 CTAs of the liquid path march two segments, and
    the slabs, whose every tile is general, give the same bits."""
    sc = inputs.scenario("dendrite3d", nx=256, ny=256, nz=144, precision="fp32_f16")
    sc["params"]["gbeta_c"] = [2e-3, 0.0]
    phi0, mu0 = inputs.initial_state(sc)
    layer, steps = 256 * 256, 6
    whole = gpflbm.Sim(sc)
    whole.set_state(phi0, mu0)
    whole.step(steps)
    ref = whole.fields(("phi", "mu", "f"))
    whole.close()
    runs = []
    for r, (v0, n) in enumerate([(0, 73), (73, 71)]):
        sim = gpflbm.Sim(sc, slab=(v0, n))
        cut = [a.reshape(-1, 144 * layer)[:, v0 * layer:(v0 + n) * layer].reshape(-1) for a in (phi0, mu0)]
        sim.set_state(*cut)
        runs.append((v0, n, slabs.Slab(sim, r, 2)))
    for _ in range(steps):
        slabs.step_all([s for _, _, s in runs])
    for v0, n, s in runs:
        got = s.sim.fields(("phi", "mu", "f"))
        for k in got:
            np.testing.assert_array_equal(got[k], ref[k][:, v0 * layer:(v0 + n) * layer], err_msg=k)


def _liquid(sc):
    n = inputs.cells(sc)
    phi = np.zeros((sc["n_phases"], n))
    phi[0] = 1.0
    return phi.reshape(-1), np.zeros(sc["n_solutes"] * n)


@pytest.mark.parametrize("name,size", [("dendrite3d", dict(nx=64, ny=60, nz=66)),
                                       ("eutectic3d", dict(nx=62, ny=60, nz=66))])
def test_planes_left_by_an_older_state_are_written_again(name, size):
    """The liquid path skips the phase planes that its output buffer's flags
    call pure liquid; a handle that held other states, with the liquid path
    on and off, steps a new state as a fresh handle does."""
    sc = inputs.scenario(name, precision="fp32", **size)
    sc["init"]["height" if name == "eutectic3d" else "radius"] = 14
    shrink = copy.deepcopy(sc)
    shrink["params"]["eta_rho"][1] = 0.1  # every tile general: no flags are kept
    other = copy.deepcopy(sc)
    other["init"]["height" if name == "eutectic3d" else "radius"] = 40 if name == "eutectic3d" else 25
    state, solid = inputs.initial_state(sc), inputs.initial_state(other)

    def run(sim):
        sim.set_state(*state)
        sim.step(5)
        return sim.fields(("phi", "mu", "f"))

    want = run(gpflbm.Sim(sc))
    sim = gpflbm.Sim(sc)
    for before in (_liquid(sc), solid, _liquid(sc)):
        sim.set_state(*before)
        sim.step(3)
        got = run(sim)
        for k in got:
            np.testing.assert_array_equal(got[k], want[k], err_msg=k)
    sim.set_state(*_liquid(sc))
    sim.step(2)
    sim.set_params(shrink)
    sim.set_state(*solid)
    sim.step(3)
    sim.set_params(sc)
    for k, v in run(sim).items():
        np.testing.assert_array_equal(v, want[k], err_msg=k)
