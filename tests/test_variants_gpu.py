"""Every variant of the step kernels that a size or a model switches to,
against the FP64 oracle: the 3D tiles in FP64 at their edges, with each model,
the anisotropic 3D kernels of three and four phases, both 2D tiles in FP64, and
the two-segment march at a ragged end.
Tolerances of the plain step after 100 steps (test_parity_gpu): FP64 1e-10 (U
and the population deviations 1e-8), FP32 1e-5."""
import numpy as np
import pytest

from parity import device_run, reference, rel_err
from paper_2608_26908_gb300 import gpflbm, inputs, slabs

pytestmark = pytest.mark.gpu

TILT = [[0.3 if (a == 0) != (b == 0) else 0.0 for b in range(4)] for a in range(4)]
SLOPES = [[0.4, -0.2], [0.1, 0.3], [-0.3, 0.05], [0.2, 0.2]]


def _model(sc, model):
    p, NP = sc["params"], sc["n_phases"]
    if model in ("aniso", "tilt", "combined"):
        for a in range(1, NP):
            p["delta"][0][a] = p["delta"][a][0] = 0.03
    if model in ("tilt", "combined"):
        p["tilt"] = [[TILT[a][b] if a < NP and b < NP else 0.0 for b in range(4)] for a in range(4)]
    if model in ("ceqT", "combined"):
        p["dceq_dT"] = [row[:] for row in SLOPES]
        p["G"], p["V"] = 4e-3, 2e-2
    if model in ("shrinkage", "combined"):
        p["eta_rho"] = [0.0] + [0.2 if a < NP else 0.0 for a in range(1, 4)]
    p["gbeta_c"] = [2e-3, 1e-3]
    return sc


def _check(sc, steps, **state):
    ref = reference(sc, steps, **state)
    sim, got = device_run(sc, steps, **state)
    sim.close()
    for k in ("phi", "mu", "c", "rho", "u", "dev"):
        tol = 1e-5 if sc["precision"] == "fp32" else (1e-8 if k in ("u", "dev") else 1e-10)
        assert rel_err(got[k], ref[k]) <= tol, (k, rel_err(got[k], ref[k]))


# FP64 tiles own 30 x 6 columns and march 16 planes
@pytest.mark.parametrize("name,size,lattice,model", [
    ("eutectic3d", (60, 18, 32), 19, "plain"),       # whole tiles
    ("eutectic3d", (31, 13, 17), 19, "ceqT"),        # one cell more on every axis
    ("eutectic3d", (36, 34, 40), 19, "shrinkage"),
    ("eutectic3d", (29, 11, 31), 27, "plain"),       # one cell fewer
    ("dendrite3d", (61, 37, 33), 19, "plain"),
    ("dendrite3d", (60, 24, 48), 27, "tilt"),
    ("dendrite3d", (33, 32, 30), 27, "shrinkage"),
])
def test_3d_fp64(name, size, lattice, model):
    sc = inputs.scenario(name, **dict(zip(("nx", "ny", "nz"), size)), precision="fp64")
    sc["grid"]["lattice"] = lattice
    if name == "eutectic3d":
        sc["init"]["height"] = 9
    _check(_model(sc, model), 25)


def _eutectic3d(size, prec, phases, solutes, lattice=19):
    sc = inputs.scenario("eutectic3d", **dict(zip(("nx", "ny", "nz"), size)), precision=prec)
    sc["grid"]["lattice"] = lattice
    sc["init"]["height"] = 12
    sc["n_phases"], sc["n_solutes"] = phases, solutes
    return sc


@pytest.mark.parametrize("prec,phases,solutes,lattice,model", [
    ("fp32", 4, 2, 19, "aniso"),
    ("fp32", 3, 1, 19, "aniso"),
    ("fp64", 4, 1, 19, "aniso"),
    ("fp64", 3, 2, 27, "aniso"),
    ("fp32", 4, 2, 27, "aniso"),
    ("fp32", 4, 2, 19, "tilt"),
    ("fp64", 3, 1, 19, "tilt"),
    ("fp64", 4, 2, 19, "combined"),
])
def test_3d_anisotropic(prec, phases, solutes, lattice, model):
    _check(_model(_eutectic3d((33, 29, 31), prec, phases, solutes, lattice), model), 25)


@pytest.mark.parametrize("prec,phases,solutes,lattice,model", [
    ("fp32_bf16", 4, 2, 19, "aniso"),
    ("fp32", 3, 1, 19, "aniso"),
    ("fp64", 4, 1, 19, "aniso"),
    ("fp32", 3, 2, 27, "aniso"),
    ("fp32", 4, 2, 19, "tilt"),
    ("fp64", 3, 1, 27, "tilt"),
    ("fp32_f16", 4, 2, 19, "ceqT"),
    ("fp64", 4, 2, 19, "plain"),
    ("fp32", 3, 1, 19, "plain"),
    ("fp32_bf16", 2, 2, 19, "aniso"),
    ("fp64", 2, 1, 27, "tilt"),
])
def test_3d_slabs_match_the_whole_grid(prec, phases, solutes, lattice, model):
    """The same bits, also after a change of parameters from isotropic ones
    (another kernel of the same handle)."""
    def scenario(m):
        return _model(_eutectic3d((40, 34, 32), prec, phases, solutes, lattice), m)

    sc = scenario(model)
    phi0, mu0 = inputs.initial_state(sc)
    layer, steps = 40 * 34, 6
    whole = gpflbm.Sim(scenario("plain"))
    whole.set_state(phi0, mu0)
    whole.step(4)
    whole.set_params(sc)
    whole.set_state(phi0, mu0)
    whole.step(steps)
    ref = whole.fields(("phi", "mu", "f"))
    runs = []
    for r, (v0, n) in enumerate([(0, 9), (9, 2), (11, 21)]):
        sim = gpflbm.Sim(sc, slab=(v0, n))
        sim.set_state(*[a.reshape(-1, 32 * layer)[:, v0 * layer:(v0 + n) * layer].reshape(-1) for a in (phi0, mu0)])
        runs.append((v0, n, slabs.Slab(sim, r, 3)))
    for _ in range(steps):
        slabs.step_all([s for _, _, s in runs])
    for v0, n, s in runs:
        got = s.sim.fields(("phi", "mu", "f"))
        for k in got:
            np.testing.assert_array_equal(got[k], ref[k][:, v0 * layer:(v0 + n) * layer], err_msg=k)


def _case2d(nx, ny, phases, solutes):
    """Stripes of every solid phase below a melt, with blurred edges."""
    sc = inputs.scenario("eutectic2d", nx=nx, ny=ny, precision="fp64")
    ternary = inputs.scenario("eutectic3d", nx=nx, ny=ny, nz=3)["params"]
    for k in ("gamma", "ceq", "S", "A"):
        sc["params"][k] = ternary[k]
    sc["n_phases"], sc["n_solutes"] = phases, solutes
    x, y = np.meshgrid(np.arange(nx), np.arange(ny))
    phi = np.zeros((phases, ny, nx))
    for a in range(1, phases):
        phi[a] = (y < 40 + 5 * a) & (1 + (x // 11) % (phases - 1) == a)
    phi[0] = 1.0 - phi[1:].sum(axis=0)
    for _ in range(2):  # three-cell means: interfaces a few cells wide
        phi = (np.roll(phi, 1, 2) + phi + np.roll(phi, -1, 2)) / 3.0
        up, down = np.concatenate([phi[:, :1], phi[:, :-1]], 1), np.concatenate([phi[:, 1:], phi[:, -1:]], 1)
        phi = (up + phi + down) / 3.0
    mu = 0.02 * np.sin(np.arange(solutes * nx * ny) * 0.37)
    return sc, phi.reshape(-1), mu


# 32 x 8 tiles own 30 x 6 cells: 305 of them on 150 x 366 (the first grid of
# large tiles), 304 on 480 x 114 (the last of small ones)
@pytest.mark.parametrize("nx,ny", [(150, 366), (480, 114)])
@pytest.mark.parametrize("phases,solutes,model", [
    (2, 1, "plain"), (2, 2, "plain"), (3, 2, "plain"), (4, 1, "plain"),
    (2, 2, "shrinkage"), (3, 1, "shrinkage"), (4, 2, "shrinkage"),
    (2, 1, "tilt"), (4, 1, "tilt"),
    (2, 2, "ceqT"), (3, 1, "ceqT"), (4, 2, "ceqT"),
    (2, 1, "combined"), (3, 2, "combined"), (4, 2, "combined"),
])
def test_2d_fp64_on_both_sides_of_the_tile_rule(nx, ny, phases, solutes, model):
    sc, phi0, mu0 = _case2d(nx, ny, phases, solutes)
    _check(_model(sc, model), 12, phi0=phi0, mu0=mu0)


@pytest.mark.parametrize("nz,phases", [(256, 2), (259, 2), (261, 4)])
def test_two_segments_a_march_at_a_ragged_end(nz, phases):
    """16-bit populations: 43 and 44 segments of six planes, marched by twos,
    the last one ragged; the slabs, whose every tile is general, give the same
    bits."""
    sc = inputs.scenario("eutectic3d" if phases == 4 else "dendrite3d", nx=190, ny=180, nz=nz, precision="fp32_f16")
    sc["params"]["gbeta_c"] = [2e-3, 1e-3]
    # tiles of 30 x 14 columns; below 2000 CTAs a march takes one segment
    assert (190 + 29) // 30 * ((180 + 13) // 14) * (((nz + 5) // 6 + 1) // 2) >= 2000
    phi0, mu0 = inputs.initial_state(sc)
    layer, steps = 190 * 180, 3
    whole = gpflbm.Sim(sc)
    whole.set_state(phi0, mu0)
    whole.step(steps)
    ref = whole.fields(("phi", "mu", "f"))
    whole.close()
    runs = []
    for r, (v0, n) in enumerate([(0, 129), (129, nz - 129)]):
        sim = gpflbm.Sim(sc, slab=(v0, n))
        sim.set_state(*[a.reshape(-1, nz * layer)[:, v0 * layer:(v0 + n) * layer].reshape(-1) for a in (phi0, mu0)])
        runs.append((v0, n, slabs.Slab(sim, r, 2)))
    for _ in range(steps):
        slabs.step_all([s for _, _, s in runs])
    for v0, n, s in runs:
        got = s.sim.fields(("phi", "mu", "f"))
        for k in got:
            np.testing.assert_array_equal(got[k], ref[k][:, v0 * layer:(v0 + n) * layer], err_msg=k)
