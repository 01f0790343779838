"""Every variant of the step kernels that a size or a model switches to,
against the FP64 oracle: the 3D tiles in FP64 at their edges, with each model.
Tolerances of the plain step after 100 steps (test_parity_gpu): FP64 1e-10 (U
and the population deviations 1e-8), FP32 1e-5."""
import pytest

from parity import errors
from paper_2608_26908_gb300 import inputs

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


def _check(sc, steps, **kw):
    errs = errors(sc, steps, **kw)[0]
    for k, e in errs.items():
        tol = 1e-5 if sc["precision"] == "fp32" else (1e-8 if k in ("u", "dev") else 1e-10)
        assert e <= tol, (k, e)


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
