"""The conservation totals where their integer population sum and their
skipped phase terms could go wrong: populations of one magnitude, of a spread
at and beyond the 2^24 window of the integer sum, zeros of both signs, cells
of one, two, three and four phases, phases of different A, and values that are
not finite.  Every total equals, bit for bit, the host re-summation of the
downloaded state in the documented order."""
import numpy as np
import pytest

from oracle import oracle
from paper_2608_26908_gb300 import gpflbm, inputs
from test_invariants_gpu import host_invariants

pytestmark = pytest.mark.gpu


def _state(sc, seed):
    rng = np.random.default_rng(seed)
    n = inputs.cells(sc)
    NP, NC = sc["n_phases"], sc["n_solutes"]
    present = 1 + np.arange(n) % NP  # phases in a cell: 1 .. NP, side by side in a warp
    raw = rng.random((NP, n)) * (np.argsort(rng.random((NP, n)), axis=0) < present)
    phi = raw / raw.sum(axis=0)
    phi[:, present == 1] = np.round(phi[:, present == 1])
    mu = rng.normal(size=(NC, n)) * 10.0 ** rng.integers(-12, 1, size=(NC, n))
    mu[:, ::7] = 0.0
    mu[:, 3::7] = -0.0
    f = oracle.rest_populations(sc).reshape(-1, n)
    q = f.shape[0]
    # deviations of a cell: magnitudes 2^e with e spread over 0, 20, 24, 25 and
    # 40 binades, then rounded by f's own format
    spread = np.array([0, 20, 24, 25, 40])[np.arange(n) % 5]
    e = -6.0 - rng.random((q, n)) * spread
    d = np.where(rng.random((q, n)) < 0.5, -1.0, 1.0) * 2.0 ** e
    d[:, ::11] = 0.0
    return phi.reshape(-1), mu.reshape(-1), (f + d).reshape(-1)


@pytest.mark.parametrize("name,size,prec,lattice", [
    ("dendrite2d", dict(nx=70, ny=37), "fp32", 9),
    ("dendrite2d", dict(nx=33, ny=21), "fp64", 9),
    ("eutectic2d", dict(nx=129, ny=31), "fp32_f16", 9),
    ("eutectic3d", dict(nx=37, ny=22, nz=25), "fp32", 19),
    ("eutectic3d", dict(nx=24, ny=20, nz=11), "fp32_bf16", 19),
    ("eutectic3d", dict(nx=24, ny=20, nz=11), "fp32", 27),
    ("eutectic3d", dict(nx=19, ny=20, nz=11), "fp64", 19),
])
@pytest.mark.parametrize("same_a", [True, False])
def test_totals_bit_for_bit_on_edge_values(name, size, prec, lattice, same_a):
    sc = inputs.scenario(name, precision=prec, **size)
    sc["grid"]["lattice"] = lattice
    if not same_a:
        sc["params"]["A"] = [1.0, 1.3, 0.7, 2.0]
    sim = gpflbm.Sim(sc)
    sim.set_state(*_state(sc, 5))
    m, s, fr, _ = sim.invariants()
    hm, hs, hf = host_invariants(sim, sc)
    assert (m, tuple(s), fr) == (hm, tuple(hs), hf)


@pytest.mark.parametrize("where", ["phi", "mu", "f"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_one_value_that_is_not_finite_is_reported(where, bad):
    sc = inputs.scenario("eutectic3d", nx=24, ny=20, nz=11)
    state = [a.copy() for a in _state(sc, 6)]
    state[("phi", "mu", "f").index(where)][1234] = bad
    sim = gpflbm.Sim(sc)
    sim.set_state(*state)
    assert sim.invariants(allow_nonfinite=True)[3] == gpflbm.ERR_NONFINITE
