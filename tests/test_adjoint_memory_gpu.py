"""Where Sim.adjoint and Sim.vjp take their workspace from."""
import numpy as np
import pytest

from paper_2608_26908_gb300 import gpflbm, inputs

pytestmark = pytest.mark.gpu

OBJ = dict(w_frac=1.0, w_tip=1.0, kappa=2.0, x0=32, y0=28)


def test_vjp_reuses_the_adjoints_workspace():
    """Both take it from torch's cache: a vjp after an adjoint of the same
    horizon needs no more device memory, torch's or any other."""
    import torch

    sc = inputs.scenario("adjoint2d", nx=64, ny=56)
    sim = gpflbm.Sim(sc)
    state = inputs.initial_state(sc)
    H, K = 12, 4
    sim.set_state(*state)
    sim.adjoint(OBJ, H, K)
    sim.set_state(*state)
    need, held = sim.adjoint_workspace_bytes(H, K), torch.cuda.memory_allocated()
    reserved = torch.cuda.memory_reserved()
    torch.cuda.reset_peak_memory_stats()
    sim.vjp(np.ones((11, sim.cells), dtype=sim.dtype), H, K)
    assert torch.cuda.max_memory_allocated() - held >= need
    assert torch.cuda.memory_reserved() == reserved


@pytest.mark.parametrize("error", [TypeError("2^63 bytes"), "oom"])
def test_the_librarys_own_workspace_where_torch_has_none(monkeypatch, error):
    import torch

    sc = inputs.scenario("adjoint2d", nx=64, ny=56)
    sim = gpflbm.Sim(sc)
    state = inputs.initial_state(sc)
    sim.set_state(*state)
    want = sim.adjoint(OBJ, 6, 3)
    sim.set_state(*state)

    def empty(*a, **k):
        raise torch.cuda.OutOfMemoryError("full") if error == "oom" else error

    monkeypatch.setattr(torch, "empty", empty)
    got = sim.adjoint(OBJ, 6, 3)
    assert got[0] == want[0]
    np.testing.assert_array_equal(got[1], want[1])
    np.testing.assert_array_equal(got[2], want[2])
