"""Calls on a stream that does not synchronise with the legacy default stream:
what one call queues is finished before the next one, without a wait between
them, reads or rewrites it."""
import copy

import numpy as np
import pytest

from paper_2608_26908_gb300 import gpflbm, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["dendrite3d", "eutectic3d"])
def test_parameters_changed_with_steps_in_flight(name):
    """Shrinkage off again while shrinkage steps run: the liquid flags of both
    buffers are taken after those steps, so the steps that follow are those of
    a run that waits before the change."""
    import torch

    sc = inputs.scenario(name, nx=120, ny=112, nz=100)
    sc["init"]["height" if name == "eutectic3d" else "radius"] = 30
    shrink = copy.deepcopy(sc)
    shrink["params"]["eta_rho"][1] = 0.1
    state = [torch.as_tensor(a, dtype=torch.float32, device="cuda") for a in inputs.initial_state(sc)]
    torch.cuda.synchronize()

    def run(wait):
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            sim = gpflbm.Sim(sc)
            sim.set_state(*state)
            sim.step(3)
            sim.set_params(shrink)
            sim.step(41)
            if wait:
                torch.cuda.synchronize()
            sim.set_params(sc)
            sim.step(5)
            return sim.fields(("phi", "mu", "f"))

    want, got = run(True), run(False)
    for k in want:
        np.testing.assert_array_equal(got[k], want[k], err_msg=k)


def test_a_state_loaded_right_after_creation_stays():
    """A load on a side stream directly after gpflbm_create waits for the
    clearing of the workspace and is not wiped by it."""
    import torch

    sc = inputs.scenario("eutectic3d", nx=256, ny=256, nz=128)
    phi, mu = (torch.as_tensor(a, dtype=torch.float32, device="cuda") for a in inputs.initial_state(sc))
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        sim = gpflbm.Sim(sc)
        sim.set_state(phi, mu)
        got = sim.fields(("phi", "mu"), device=True)
        side.synchronize()
        assert torch.equal(got["phi"].reshape(-1), phi.reshape(-1))
        assert torch.equal(got["mu"].reshape(-1), mu.reshape(-1))


def test_handles_created_while_another_thread_captures_steps():
    """The steps' stream capture of one thread and the creation of handles in
    another do not disturb each other."""
    import threading

    import torch

    sc = inputs.scenario("dendrite2d", nx=64, ny=48, precision="fp32")
    state = inputs.initial_state(sc)
    errors, done = [], threading.Event()

    def create():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                while not done.is_set():
                    gpflbm.Sim(sc).close()
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            errors.append(e)

    sim = gpflbm.Sim(sc)
    sim.set_state(*state)
    t = threading.Thread(target=create)
    t.start()
    try:
        for _ in range(60):
            sim.set_params(sc)  # drops the captured steps
            sim.step(18)
    finally:
        done.set()
        t.join()
    assert not errors
    torch.cuda.synchronize()
