"""The field read-back by 16-byte words (grids that fill the chip, rows a
multiple of a word, aligned destinations) gives the bits of the one-cell-a-
thread form, which a destination off the 16-byte grid takes; and on rows that
end in a partial word only the latter runs, in bounds."""
import ctypes

import numpy as np
import pytest

from paper_2608_26908_gb300 import gpflbm, inputs

pytestmark = pytest.mark.gpu

NAMES = ("phi", "mu", "c", "f", "rho", "u")


def _read(sim, offset):
    import torch

    outs, ptrs = [], []
    for name in NAMES:
        n = sim._planes(name) * sim.cells
        t = torch.full((n + 8,), 7.0, dtype=sim.tdtype, device="cuda")
        outs.append(t)
        ptrs.append(t.data_ptr() + offset * t.element_size())
    mask = sum(gpflbm.FIELD[n] for n in NAMES)
    st = gpflbm.lib().gpflbm_get_fields(sim.h, mask, (ctypes.c_void_p * len(ptrs))(*ptrs), 1,
                                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == gpflbm.OK
    torch.cuda.synchronize()
    got = []
    for name, t in zip(NAMES, outs):
        n = sim._planes(name) * sim.cells
        a = t.cpu().numpy()
        assert (a[:offset] == 7.0).all() and (a[offset + n:] == 7.0).all(), name  # nothing outside
        got.append(a[offset:offset + n])
    return got


@pytest.mark.parametrize("name,size,prec,lattice", [
    ("dendrite2d", dict(nx=400, ny=400), "fp32", 9),
    ("dendrite2d", dict(nx=302, ny=300), "fp64", 9),
    ("eutectic2d", dict(nx=398, ny=420), "fp32_f16", 9),
    ("eutectic3d", dict(nx=64, ny=60, nz=44), "fp32", 19),
    ("dendrite3d", dict(nx=60, ny=64, nz=44), "fp32_bf16", 19),
    ("dendrite3d", dict(nx=52, ny=64, nz=50), "fp32", 27),
    ("eutectic3d", dict(nx=36, ny=40, nz=31), "fp32", 19),  # too small for words
])
def test_words_and_single_cells_read_the_same_fields(name, size, prec, lattice):
    sc = inputs.scenario(name, precision=prec, **size)
    sc["grid"]["lattice"] = lattice
    sc["params"]["gbeta_c"] = [2e-3, 1e-3]
    sim = gpflbm.Sim(sc)
    sim.set_state(*inputs.initial_state(sc))
    sim.step(5)
    wide, single = _read(sim, 0), _read(sim, 1)
    for n, a, b in zip(NAMES, wide, single):
        np.testing.assert_array_equal(a, b, err_msg=n)


@pytest.mark.parametrize("size", [dict(nx=80, ny=64, nz=64), dict(nx=73, ny=66, nz=65), dict(nx=40, ny=36, nz=20)])
def test_write_back_after_an_asynchronous_host_load(size):
    """The write-back that expects another load over the host link beside it
    (the first after an asynchronous load from host memory, on a grid that
    fills the chip) gives the bits of the next one, which does not."""
    import torch

    sc = inputs.scenario("dendrite3d", precision="fp32", **size)
    sim = gpflbm.Sim(sc)
    state = [torch.as_tensor(a, dtype=torch.float32).pin_memory() for a in inputs.initial_state(sc)]
    sim.set_state(*state)
    st = gpflbm.lib().gpflbm_set_state(sim.h, state[0].data_ptr(), state[1].data_ptr(), None, gpflbm.ASYNC, 0,
                                       ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == gpflbm.OK
    sim.step(4)
    first, second = _read(sim, 0), _read(sim, 0)
    for n, a, b in zip(NAMES, first, second):
        np.testing.assert_array_equal(a, b, err_msg=n)
