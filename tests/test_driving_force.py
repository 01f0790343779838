"""The driving force of the 3D step (three and four phases) in FP32 against
64 bits, compiled for the host: on cells with a trace of a phase beside a nearly
pure one, each component is right to the rounding of its own terms."""
import subprocess

import numpy as np
import pytest

from paper_2608_26908_gb300 import build

SOURCE = r"""
#include <cstdio>
#include "gpflbm_kernels.cuh"
template <int NP>
int run() {
  float p[NP], psi[NP], d[NP];
  for (;;) {
    if (std::fread(p, sizeof(p), 1, stdin) != 1) return 0;
    if (std::fread(psi, sizeof(psi), 1, stdin) != 1) return 1;
    gpflbm::driving_force<NP>(p, psi, d);
    std::fwrite(d, sizeof(d), 1, stdout);
  }
}
int main(int argc, char** argv) { return argc > 1 && argv[1][0] == '3' ? run<3>() : run<4>(); }
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("driving_force")
    (d / "main.cu").write_text(SOURCE)
    cmd = [build.nvcc()] + build.ARCH + build.FLAGS + [str(d / "main.cu"), "-o", str(d / "main")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "main")


def _exact(p, psi):
    """sum_b psi_b dh_b/dphi_a pair by pair, and the sum of the magnitudes."""
    n, NP = p.shape
    d, size = np.zeros((n, NP)), np.zeros((n, NP))
    for a in range(NP):
        for b in range(NP):
            others = [g for g in range(NP) if g not in (a, b)]
            if a == b:
                pairs = sum(p[:, g] * p[:, h] for i, g in enumerate(others) for h in others[i + 1:])
                t = 6 * p[:, a] * (1 - p[:, a]) + 2 * pairs
            else:
                t = 2 * p[:, b] * sum(p[:, g] for g in others)
            d[:, a] += psi[:, b] * t
            size[:, a] += np.abs(psi[:, b]) * t
    return d, size


@pytest.mark.parametrize("NP", [3, 4])
def test_driving_force_of_trace_phases(program, NP):
    rng = np.random.default_rng(1)
    n = 4000
    p = 10.0 ** rng.uniform(-7, 0, size=(n, NP))
    p[np.arange(n), rng.integers(0, NP, n)] = 1.0
    p[rng.random((n, NP)) < 0.1] = 0.0
    p[p.sum(axis=1) == 0, 0] = 1.0
    p = (p / p.sum(axis=1, keepdims=True)).astype(np.float32)
    psi = (rng.normal(size=(n, NP)) * 10.0 ** rng.uniform(-2, 1, size=(n, 1))).astype(np.float32)
    data = np.concatenate([p, psi], axis=1).astype(np.float32).tobytes()
    r = subprocess.run([program, str(NP)], input=data, capture_output=True)
    assert r.returncode == 0
    got = np.frombuffer(r.stdout, dtype=np.float32).reshape(n, NP).astype(np.float64)
    want, size = _exact(p.astype(np.float64), psi.astype(np.float64))
    # no term passes through more than a dozen roundings, each half a unit of
    # at most the sum of the magnitudes (the smallest normals: absolute)
    assert (np.abs(got - want) <= 12 * 2.0 ** -24 * size + 1e-37).all()
