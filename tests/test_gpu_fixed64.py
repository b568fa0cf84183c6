"""FP64 storage: the fixed-point MRT update and, in the same launch, the nodes
that leave its range and take the FP64 instructions, against the oracle.

One step from a state that holds every kind of node.  Tolerance: either update
is a chain of about ten roundings of terms of at most 4 rho (the e and eps
rows of Eq. 15), so its error is below 10 * 2^-53 * 4 rho = 4.4e-15 rho; the
oracle's own is as large.  With rho <= 2 rho0 and the largest population
above rho0 / 3: 2 * 4.4e-15 * 2 * 3 = 5.3e-14 of the largest population.
"""
import numpy as np
import pytest

import workloads as wl
from helpers import make_pair, moving_bodies, rel_err

pytestmark = pytest.mark.gpu

TOL = 5.3e-14


@pytest.fixture(scope="module", autouse=True)
def _library(gpu_library):
    return gpu_library


def _state(nx, ny, rho0, seed):
    """Near-equilibrium populations with, here and there, a node of each kind that is out of range."""
    rng = np.random.default_rng(seed)
    f = rho0 * wl.random_populations(nx, ny, seed)
    kind = rng.integers(0, 40, (ny, nx))
    f[5][kind == 1] *= -1.0                       # a negative population
    f[6][kind == 2] = 0.0
    f[7][kind == 3] = 1e-12 * rho0                # below the grid's smallest
    f[:, kind == 4] *= 1.8                        # density beyond the range, both ways
    f[:, kind == 5] *= 0.4
    f[1][kind == 6] += 0.45 * rho0                # |j| beyond the range
    f[3][kind == 6] *= 0.1
    return f


@pytest.mark.parametrize("kernel", ["scalar", "scalar48", "scalar40"])
@pytest.mark.parametrize("rho0", [1.0, 0.7, 2.0, 1e-3, 1e20])
@pytest.mark.parametrize("g", [(0.0, 0.0), (1e-3, -2e-3), (0.1, 0.0)])
def test_every_kind_of_node_matches_the_oracle(kernel, rho0, g):
    nx, ny = 67, 45
    p = wl.mixed_bc_box(nx, ny, seed=3, body=moving_bodies(nx, ny)["free"], tau=0.7, rates=wl.random_rates(7))
    p["rho0"], p["g_fluid"] = rho0, g
    f0 = _state(nx, ny, rho0, seed=5)
    gpu, orc = make_pair(p, "f64", f0=f0)
    gpu.set_launch(kernel, 128, 2)
    gpu.step(1)
    orc.step(1)
    assert rel_err(gpu.populations(), orc.populations()) < TOL
    hg, ho = gpu.history(), orc.history()
    assert rel_err(hg[:, 1:4], ho[:, 1:4]) < 1e-10 and rel_err(hg[:, 12:15], ho[:, 12:15]) < 1e-10
