"""The resident kernel (many steps of a small lattice in one launch) against
the one-step kernel.

Populations, poses and the convective outlet's state equal the one-step
kernel's bit for bit wherever the body's path does not depend on the force
(a free body is driven by sums added in another order, and is compared within
their rounding).  Sizes: one tile, several, ragged ones, tile edges next to
lattice edges and inside the body, each number of nodes per thread that the
kernel is built for, and the largest lattice it takes.
"""
import numpy as np
import pytest

import workloads as wl
from helpers import REC, moving_bodies, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library(gpu_library):
    return gpu_library


BCS = [("periodic", "periodic", "periodic", "periodic"), ("velocity", "zerograd", "noslip", "velocity"),
       ("velocity", "convective", "symmetry", "symmetry"), ("periodic", "periodic", "symmetry", "noslip"),
       ("zerograd", "zerograd", "periodic", "periodic")]


def _pair(p, precision, steps, f0=None, rtol=1e-9):
    """Run `steps` (a list of calls) on both kernels; populations and poses, then the force records."""
    import paper_1905_05110_gb300 as vp
    runs = []
    for kernel in ("scalar", "resident"):
        sim = vp.Simulation(p, precision, history_capacity=512)
        sim.set_launch(kernel, 128, 2)
        if f0 is None:
            sim.init_from_problem()
        else:
            sim.set_populations(f0)
        for n in steps:
            sim.step(n)
        assert sim.launch()[0] == kernel
        runs.append((sim.populations(), sim.history(max(0, sim.nstep - 512)), np.concatenate(sim.body_state()), sim.nstep))
        sim.close()
    (f1, h1, b1, n1), (f2, h2, b2, n2) = runs
    assert n1 == n2
    return f1, h1, b1, f2, h2, b2


def _same(p, precision, steps, f0=None):
    f1, h1, b1, f2, h2, b2 = _pair(p, precision, steps, f0)
    assert np.array_equal(f1, f2)
    assert np.array_equal(b1, b2)
    exact = [REC[k] for k in ("t", "x", "y", "theta", "vx", "vy", "omega", "n_solid")]
    assert np.array_equal(h1[:, exact], h2[:, exact])
    for k in ("fx", "fy", "torque", "fpen_x", "fpen_y", "tpen"):
        # float-float (44-bit) or FP64 sums of a few hundred terms in another order
        assert rel_err(h2[:, REC[k]], h1[:, REC[k]]) < 1e-9, k


@pytest.mark.parametrize("bcs", BCS)
@pytest.mark.parametrize("size", [(5, 4), (16, 9), (67, 45), (131, 97)])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_boundaries_from_a_random_state(bcs, size, precision):
    nx, ny = size
    w, e, s, n = bcs
    p = wl.mixed_bc_box(nx, ny, seed=nx, west=w, east=e, south=s, north=n, rates=wl.random_rates(ny),
                        body=moving_bodies(nx, ny)["imposed"] if nx > 20 else None)
    if e == "convective":
        p["bc"]["east"] = {"kind": "convective", "u": (0.31, 0.0)}
    _same(p, precision, [1, 2, 37], wl.random_populations(nx, ny, seed=3, amp=0.03))


@pytest.mark.parametrize("motion", ["fixed", "imposed", "free"])
@pytest.mark.parametrize("shape", ["disk", "ellipse", "rectangle"])
@pytest.mark.parametrize("collision", ["mrt", "bgk"])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_bodies(motion, shape, collision, precision):
    nx, ny = 150, 110
    body = dict(moving_bodies(nx, ny)[motion], shape=shape)
    if shape != "disk":
        body["radius_b"] = 0.6 * body["radius"]
    p = wl.mixed_bc_box(nx, ny, seed=5, body=body, tau=0.62)
    p["bc"]["west"] = {"kind": "velocity", "u": (0.05, 0.0)}
    p["collision"] = collision
    if motion != "free":
        _same(p, precision, [40, 3, 50])
        return
    f1, h1, b1, f2, h2, b2 = _pair(p, precision, [40, 3, 50])
    # the pose follows the force sums: a difference of 1e-13 of the force
    # over a mass of some hundred, integrated over 93 steps
    assert np.max(np.abs(b1 - b2)) < 1e-10
    assert rel_err(f2, f1) < (1e-6 if precision == "f32" else 1e-11)
    assert np.array_equal(h1[:, REC["n_solid"]], h2[:, REC["n_solid"]])


@pytest.mark.parametrize("precision,size", [("f32", (300, 250)), ("f32", (600, 400)), ("f32", (1230, 410)),
                                            ("f32", (1024, 512)), ("f64", (300, 200)), ("f64", (512, 256))])
def test_every_number_of_nodes_per_thread(precision, size):
    nx, ny = size
    p = wl.oscillating_disk(nx, ny, diameter=ny / 10.0 + 0.3, x_c=0.31 * nx)
    _same(p, precision, [70])


def test_no_body_and_long_calls():
    p = wl.periodic_box(61, 40, tau=0.8, g_fluid=(1e-6, 0.0))
    _same(p, "f32", [4096 + 5, 2], wl.random_populations(61, 40, seed=2))


def test_wait_gives_up_and_the_context_stays_usable():
    import paper_1905_05110_gb300 as vp
    p = wl.channel_fixed_disk(96, 64, diameter=12, center=(30, 31))
    sim = vp.Simulation(p, "f32", history_capacity=64)
    sim.set_launch("resident")
    sim.init_from_problem()
    sim.step(8)
    f = sim.populations()
    vp.vplbm_inject_wait_timeout(sim.ctx, True)
    sim.step(4)
    with pytest.raises(vp.VplbmError) as ei:
        sim.sync()
    assert ei.value.status == 5
    vp.vplbm_inject_wait_timeout(sim.ctx, False)
    sim.init_from_problem()
    sim.step(8)
    assert np.array_equal(sim.populations(), f)
    sim.close()


def test_captured_steps_are_launched_one_by_one():
    import torch
    import paper_1905_05110_gb300 as vp
    p = wl.channel_fixed_disk(96, 64, diameter=12, center=(30, 31))
    stream = torch.cuda.Stream()
    a = vp.Simulation(p, "f32", history_capacity=64, stream=stream)
    b = vp.Simulation(p, "f32", history_capacity=64, stream=stream)
    for s in (a, b):
        s.init_from_problem()
        s.step(2)
        s.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        a.step(6)
    g.replay()
    torch.cuda.synchronize()
    b.step(6)
    assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()
