"""The resident kernel as a user's program meets it: what the launch queries
say of a context that runs it by default, after a trial run or on request."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library(gpu_library):
    return gpu_library


def _sim(precision="f32", nx=96, ny=64, **kw):
    import paper_1905_05110_gb300 as vp
    p = wl.channel_fixed_disk(nx, ny, diameter=12, center=(30, 31))
    sim = vp.Simulation(p, precision, history_capacity=64, **kw)
    sim.init_from_problem()
    return sim


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_launch_names_the_kernel_that_runs_and_is_taken_back(precision):
    sim = _sim(precision)
    named = sim.launch()
    assert named[0] == "resident"
    sim.set_launch("scalar48", 128, 2)
    assert sim.launch() == ("scalar48", 128, 2)
    sim.set_launch(*named)
    assert sim.launch() == named
    sim.set_launch("scalar48", 128, 2)
    sim.set_launch("resident")            # keeps the one-step kernel and blocks
    assert sim.launch() == ("resident", 128, 2)
    sim.set_launch(*sim.launch())
    assert sim.launch() == ("resident", 128, 2)
    one_step = sim.autotune(8)
    named = sim.launch()
    assert named == ("resident",) + one_step[1:] and one_step[0] != "resident"
    other = _sim(precision)
    other.set_launch(*named)
    assert other.launch() == named
    for s in (sim, other):
        s.step(9)
    assert np.array_equal(sim.populations(), other.populations())
    other.close()
    sim.close()


def test_wait_limit_of_a_default_context():
    import paper_1905_05110_gb300 as vp
    sim = _sim()
    vp.vplbm_inject_wait_timeout(sim.ctx, True)
    sim.step(2)
    with pytest.raises(vp.VplbmError) as ei:
        sim.sync()
    assert ei.value.status == 5
    vp.vplbm_inject_wait_timeout(sim.ctx, False)
    sim.init_from_problem()
    sim.step(8)
    sim.sync()
    sim.close()


def test_lattice_that_does_not_fit_names_its_kernel():
    import paper_1905_05110_gb300 as vp
    sim = vp.Simulation(wl.oscillating_disk(), "f32", history_capacity=64)
    assert sim.launch() == ("scalar40", 256, 1)
    with pytest.raises(vp.VplbmError) as ei:
        sim.set_launch("resident")
    assert ei.value.status == 6
    sim.close()


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_launch_counts_are_of_launches(precision):
    import paper_1905_05110_gb300 as vp
    sim = _sim(precision)
    sim.step(70)
    sim.step(1)
    assert sim.launches == 2 and sim.kernel_launches() == {"one_step": 0, "two_step": 0, "lookahead": 0, "tma": 0, "resident": 2}
    assert vp.vplbm_get_resident_launches(sim.ctx) == (2, 71)
    sim.set_launch("scalar48", 128, 2)
    sim.step(40)
    assert sim.launches == 42 == sum(sim.kernel_launches().values())
    sim.sync()
    sim.close()


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_no_device_memory_beside_the_callers_buffers(precision):
    """A free body's workspace is of some MB; a context on the caller's buffers takes it from these."""
    import torch
    import paper_1905_05110_gb300 as vp
    nx, ny = (700, 400) if precision == "f32" else (400, 240)
    r = ny / 3.0
    body = {"radius": r, "x": nx * 0.5, "y": ny * 0.5, "motion": "free", "mass": 4 * r * r, "inertia": r ** 4, "dof_mask": 7,
            "u_ref": 0.05, "d_ref": 2 * r}
    p = wl.mixed_bc_box(nx, ny, seed=2, body=body)
    first = vp.Simulation(p, precision, history_capacity=64)
    first.step(20)      # the kernels are loaded by their first launch
    first.init_equilibrium()
    sim = vp.Simulation(p, precision, history_capacity=64)
    assert sim.launch()[0] == "resident"
    f = sim.populations()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for state in ("rest", "equilibrium", "populations"):
        if state == "equilibrium":
            sim.init_equilibrium()
        elif state == "populations":
            sim.set_populations(f)
        sim.step(20)
        sim.sync()
    assert torch.cuda.mem_get_info()[0] == free
    assert vp.vplbm_get_resident_launches(sim.ctx) == (3, 60)
    first.close()
    sim.close()


def test_a_refused_launch_is_not_the_end_of_the_kernel():
    import paper_1905_05110_gb300 as vp
    a, b = _sim(), _sim()
    a.set_launch("resident", 128, 2)
    a.step(5)
    vp.vplbm_inject_wait_timeout(a.ctx, 2)
    a.step(40)      # launched one by one
    assert a.kernel_launches() == {"one_step": 40, "two_step": 0, "lookahead": 0, "tma": 0, "resident": 1}
    assert a.autotune(4)[0] != "resident" and a.launch()[0] != "resident"   # measured what can be launched
    a.set_launch("resident")
    vp.vplbm_inject_wait_timeout(a.ctx, 0)
    a.step(7)
    assert a.kernel_launches()["resident"] == 2
    b.step(52)
    assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()


@pytest.mark.parametrize("precision,limit", [("f32", 3), ("f64", 2)])
def test_contexts_on_many_streams_step_by_launches(precision, limit):
    """Resident launches of different streams cannot overlap: beyond the limit the contexts' single launches do."""
    import torch
    streams = [torch.cuda.Stream() for _ in range(limit)]
    sims = [_sim(precision, stream=s) for s in streams]
    same = _sim(precision, stream=streams[0])           # on a stream in use already
    assert all(s.launch()[0] == "resident" for s in sims + [same])
    asked = _sim(precision, stream=torch.cuda.Stream())
    crowd = sims + [same]
    assert all(s.launch()[0] != "resident" for s in crowd + [asked])
    asked.set_launch("resident")
    assert asked.launch()[0] == "resident"
    for s in crowd + [asked]:
        s.step(40)
    for s in crowd + [asked]:
        s.sync()
    assert all(s.kernel_launches() == {"one_step": 40, "two_step": 0, "lookahead": 0, "tma": 0} for s in crowd)
    assert asked.kernel_launches()["resident"] == 1
    asked.close()
    assert all(s.launch()[0] == "resident" for s in crowd)
    for s in crowd:
        s.step(9)
        s.sync()
        assert s.kernel_launches()["resident"] == 1
        assert np.array_equal(s.populations(), crowd[0].populations())
    ref = _sim(precision, stream=streams[0])
    ref.step(49)
    assert np.array_equal(ref.populations(), crowd[0].populations())
    for s in crowd + [ref]:
        s.close()
