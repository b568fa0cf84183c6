"""FP64 storage at the ends of the accepted penalization and relaxation
parameters, on every stepping path, against the oracle.

One step; tolerance 5.3e-14 of the largest population (two chains of ten
roundings of terms of at most 4 rho, the populations of rho <= 2 rho0 above
rho0 / 3).
"""
import numpy as np
import pytest

import workloads as wl
from helpers import make_pair, moving_bodies, rel_err

pytestmark = pytest.mark.gpu

TOL = 5.3e-14
ENDS = [dict(eta=e) for e in (1e-9, 1.2e-10, 1.1e-10, 1e-12, 1e-20)] + [
    {"s7": 2 - 1e-10}, {"s8": 2 - 1e-10}, {"s7": 1e-10, "g": (1e-3, 0.0)}, {"s8": 1e-10, "g": (1e-3, 0.0)}]


@pytest.fixture(scope="module", autouse=True)
def _library(gpu_library):
    return gpu_library


def _ended(p, end):
    p["s"] = list(p["s"])
    for k, v in end.items():
        if k == "eta":
            p["eta"] = v
        elif k == "g":
            p["g_fluid"] = v
        else:
            p["s"][int(k[1:])] = v
    return p


@pytest.mark.parametrize("end", ENDS, ids=str)
@pytest.mark.parametrize("path", ["scalar", "resident", "several"])
def test_one_step_at_the_ends_of_the_parameters(end, path):
    nx, ny = 67, 45
    bodies = moving_bodies(nx, ny)
    p = _ended(wl.mixed_bc_box(nx, ny, seed=3, body=dict(bodies["free"], omega=0.0), tau=0.7), end)
    if path == "several":
        p["bodies"] = [dict(p.pop("body"), radius=6.0), dict(bodies["imposed"], radius=5.0, x=50.0, y=30.0)]
    gpu, orc = make_pair(p, "f64", f0=wl.random_populations(nx, ny, seed=5, amp=0.03))
    if path != "several":
        gpu.set_launch(path, 128, 2)
    gpu.step(1)
    orc.step(1)
    assert rel_err(gpu.populations(), orc.populations()) < TOL
    for k in range(2 if path == "several" else 1):
        hg, ho = gpu.history(0, 1, body=k), orc.history(0, 1, body=k)
        # sums of some hundred terms of the populations' size
        assert rel_err(hg[:, 1:4], ho[:, 1:4]) < 1e-10 and rel_err(hg[:, 12:15], ho[:, 12:15]) < 1e-10
    gpu.close()


@pytest.mark.parametrize("eta", [1.2e-10, 1.1e-10, 1e-20])
def test_allocation_free_step_at_the_smallest_eta(eta):
    import torch
    import paper_1905_05110_gb300 as vp
    from test_zz_no_alloc import _caller_buffers, _problem, _state_bytes, _stored_to_full
    p = dict(_problem("disk"), eta=eta)
    gpu, orc = make_pair(p, "f64", hist_cap=8)
    dev = torch.device("cuda")
    lat, body = vp.lattice_desc(p, "f64"), vp.body_desc(p["body"])
    sizes, pops, state = _caller_buffers(lat, body, 8, dev)
    src = gpu._tensors["f0"]
    off = (-src.data_ptr()) % 256
    pops[0].copy_(src[off:off + int(sizes.populations)])
    sb = _state_bytes(p["body"])
    state[:sb.size].copy_(torch.from_numpy(sb))
    vp.vplbm_step_noalloc(lat, body, [t.data_ptr() for t in pops], state.data_ptr(), None, 8, 1,
                          torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    orc.step(1)
    raw = pops[1].cpu().numpy().view(np.float64)
    assert rel_err(_stored_to_full(raw, p["nx"], p["ny"], "f64"), orc.populations()) < TOL
    gpu.close()


@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
@pytest.mark.parametrize("rho0", [1.0, 0.99])
def test_equilibrium_of_fast_nodes(precision, rho0):
    """Velocities of up to 1/4 in each direction: the stored populations against FP64 arithmetic, within the rounding of
    the storage (half a unit of the deviation; FP16: of its smallest step too)."""
    import paper_1905_05110_gb300 as vp
    v = np.array([-0.249, -0.22, -0.19, -0.1, 0.0, 0.1, 0.19, 0.22, 0.249])
    ux, uy = np.meshgrid(v, v)
    rho = rho0 * (1 + 0.01 * np.random.default_rng(4).uniform(-1, 1, ux.shape))
    p = wl.periodic_box(9, 9)
    p["rho0"] = rho0
    sim = vp.Simulation(p, precision, history_capacity=4)
    sim.init_equilibrium(rho, ux, uy)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    c = np.array([[0, 0], [1, 0], [0, 1], [-1, 0], [0, -1], [1, 1], [-1, 1], [-1, -1], [1, -1]], dtype=float)
    cu = c[:, 0, None, None] * ux + c[:, 1, None, None] * uy
    feq = w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy))
    unit = {"f64": 0.0, "f32": 2.0 ** -24, "f16": 2.0 ** -11}[precision]
    err = np.abs(sim.populations() - feq) - unit * np.abs(feq - w * rho0)
    assert np.max(err) < TOL + (6e-8 if precision == "f16" else 0)
    sim.close()


@pytest.mark.parametrize("u", [1e-6, 1e-15, 1e-20, 1e-28])
def test_equilibrium_of_slow_nodes(u):
    """FP32 storage keeps the relative precision of any velocity: half a unit of each stored deviation."""
    import paper_1905_05110_gb300 as vp
    p = wl.periodic_box(8, 6)
    sim = vp.Simulation(p, "f32", history_capacity=4)
    sim.init_equilibrium(None, u, -0.5 * u)
    c = np.array([[0, 0], [1, 0], [0, 1], [-1, 0], [0, -1], [1, 1], [-1, 1], [-1, -1], [1, -1]], dtype=float)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
    cu, u2 = c @ np.array([u, -0.5 * u]), 1.25 * u * u
    want = w * (3 * cu + 4.5 * cu * cu - 1.5 * u2)
    off = (-sim._tensors["f0"].data_ptr()) % 256
    ps = (8 * 6 + 127) // 128 * 128
    got = sim._tensors["f0"][off:off + 9 * ps * 4].cpu().numpy().view(np.float32).reshape(9, ps)[:, :48].astype(float)
    assert np.all(np.abs(got - want[:, None]) <= 1.01 * 2.0 ** -24 * np.abs(want[:, None]) + 1e-45)
    sim.close()


@pytest.mark.parametrize("precision,u", [("f32", 0.05), ("f32", 1e-9), ("f32", 1e-14), ("f32", 1e-25), ("f16", 0.05), ("f16", 1e-3)])
def test_fields_of_a_slow_flow(precision, u):
    """u of FP32 / FP16 storage against the stored deviations' own sums, for a flow of any speed: FP64 rounding."""
    import paper_1905_05110_gb300 as vp
    nx, ny = 40, 32
    p = wl.periodic_box(nx, ny)
    sim = vp.Simulation(p, precision, history_capacity=4)
    rng = np.random.default_rng(9)
    ux, uy = u * rng.uniform(-1, 1, (2, ny, nx))
    sim.init_equilibrium(None, ux, uy)
    off = (-sim._tensors["f0"].data_ptr()) % 256
    ps = (nx * ny + 127) // 128 * 128
    dt = np.float32 if precision == "f32" else np.float16
    raw = sim._tensors["f0"][off:off + 9 * ps * dt().nbytes].cpu().numpy().view(dt)
    d = raw.reshape(9, ps)[:, :nx * ny].reshape(9, ny, nx).astype(np.longdouble)
    c = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
    d = np.array([np.roll(d[a], (c[a][1], c[a][0]), (0, 1)) for a in range(9)])   # the pulled ones
    rho = 1 + d.sum(0)
    got = sim.fields()
    want = (rho, sum(c[a][0] * d[a] for a in range(9)) / rho, sum(c[a][1] * d[a] for a in range(9)) / rho)
    for g, w in zip(got, want):
        assert np.max(np.abs(g - w)) < 1e-15 * np.max(np.abs(w))
    sim.close()


@pytest.mark.parametrize("kernel", ["scalar", "resident"])
@pytest.mark.parametrize("g", [(1e-9, -2e-9), (1e-12, 0.0), (3e-14, 1e-15)])
def test_momentum_gained_from_a_uniform_acceleration(kernel, g):
    """FP64 storage, periodic: rho g per node and step.  Tolerance: five deviations of the mean of n roundings of at most
    1e-17 rho a node and step (doubles of 2^-57 and 2^-59, half a unit each)."""
    import paper_1905_05110_gb300 as vp
    nx, ny, steps = 67, 45, 100
    p = wl.periodic_box(nx, ny, tau=0.7, g_fluid=g)
    sim = vp.Simulation(p, "f64", history_capacity=4)
    sim.set_launch(kernel, 128, 2)
    sim.set_populations(wl.random_populations(nx, ny, seed=11, amp=0.03))
    c = np.array([[0, 1, 0, -1, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1]])
    f0 = sim.populations().astype(np.longdouble)
    sim.step(steps)
    f1 = sim.populations().astype(np.longdouble)
    n = nx * ny * steps
    gain = np.tensordot(c, f1 - f0, axes=(1, 0)).sum(axis=(1, 2)) / n
    mean_rho = f0.sum() / (nx * ny)
    assert np.max(np.abs(gain - mean_rho * np.array(g))) < 5 * 1e-17 / np.sqrt(n)
    sim.close()
