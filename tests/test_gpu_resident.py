"""Small PEC and Mur grids step many times in one launch, bricks of the grid
resident on the SMs: the fields and the detector traces are bit for bit those
of single-step launches (the same expressions on the same values), with a
remainder of every kind in the columns, rows and planes, and the smallest and
the largest grid that qualify."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fd():
    import torch
    torch.cuda.set_device(0)
    import paper_1001_5341_gb300 as m
    return m


@pytest.mark.parametrize("boundary", ["FDTD_PEC", "FDTD_MUR1"])
@pytest.mark.parametrize("shape", [(4, 4, 4), (30, 33, 40), (65, 16, 7), (96, 96, 96), (127, 101, 95)])
def test_resident_steps_equal_single_steps(fd, shape, boundary):
    nx, ny, nz = shape
    dx, steps = 0.02, 75
    dt = W.courant_dt(dx, W.EPS_R_ICE)
    rng = np.random.default_rng(nx)
    start = {c: rng.standard_normal((nz + 1, ny + 1, nx + 1)).astype(np.float32) for c in ("Ex", "Ey", "Ez", "Hx", "Hz")}
    nodes = np.stack([rng.integers(1, n, 40) for n in shape], 1)
    runs = []
    for single in (True, False):
        sim = fd.Simulation(nx, ny, nz, dx, dt, W.EPS_R_ICE, getattr(fd, boundary))
        sim.set_kernel(1)
        L = 1
        sim.set_shower(oracle.profile_gaussian(1.0 * dx, dx / 3, 9, 2 * dx, dx, -1e-9), 1.0 * dx, dx / 3, 0.9 * W.C0,
                       oracle.lateral_gaussian(L, 1.0), L)
        for c, v in start.items():
            sim.set_field(c, 1e-3 * v)
        sim.set_probes(nodes * dx, steps + 4)
        if single:
            for _ in range(steps):
                sim.step(1)
        else:
            sim.step(steps - 2)
            sim.step(2)
        sim.sync()
        out = [sim.probes()] + [sim.field(c) for c in ("Ex", "Ey", "Ez", "Hx", "Hy", "Hz")]
        sim.step(1)   # a single step goes on from the set the last launch wrote
        out.append(sim.field("Ez"))
        runs.append((out, sim.launches))
        sim.close()
    (want, many), (got, few) = runs
    assert few < many // 4
    for g, w in zip(got, want):
        assert np.isfinite(w).all() and np.abs(w).max() > 0
        assert np.array_equal(g, w)


def test_resident_handles_side_by_side(fd):
    """Handles on streams of their own step at the same time, and one whose
    detectors crowd a single brick falls back to single steps."""
    import torch
    dx, steps, n = 0.02, 300, 40
    dt = W.courant_dt(dx, W.EPS_R_ICE)
    start = np.random.default_rng(3).standard_normal((n + 1, n + 1, n + 1)).astype(np.float32)
    nodes = np.array([[9, 8, 7]])
    sims = []
    for crowd in (1, 1, 1, 400):
        st = torch.cuda.Stream()
        sim = fd.Simulation(n, n, n, dx, dt, W.EPS_R_ICE, fd.FDTD_MUR1, stream=st.cuda_stream)
        sim.set_kernel(1)
        sim.set_field("Ez", start)
        sim.set_probes(np.repeat(nodes, crowd, 0) * dx, steps)
        sims.append((sim, st))
    for sim, _ in sims:
        sim.step(steps)
    traces = [sim.probes() for sim, _ in sims]
    launches = [sim.launches for sim, _ in sims]
    for sim, _ in sims:
        sim.close()
    assert max(launches[:3]) < steps < launches[3]
    for t in traces:
        assert np.abs(t).max() > 0 and np.array_equal(t, np.repeat(traces[0], len(t), 0))


@pytest.mark.parametrize("shape,npml", [((30, 33, 40), 0), ((130, 20, 12), 0), ((128, 128, 160), 8)])
def test_captured_steps_replay(fd, shape, npml):
    """An even number of steps captured into a graph (no shower, no detectors)
    replays as that many further steps, on every grid whose default steps go
    several to a launch."""
    import torch
    nx, ny, nz = shape
    dx = 0.02
    dt = W.courant_dt(dx, W.EPS_R_ICE)
    b = fd.FDTD_CPML if npml else fd.FDTD_PEC
    start = np.random.default_rng(5).standard_normal((nz + 1, ny + 1, nx + 1)).astype(np.float32)
    start[:npml + 2] = start[-npml - 2:] = 0
    start[:, :npml + 2] = start[:, -npml - 2:] = 0
    start[:, :, :npml + 2] = start[:, :, -npml - 2:] = 0
    st = torch.cuda.Stream()
    sim = fd.Simulation(nx, ny, nz, dx, dt, W.EPS_R_ICE, b, npml, stream=st)
    ref = fd.Simulation(nx, ny, nz, dx, dt, W.EPS_R_ICE, b, npml)
    for s in (sim, ref):
        s.set_field("Ez", start)
        s.sync()
    ref.set_kernel(1)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=st):
        sim.step(4)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    for _ in range(12):
        ref.step(1)
    for c in ("Ex", "Ez", "Hy"):
        want = ref.field(c)
        assert np.abs(want).max() > 0 and np.array_equal(sim.field(c), want)
    sim.close()
    ref.close()
