"""The shower's current at charge speeds that cross less than a cell, about
one cell and several cells per step (the amplitudes of a step are tabulated
up to eight planes and evaluated per edge beyond that), on every field-update
path and in the persistent batch kernel, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-4   # FP32 fields against the FP64 oracle, relative L2 (the parity bar)


@pytest.fixture(scope="module")
def fd():
    import torch
    torch.cuda.set_device(0)
    import paper_1001_5341_gb300 as m
    return m


@pytest.mark.parametrize("speed", [0.3, 1.0, 9.0])
@pytest.mark.parametrize("kernel", [0, 1, 2, "batch"])
def test_current_at_charge_speed(fd, kernel, speed):
    nx, ny, nz, dx, L = 34, 27, 60, 0.02, 3
    dt = W.courant_dt(dx, W.EPS_R_ICE)
    steps = 20 if speed < 2 else 10
    z0, bin_dz, n_bins = 5.3 * dx, dx / 3, 150
    q = oracle.profile_gaussian(z0, bin_dz, n_bins, 12 * dx, 4 * dx, -1e-9)
    w = oracle.lateral_gaussian(L, 1.0)
    xyz = np.array([[nx // 2 + 4, ny // 2 + 2, 9], [nx // 2 - 3, ny // 2, 14]]) * dx
    sim = fd.Simulation(nx, ny, nz, dx, dt, W.EPS_R_ICE, fd.FDTD_PEC)
    ref = oracle.Oracle(nx, ny, nz, dx, dt, W.EPS_R_ICE, fd.FDTD_PEC, 0)
    for s in (sim, ref):
        s.set_shower(q, z0, bin_dz, speed * W.C0, w, L)
        s.set_probes(xyz, steps)
    if kernel == "batch":
        with fd.Batch([sim]) as b:
            b.step(steps)
            b.sync()
    else:
        sim.set_kernel(kernel)
        sim.step(steps)
    ref.step(steps)
    assert np.abs(ref.probes()).max() > 0
    for got, want in ((sim.probes(), ref.probes()), (sim.field("Ez"), ref.field("Ez"))):
        assert np.linalg.norm(got - want) <= TOL * np.linalg.norm(want)
    sim.close()
