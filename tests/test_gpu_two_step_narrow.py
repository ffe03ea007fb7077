"""Two-step passes on grids of up to 128 columns, which are one tile with the x
layers inside it: the last lane full, short and empty, one to several tile rows,
z layers with and without planes between them, and many detectors in one row,
against the FP64 oracle."""
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


@pytest.mark.parametrize("npml", [0, 4, 10])
@pytest.mark.parametrize("shape", [(128, 28, 60), (127, 33, 44), (122, 29, 28), (30, 57, 40)])
def test_one_tile_column(fd, shape, npml):
    nx, ny, nz = shape
    dx, L, steps = 0.02, 2, 25
    dt = W.courant_dt(dx, W.EPS_R_ICE)
    lo = npml + 1
    q = oracle.profile_gaussian((lo + 1) * dx, dx / 3, 30, 4 * dx, 2 * dx, -1e-9)
    w = oracle.lateral_gaussian(L, 1.0)
    row = [(i, ny // 2, k) for i in range(lo, nx - lo) for k in (lo, nz // 2)]
    edge = [(i, j, nz // 2) for i in (lo, nx - lo) for j in (lo, ny - lo)]
    xyz = np.array(row + edge) * dx
    b = fd.FDTD_CPML if npml else fd.FDTD_PEC
    sim = fd.Simulation(nx, ny, nz, dx, dt, W.EPS_R_ICE, b, npml)
    sim.set_kernel(2)
    ref = oracle.Oracle(nx, ny, nz, dx, dt, W.EPS_R_ICE, b, npml)
    for s in (sim, ref):
        s.set_shower(q, (lo + 1) * dx, dx / 3, 0.9 * W.C0, w, L)
        s.set_probes(xyz, steps)
        s.step(steps)
    assert np.abs(ref.probes()).max() > 0
    # E and H as whole vectors: Hz of a vertical current is zero but for round-off
    pairs = [(sim.probes(), ref.probes())]
    pairs += [tuple(np.stack([s.field(f + c) for c in "xyz"]) for s in (sim, ref)) for f in "EH"]
    for got, want in pairs:
        assert np.linalg.norm(got - want) <= TOL * np.linalg.norm(want)
    sim.close()
