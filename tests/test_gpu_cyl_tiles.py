"""The 2D solver's tile path (the default, without cyl_set_kernel) against the
FP64 oracle: one tile and several, ragged last tiles, grids a row or column
over a whole number of tiles, detectors on tile and warp seams and on the
axis, the shower in several tiles, step counts that leave a short launch, and
against the two-kernel path on grids of the larger tile."""
import numpy as np
import pytest

from oracle import cyl_oracle as O
from test_gpu_cyl import _close, _compare, _fields, _shower

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fd():
    import torch
    torch.cuda.set_device(0)
    import paper_1001_5341_gb300 as m
    return m


def _seams(nr, nz, n, seed):
    """Detectors on the multiples of 8 (warp and halo seams) and next to them, and random ones."""
    rng = np.random.default_rng(seed)
    ii = [0, 1, nr - 1] + [k + o for k in range(8, nr, 40) for o in (-1, 0)]
    jj = [1, nz - 1] + [k + o for k in range(8, nz, 40) for o in (-1, 0, 1)]
    pts = [(ii[k % len(ii)], jj[(3 * k) % len(jj)]) for k in range(n)]
    pts += [(int(rng.integers(0, nr)), int(rng.integers(1, nz))) for _ in range(n)]
    return [(min(i, nr - 1), min(max(j, 1), nz - 1)) for i, j in pts]


def _pair(fd, nr, nz, steps, boundary, seed, select=None):
    d = 0.01
    dt = O.courant_dt(d, 3.17)
    sims = [O.CylOracle(nr, nz, d, dt, 3.17, boundary=boundary) if select is None else
            fd.Cylinder(nr, nz, d, dt, 3.17, boundary=boundary), fd.Cylinder(nr, nz, d, dt, 3.17, boundary=boundary)]
    if select is not None:
        sims[0].set_kernel(select)
    F = _fields(seed, nr, nz)
    q, z0, bdz, v, w = _shower(nz, d)
    rz = np.asarray(_seams(nr, nz, 40, seed), np.float64) * d
    for s in sims:
        if isinstance(s, O.CylOracle):
            s.Er[:], s.Ez[:], s.Hp[:] = F
            s.set_probes(rz)
        else:
            for c in range(3):
                s.set_field(c, F[c])
            s.set_probes(rz, steps)
        s.set_shower(q, z0, bdz, v, np.resize(w, min(20, nr)))
        s.step(steps)
    sims[1].sync()
    return sims


@pytest.mark.parametrize("boundary", [O.PEC, O.MUR1])
@pytest.mark.parametrize("nr,nz,steps", [(4, 4, 19), (5, 300, 19), (300, 5, 19), (63, 63, 21), (64, 63, 8), (64, 64, 37),
                                         (65, 112, 37), (112, 111, 37), (113, 128, 29), (129, 130, 16), (200, 333, 43)])
def test_tiles_match_oracle(fd, nr, nz, steps, boundary):
    o, g = _pair(fd, nr, nz, steps, boundary, nr + nz)
    assert g.kernel_info["kernel_name"].startswith("k_cyl_tile")
    _compare(o, g, steps, f"{nr}x{nz}")


@pytest.mark.parametrize("nr,nz", [(900, 701), (240, 5000), (3000, 241), (1400, 1300)])
def test_large_tiles_match_two_kernel_path(fd, nr, nz):
    a, b = _pair(fd, nr, nz, 43, O.MUR1, 3, select=0)
    for c in range(3):
        _close(b.field(c), a.field(c), tol=2e-6, what=f"comp {c}")
    _close(b.probes(), a.probes(), tol=2e-6, what="traces")
