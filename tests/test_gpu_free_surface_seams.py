"""Free surface across the periodic seams of a lattice whose last tiles are
partial (tiles are 32 x 1 x 2 cells; nx % 32 != 0, nz odd).

The neighbour of a cell at x = nx - 1 or z = nz - 1 lies in the first tile of
the row. A liquid film whose front passes the seam in a step that builds the
lists afresh (every 16th) must agree with the FP64 oracle: cell types bit-exact
and mass to 1e-10, the bounds of the drop tests.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_0912_4230_gb300 import lb, workloads as W

pytestmark = pytest.mark.gpu

REBUILD = 16


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def film(dims, axis, v):
    """A film across the box, 7 cells thick, its front 5 cells from the high
    side along `axis` and moving towards it with speed v; all sides periodic."""
    nx, ny, nz = dims
    p = W.drop(nx=nx, ny=ny, nz=nz, R=1.0, gap=1.0, perturb=0.0)
    i = np.indices((nz, ny, nx))[2 - axis]
    lo, hi = dims[axis] - 12, dims[axis] - 5
    liquid, near = (i >= lo) & (i < hi), (i == lo - 1) | (i == hi)
    ctype = np.where(liquid, W.LIQUID, np.where(near, W.INTERFACE, W.EMPTY)).astype(np.uint8)
    lam = np.where(liquid, 1.0, np.where(near, 0.5, 0.0)).astype(np.float32)
    u0 = np.zeros((p.N, 3), np.float32)
    u0[ctype.ravel() != W.EMPTY, axis] = v
    periodic = ((W.PERIODIC, W.PERIODIC),) * 3
    return p.replace(bc=periodic, sbc=periodic, solid=np.zeros(p.N, np.uint8),
                     rho0=np.ones(p.N, np.float32), u0=u0.ravel(), cell_type=ctype.ravel(),
                     lambda0=lam.ravel())


@pytest.mark.parametrize("dims,axis", [((70, 4, 3), 0), ((33, 5, 19), 2), ((6, 5, 31), 2)])
def test_film_over_the_seam_of_partial_tiles_fp64(dims, axis):
    p = film(dims, axis, 0.094)
    shape = dims[::-1]
    g = lb.Lattice(p, storage="fp64")
    o = O.Oracle(p)
    m0 = g.reduce()[0]
    born = 0
    for t in range(1, 97):
        before = o.free_surface_state()[0].reshape(shape)
        o.step(1)
        g.step(1)
        ot, om = o.free_surface_state()
        if t % REBUILD == 0:
            new = (before == W.EMPTY) & (ot.reshape(shape) == W.INTERFACE)
            born += int(new.take(0, axis=2 - axis).sum())
        gt, gm = g.free_surface_state()
        assert np.array_equal(gt, ot), t
        assert np.abs(gm - om).max() < 1e-10, t
    assert born   # the case: cells born beyond the seam as the lists are rebuilt
    assert abs(g.reduce()[0] / m0 - 1) < 1e-12
