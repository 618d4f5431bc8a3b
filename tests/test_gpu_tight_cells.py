"""Nearly impermeable cells of a full permeability tensor: K so small that
det(I + eps nu/2 K^-1) leaves the range of FP32.

With eps 0.3 .. 1 and nu 0.07 .. 0.27 a factor of the determinant is about
0.05 / K, so det passes 2^126 near K = 1e-15 (where a reciprocal flushed to 0
would lose the drag), 2^128 below it (1/det = 0, or not a number), and at K =
1e-22 its 2 x 2 minors overflow too. The velocity there is 0 to rounding and the
drag takes twice the momentum that arrives, so the fields stay within the usual
bounds against the FP64 oracle: u 1e-5 of max|u|, rho 1e-6, C 1e-5 for FP32;
1.2e-7 for the exported floats of FP64. FP16 storage: remainders per unit weight
reach 0.1 here and are rounded by 2^-12 of that; a component of the momentum
sums a third of the weight (8e-6) in each of 6 steps, so u to 5e-5.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_0912_4230_gb300 import lb, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def tight_medium(K, dims=(19, 7, 6), along=(1.0, 1.0, 1.0)):
    """random_medium with a third of the cells at permeability K (times `along`
    per axis, off-diagonal entries scaled with the axes)."""
    p = W.random_medium(*dims, seed=11)
    K6 = np.asarray(p.K6, np.float64).reshape(-1, 6).copy()
    tight = np.random.default_rng(4).uniform(size=p.N) < 1 / 3
    s = np.sqrt(np.array(along))
    scale = np.array([s[0] * s[0], s[1] * s[1], s[2] * s[2], s[0] * s[1], s[1] * s[2], s[2] * s[0]])
    K6[tight] *= (K / K6[tight, :1]) * scale
    return p.replace(K6=K6.astype(np.float32).ravel())


def check(p, storage):
    g = lb.Lattice(p, storage=storage, check_every=1)
    o = O.Oracle(p)
    g.step(6)
    o.step(6)
    rho, u, C, _ = g.fields()   # raises where a sum is not finite
    r_rho, r_u, r_C, _ = o.fields()
    live = p.solid == 0
    assert np.isfinite(u).all() and np.isfinite(rho).all() and np.isfinite(C).all()
    if storage == "fp16":
        assert np.abs(u - r_u)[live].max() <= 5e-5
    else:
        tu, trho, tC = (1e-5, 1e-6, 1e-5) if storage == "fp32" else (1.2e-7,) * 3
        assert np.abs(u - r_u)[live].max() <= tu * np.abs(r_u[live]).max()
        assert np.abs(rho - r_rho)[live].max() <= trho
        assert np.abs(C - r_C)[live].max() <= tC


@pytest.mark.parametrize("storage", ["fp32", "fp64", "fp16"])
@pytest.mark.parametrize("K", [1e-12, 1e-14, 1e-15, 6e-16, 1e-16, 1e-18, 1e-20, 1e-22])
def test_full_tensor_of_nearly_tight_cells(K, storage):
    check(tight_medium(K), storage)


@pytest.mark.parametrize("along", [(1.0, 1.0, 1e12), (1.0, 1e-8, 1e8), (1e4, 1.0, 1.0)])
def test_full_tensor_tight_along_some_axes(along):
    check(tight_medium(1e-18, along=along), "fp32")


@pytest.mark.parametrize("storage", ["fp32", "fp64"])
def test_diagonal_tensor_at_the_smallest_permeability(storage):
    """K = 1.5e-38 at nu = 4.8: 1 + eps nu k / 2 is 0.5e38 .. 1.6e38, on both sides
    of 2^126 (the reciprocal of more is subnormal)."""
    p = W.random_medium(19, 7, 6, seed=11, spd=False, visc_law=0)
    K6 = np.asarray(p.K6, np.float64).reshape(-1, 6).copy()
    tight = np.random.default_rng(4).uniform(size=p.N) < 1 / 3
    K6[tight, :3] = 1.5e-38
    check(p.replace(K6=K6.astype(np.float32).ravel(), params=dict(p.params, tau=15.0)), storage)
