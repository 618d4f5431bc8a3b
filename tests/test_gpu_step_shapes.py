"""The per-cell step kernel at the edges of its launch shapes and features,
against the FP64 oracle.

Cells are taken in rows where those fill whole blocks and else in the order of
n, by blocks of one warp while all warps are resident at once and of 128
threads beyond; the sizes lie on both sides of each line. Tolerances are those
of the parity tests: FP32 fields to 1e-5 of max|u|, 1e-6 in rho, 1e-5 in C, FP64
populations to 1e-13.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_0912_4230_gb300 import lb, workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": dict(u=1e-5, rho=1e-6, C=1e-5), "fp64": dict(u=1.2e-7, rho=1.2e-7, C=1.2e-7)}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def check(prob, storage, steps, species=1):
    g = lb.Lattice(prob, storage=storage, check_every=1)
    o = O.Oracle(prob)
    g.step(steps)
    o.step(steps)
    rho, u, C, _ = g.fields()
    r_rho, r_u, r_C, _ = o.fields()
    live = prob.solid == 0
    tol = TOL[storage]
    assert np.abs(u - r_u)[live].max() <= tol["u"] * np.abs(r_u[live]).max()
    assert np.abs(rho - r_rho)[live].max() <= tol["rho"]
    assert np.abs(C - r_C)[live].max() <= tol["C"]
    if storage == "fp64":
        f, h = g.populations()
        rf, rh = o.populations()
        assert np.abs(f - rf)[:, live].max() <= 1e-13
        if h is not None:
            assert np.abs(h - rh)[:, live].max() <= 1e-13
    return g, o


@pytest.mark.parametrize("storage", ["fp64", "fp32"])
@pytest.mark.parametrize("dims", [(1, 1, 33), (16, 3, 5), (31, 2, 3), (33, 1, 7), (64, 3, 2),
                                  (96, 4, 3), (117, 5, 4), (128, 3, 2), (160, 2, 3)])
def test_cells_of_every_row_width(dims, storage):
    """Walls, solid cells, inlet and outlet, full K, at widths that fill whole
    warps and blocks and at those that do not."""
    check(W.random_medium(*dims, seed=sum(dims)), storage, 5)


@pytest.mark.parametrize("storage,dims", [
    ("fp32", (48, 48, 50)), ("fp32", (48, 48, 51)),    # 152 * 32 * 24 cells lie between
    ("fp64", (36, 40, 40)), ("fp64", (36, 40, 41)),    # 152 * 32 * 12
])
def test_both_sides_of_the_one_warp_blocks(storage, dims):
    check(W.miscible(*dims, seed=2), storage, 3)


@pytest.mark.parametrize("storage", ["fp64", "fp32"])
@pytest.mark.parametrize("A", [0.0, 1e-3])
def test_species_with_and_without_surface_tension(storage, A):
    p = W.with_species(W.random_medium(19, 7, 6, seed=8, A=A), tau_D=(1.1,), C_in=(0.4,))
    g, o = check(p, storage, 6)
    C, _, _ = g.species_state(1)
    r_C = o.species_state(1)[0]
    live = p.solid == 0
    assert np.abs(C - r_C)[live].max() <= TOL[storage]["C"]


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_a_non_finite_population_is_flagged_at_the_next_checked_step(storage, value):
    g = lb.Lattice(W.miscible(33, 5, 4, seed=1), storage=storage, check_every=1)
    g.step(2)
    g.sync()
    f, h = g.populations()
    h[3, 77] = value
    g.set_populations(f, h)
    g.step(1)
    with pytest.raises(lb.LbError) as e:
        g.sync()
    assert e.value.code == lb.LB_ENONFINITE


@pytest.mark.parametrize("dims,R,gap", [((37, 21, 23), 6.0, 1.5), ((33, 34, 19), 5.0, 0.5)])
def test_drop_across_tile_edges_and_list_rebuilds(dims, R, gap):
    """A drop that lands, spreads over tile edges and the periodic sides of a
    lattice of partial tiles: FP64 cell types bit-exact and mass to 1e-10 at
    step counts around the rebuilding of the tile list (every 16 steps)."""
    p = W.drop(*dims, R=R, gap=gap, seed=5, u_drop=0.05)
    g = lb.Lattice(p, storage="fp64")
    o = O.Oracle(p)
    done = 0
    for t in (1, 15, 16, 17, 33, 80, 161):
        g.step(t - done)
        o.step(t - done)
        done = t
        gt, gm = g.free_surface_state()
        ot, om = o.free_surface_state()
        assert np.array_equal(gt, ot), t
        assert np.abs(gm - om).max() < 1e-10, t
    rho, u, _, _ = g.fields()
    rr, ru, _, _ = o.fields()
    live = ot != W.EMPTY
    assert np.abs(rho - rr)[live].max() <= 1.2e-7 * max(1.0, np.abs(rr[live]).max())
    assert np.abs(u - ru)[live].max() <= 1.2e-7 * np.abs(ru[live]).max() + 1e-9
    assert not rho[~live].any() and not u[~live].any()
