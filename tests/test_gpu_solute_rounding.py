"""Rounding of the FP32 solute collision: unbiased, so that a closed box keeps
its solute far below one rounding per step.

A step rounds a cell's 19 populations once each: 2^-24 / sqrt(12) of each at
random, 0.4 of that of their sum (the root of sum w_q^2), over sqrt(N) cells and
sqrt(60) steps 6e-10 of the total at N = 8568. The bound 2^-24 leaves a factor of
100 for correlated roundings; a collision that loses 1e-8 of it every time is at
3e-7 .. 5e-7 after 60 steps.
"""
import numpy as np
import pytest

from paper_0912_4230_gb300 import lb, workloads as W

pytestmark = pytest.mark.gpu

BOUND = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("tau_D", [0.6, 0.75, 0.8, 1.2])
def test_closed_box_keeps_its_solute_fp32(tau_D):
    p = W.random_medium(21, 24, 17, seed=3, inlet=False)
    p = p.replace(params=dict(p.params, tau_D=tau_D))
    p = W.with_species(p, tau_D=(tau_D,), C_in=(0.0,), C0=(np.full(p.N, 0.3),))
    g = lb.Lattice(p, storage="fp32")
    s0 = g.reduce()[1]
    t0 = g.species_state(1)[1][0]
    g.step(60)
    assert abs(g.reduce()[1] / s0 - 1) <= BOUND
    assert abs(g.species_state(1)[1][0] / t0 - 1) <= BOUND
