"""Exported viscosity of FP32 lattices to rounding.

nu = (tau - 1/2)/3 is formed from the law's own constants: rounded once each
(2^-24), and once in the result. Through a rounded tau = 0.6 the difference
tau - 1/2 was off by 2.4e-7, and with it the drag.
"""
import numpy as np
import pytest

from paper_0912_4230_gb300 import lb, workloads as W

pytestmark = pytest.mark.gpu

BOUND = 2 * 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("tau", [0.6, 0.51, 0.7])
@pytest.mark.parametrize("law", [0, 1, 2])
def test_viscosity_of_each_law_fp32(law, tau):
    p = W.random_medium(19, 6, 5, seed=4, inlet=False)
    nu = (tau - 0.5) / 3
    p = p.replace(C0=np.zeros(p.N, np.float32), params=dict(
        p.params, visc_law=law, tau=tau, tau0=tau, tau1=1.5, nu_g=nu, a=0.0, beta=0.0, A=0.0))
    g = lb.Lattice(p, storage="fp32")
    g.step(2)
    got = g.fields()[3][p.solid == 0]
    assert np.abs(got / nu - 1).max() <= BOUND
