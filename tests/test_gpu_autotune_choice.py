"""The autotuner tells the cells in order from rows of as many threads: at nx =
16 a warp of a row is half empty, so a launch over the cells in order wins."""
import pytest

from paper_0912_4230_gb300 import lb, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("dims,choice", [((16, 64, 256), 2128)])
def test_the_linear_launch_has_a_code_of_its_own(dims, choice):
    g = lb.Lattice(W.miscible(*dims, seed=4), storage="fp16")
    assert lb.lb_autotune(g.ctx, 5) == choice
