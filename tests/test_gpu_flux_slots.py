"""Flux totals do not depend on the per-cell launch: lb_step and lb_step_batch
after lb_autotune has chosen rows, bit for bit (FP16 storage, whose only kernels
are the per-cell ones)."""
import numpy as np
import pytest

from paper_0912_4230_gb300 import lb, workloads as W

pytestmark = pytest.mark.gpu

# widths near a whole number of warps, where rows may win over the order of n
DIMS = [(127, 64, 48), (63, 96, 40), (125, 60, 41), (95, 48, 40), (31, 128, 60), (128, 64, 48),
        (64, 96, 40)]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def test_batch_and_own_steps_agree_after_autotune():
    probs = [W.miscible(*d, seed=i) for i, d in enumerate(DIMS)]
    own = [lb.Lattice(p, storage="fp16") for p in probs]
    bat = [lb.Lattice(p, storage="fp16") for p in probs]
    # (timings vary: several tries, until both took the same launch)
    pairs = []
    for a, b in zip(own, bat):
        for _ in range(6):
            if lb.lb_autotune(a.ctx, 1) == lb.lb_autotune(b.ctx, 1):
                pairs.append((a, b))
                break
    for a, _ in pairs:
        a.step(21)
    lb.lb_step_batch([b.ctx for _, b in pairs], 21)
    for a, b in pairs:
        assert np.array_equal(a.reduce(), b.reduce())


def test_a_batch_follows_a_member_that_is_tuned_between_calls():
    """A graph of the batch holds the members' launches of its capture."""
    probs = [W.random_medium(37, 9, 8, seed=1), W.random_medium(19, 12, 7, seed=3)]
    own = [lb.Lattice(p, storage="fp16") for p in probs]
    bat = [lb.Lattice(p, storage="fp16") for p in probs]
    lb.lb_step_batch([g.ctx for g in bat], 8)
    lb.lb_autotune(bat[1].ctx, 3)
    lb.lb_step_batch([g.ctx for g in bat], 8)
    for a, b in zip(own, bat):
        a.step(16)
        fa, ha = a.populations()
        fb, hb = b.populations()
        assert np.array_equal(fa, fb) and np.array_equal(ha, hb)
