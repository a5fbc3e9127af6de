"""The persistent ensemble's band sweep with its grid barrier (planes in memory):
taken for runs of fewer than 8 steps, and at any length when an instance has no
tiling on chip.  Every schedule, bitwise against the plain form."""
import pytest
import torch

import pf_inputs as G

pytestmark = pytest.mark.gpu


def ensemble(shapes):
    import paper_2601_06079_gb300 as pf
    e = pf.Ensemble(shapes)
    e.set_params([dict(W=0.8 + 0.1 * (i % 4), kappa=1.0 - 0.1 * (i % 3), L=1.0, dt=0.01)
                  for i in range(len(shapes))])
    st = e.pack([G.ac_initial(20 + i, s) for i, s in enumerate(shapes)])
    return e, st


def check(shapes, steps, schedules):
    e, st0 = ensemble(shapes)
    plain = st0.clone()
    e.step(plain, steps, "plain")
    cands = e.candidates()
    for k in schedules:
        sched = [cands[(k + i) % len(cands)] for i in range(len(shapes))]
        e.set_schedule([c[0] for c in sched], [c[1] for c in sched])
        st = st0.clone()
        e.step(st, steps, "persistent")
        assert torch.equal(st, plain), k


@pytest.mark.parametrize("steps", [1, 2, 7])
def test_short_runs(steps):
    check([(64, 64), (37, 100), (128, 128), (91, 37), (130, 256), (4, 5)], steps, range(9))


def test_an_instance_too_large_for_the_chip():
    # 9 million nodes: 288 tiles of 128 columns would need 250 rows each
    check([(3000, 3000), (64, 64), (129, 61)], 12, (0, 4, 8))
